// K1-TC for the 32^3 window (Sec. 2 steps 1-3; Eq. 2, Eq. 1): stages 2 and 3 (the DFTs along x and y) on the tensor
// cores, as for the smaller windows, with the shapes of n = 32:
//   brick: one t0, 4 positions x0, 16 outputs y0; MMA rows m = (x0 - xb) * 32 + k_x, 128 of them;
//   stage 1 (t), once for all k_t: a thread per halo position (x, y) takes its 32 samples from global memory, scaled by
//     the brick's 1/max|V| and rounded to FP16, through a real FFT in FP32; every k_t's G1 is kept in 16 bits (the
//     rounding of the stage-2 operand), [slot][position] pairs (re, im), slot 0 = (k_t = 0, k_t = 16), both real;
//   stage 2 (x), per k_t: B2[(re|im, y)][(cos|sin, x)] = [[G1r, G1i], [G1i, -G1r]] (K-major, x over a 40-row halo) is
//     laid out from G1, 16 bytes (8 x) at a time; A2 = the Toeplitz twiddles h(x - x0) [cos | sin](2 pi k_x (x - x0) / n),
//     so one MMA chain (K = 80, N = 96) gives Re G2 and Im G2 of every (x0, k_x) row and halo column y, which are
//     rounded into the stage-3 A operands;
//   stage 3 (y): B = the 32 twiddle columns over 32 taps (two K steps), each bin's cosine and sine side by side (columns
//     0, 1: cos 0 and cos 16, the self-paired bins; 2j, 2j + 1: cos j, sin j); one output y0 = 64 columns (A_re B | A_im B).
// A pass is two outputs, one of three accumulator buffers in turn.  The 16 warps (four per tensor-memory lane quarter) form
// two groups that take the passes alternately, a warp per output and quarter, so that the square roots of one group fill
// the waits of the other.  They meet only on mbarriers: when a pass's eight warps have read its buffer, one of them (another
// one each pass) issues the buffer's next MMAs; D2 has columns of its own and A3 is double-buffered by k_t, so the next tile's
// operands are laid out in the middle of this one and the passes run on across tiles.  Whoever issued them, a pass's MMAs
// are complete once its barrier is, and a warp that reads pass P knows (through the barriers of the passes between) that
// those of P - 3 and before are.
// Bound: latency between the passes (about 12 k cycles a k_t tile, of which the MUFU pipe needs 4.1 k for the 17,408
// square roots a voxel, the MMAs 3 to 4 k, and a group's four epilogues take 6.4 k); stage 1 takes 30 k of 235 k cycles a
// brick.  64 x 96 x 96: 12.4 -> 6.3 ms, the call 6.4 (before: CTA-wide barriers around every pass, the FP32 sums of stage 1 again for
// every k_t, a maximum pass over every brick, operands laid out in 2-byte pieces with a division each).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "spectra_f32_fft.cuh"
#include "tc_sm100.cuh"

namespace sal {
namespace {

using f32::bin_mag;
using f32::Tw;

constexpr int N = 32, H = N / 2 + 1, P = 128 / N, BY = 16;
constexpr int XH = P + N - 1, YH = BY + N - 1, POS = XH * YH;
constexpr int KROWS = BY + N - 1;                        // window start + 32 taps
constexpr uint32_t SBO_A = KROWS * 16;
constexpr int kWarps = 16, kThreads = 32 * kWarps;
constexpr int kOuts = 2, kPasses = BY / kOuts, kBufs = 3;   // outputs per pass (one accumulator buffer), passes per tile
constexpr int kOwn = kPasses / 2;                        // passes of a tile that a group takes
constexpr uint32_t kTmemCols = 512;                      // three buffers of 2 outputs x 64 columns, then D2
constexpr uint32_t kColD2 = kBufs * kOuts * 64;
constexpr uint32_t kWaitLimit = 1u << 22;

constexpr int XHP = 40;                                  // x halo rows of stage 2 (>= XH, multiple of 8)
constexpr int YP = 48;                                   // y columns of stage 2 (>= YH, multiple of 8)
constexpr int K2 = 2 * XHP;                              // stage-2 K: cos taps | sin taps
constexpr int N2 = 2 * YP;                               // stage-2 N: re | im over y
constexpr uint32_t SBO_K2 = K2 / 8 * 128;                // 8-row group stride of the K-major A2 / B2
constexpr size_t G1_B = (size_t)(N / 2) * POS * 4;
constexpr size_t B2_B = (size_t)N2 / 8 * SBO_K2;         // stage-2 B (one k_t)
constexpr size_t A2_B = (size_t)16 * SBO_K2;             // stage-2 A (128 rows)
constexpr size_t A_B = (size_t)16 * SBO_A;
constexpr size_t B_B = 2048;
constexpr size_t OFF_B2 = (G1_B + 127) / 128 * 128;
constexpr size_t OFF_TAB = OFF_B2 + B2_B;                // A2, then the stage-3 B (the constant operands)
constexpr size_t TAB_B = A2_B + B_B;
constexpr size_t OFF_A = OFF_TAB + TAB_B;
constexpr size_t WT_B = ((size_t)3 * H * H * 4 + 15) / 16 * 16;   // Eq. 1 weights of one k_t, [map][|k_y|][|k_x|]; two, by k_t
constexpr size_t OFF_WT = OFF_A + 4 * A_B;               // (A_re, A_im) twice, by k_t
constexpr size_t OFF_MISC = OFF_WT + 2 * WT_B;
// mbarriers (arrivals): pass P complete (commit; by P % 6, so that a group waits for every phase of those it uses), buffer
// read (the 8 warps of a group; by P % 3), stage-3 A written (16 warps; two, by k_t), stage-2 B written (16 warps), D2 complete
// (commit), constant operands landed, weights landed (two, by k_t)
enum : int { B_FULL = 0, B_READ = 6, B_A3 = 9, B_B2 = 11, B_D2 = 12, B_TAB = 13, B_WT = 14, kBars = 16 };
constexpr size_t SMEM = OFF_MISC + 8 * kBars + 16;
constexpr size_t WT_FLOATS = H * WT_B / 4;               // of all k_t
static_assert(SMEM <= 227 * 1024, "shared memory");
static_assert(XH <= XHP && YH <= YP && N2 <= 256 && N2 % 16 == 0, "stage-2 shapes");
static_assert(OFF_B2 % 128 == 0 && OFF_TAB % 128 == 0 && OFF_A % 16 == 0 && TAB_B % 16 == 0 && OFF_WT % 16 == 0 &&
                  WT_B % 16 == 0, "operand alignment");
static_assert(kColD2 + N2 <= kTmemCols && kWarps == 2 * 4 * kOuts, "a warp per output and lane quarter in each group");

template <int FMT> struct Pack;
template <> struct Pack<1> {
    __device__ static uint16_t one(float a) {
        __nv_bfloat16 v = __float2bfloat16_rn(a);
        return *reinterpret_cast<uint16_t*>(&v);
    }
    __device__ static uint32_t two(float a, float b) {
        __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
        return *reinterpret_cast<uint32_t*>(&v);
    }
};
template <> struct Pack<0> {
    __device__ static uint16_t one(float a) {
        __half v = __float2half_rn(a);
        return *reinterpret_cast<uint16_t*>(&v);
    }
    __device__ static uint32_t two(float a, float b) {
        __half2 v = __floats2half2_rn(a, b);
        return *reinterpret_cast<uint32_t*>(&v);
    }
};

// The constant operands, once per handle: A2[(x0l, k_x)][k2] (k2 < XHP: cos, else sin, of (k_x, x - x0l), x = k2 % XHP;
// zero outside the window), then the stage-3 B [column][tap].
template <int FMT>
__global__ void k1_tc32_tables(const __grid_constant__ Tw<N> tw, unsigned char* __restrict__ out) {
    for (int i = threadIdx.x; i < 128 * K2; i += blockDim.x) {
        const int mm = i / K2, k2 = i % K2;
        const int x0 = mm / N, kxx = mm % N, u = k2 % XHP - x0;
        float v = 0.f;
        if (u >= 0 && u < N) {
            const bool lo = kxx <= N / 2;
            const int kk = lo ? kxx : N - kxx;
            v = k2 < XHP ? tw.c[kk][u] : (lo ? tw.s[kk][u] : -tw.s[kk][u]);
        }
        *reinterpret_cast<uint16_t*>(out + (mm / 8) * SBO_K2 + (k2 / 8) * 128 + (mm % 8) * 16 + (k2 % 8) * 2) =
            Pack<FMT>::one(v);
    }
    for (int i = threadIdx.x; i < 32 * 32; i += blockDim.x) {
        const int n = i / 32, k = i % 32;
        const float v = n == 0 ? tw.c[0][k] : n == 1 ? tw.c[N / 2][k] : (n & 1) ? tw.s[n / 2][k] : tw.c[n / 2][k];
        *reinterpret_cast<uint16_t*>(out + A2_B + (n / 8) * 512 + (k / 8) * 128 + (n % 8) * 16 + (k % 8) * 2) =
            Pack<FMT>::one(v);
    }
}

// Per-axis taper h(u) of the window (1 for the rect cube).
struct Taper32 {
    float h[N];
};

// max|V| of every (plane t, brick)'s halo, [T][x bricks][y bricks]: a brick's maximum is then that of its 32 planes
// instead of a pass of its own over its 52,640 samples (21 k of 290 k cycles a brick).  A warp per (plane, brick).
__global__ void __launch_bounds__(256)
k1_tc32_max(const float* __restrict__ V, float* __restrict__ pmax, int T, int X, int Y, int bnd, int nyb, int nxb) {
    const int lane = threadIdx.x & 31;
    const long long w = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (w >= (long long)T * nxb * nyb) return;
    const int yb = (int)(w % nyb) * BY, xb = (int)(w / nyb % nxb) * P;
    const float* p = V + (size_t)(w / nyb / nxb) * X * Y;
    const int gy0 = ext_index(yb - N / 2 + lane, Y, bnd);
    const int gy1 = lane + 32 < YH ? ext_index(yb - N / 2 + lane + 32, Y, bnd) : -1;
    float m = 0.f;
#pragma unroll 7
    for (int x = 0; x < XH; ++x) {
        const int gx = ext_index(xb - N / 2 + x, X, bnd);
        const float a = gx >= 0 && gy0 >= 0 ? __ldg(p + (size_t)gx * Y + gy0) : 0.f;
        const float b = gx >= 0 && gy1 >= 0 ? __ldg(p + (size_t)gx * Y + gy1) : 0.f;
        m = fmaxf(m, fmaxf(fabsf(a), fabsf(b)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) pmax[w] = m;
}

template <int FMT, bool EN>
__global__ void __launch_bounds__(kThreads, 1)
k1_spectra_tc32(const float* __restrict__ V, float* __restrict__ E, int T, int X, int Y, int bnd, int stride,
                const unsigned char* __restrict__ tables, const float* __restrict__ wtab,
                const float* __restrict__ pmax, const __grid_constant__ Taper32 taper, int* __restrict__ err) {
    extern __shared__ __align__(128) unsigned char smem[];
    uint32_t* s_g1 = reinterpret_cast<uint32_t*>(smem);                 // [N / 2][XH][YH] (re, im) in 16 bits
    unsigned char* s_b2 = smem + OFF_B2;                                // stage-2 B (K-major)
    unsigned char* s_tab = smem + OFF_TAB;                              // stage-2 A (K-major), stage-3 B (K-major)
    unsigned char* s_a3 = smem + OFF_A;                                 // [2][re | im]
    uint64_t* s_mbar = reinterpret_cast<uint64_t*>(smem + OFF_MISC);
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(smem + OFF_MISC + 8 * kBars);
    int* s_fail = reinterpret_cast<int*>(smem + OFF_MISC + 8 * kBars + 4);
    float* s_max = reinterpret_cast<float*>(smem + OFF_MISC + 8 * kBars + 8);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int yb = blockIdx.x * BY, xb = blockIdx.y * P, t0 = blockIdx.z * stride;   // stride s: planes t0 = k s

    const float* s_wt = reinterpret_cast<const float*>(smem + OFF_WT);
    auto load_wt = [&](int kt) {   // one thread
        const uint32_t bar = tc::smem_u32(&s_mbar[B_WT + (kt & 1)]);
        tc::mbar_arrive_expect_tx(bar, (uint32_t)WT_B);
        tc::bulk_g2s(tc::smem_u32(smem + OFF_WT + (kt & 1) * WT_B), wtab + (size_t)kt * (WT_B / 4), (uint32_t)WT_B, bar);
    };

    if (warp == 0) tc::tmem_alloc(tc::smem_u32(s_tmem), kTmemCols);
    if (tid == 0) {
        for (int b = 0; b < kBars; ++b)
            tc::mbar_init(tc::smem_u32(&s_mbar[b]), b >= B_READ && b < B_A3 ? kWarps / 2 : b >= B_A3 && b <= B_B2 ? kWarps : 1);
        *s_fail = 0;
        tc::mbar_arrive_expect_tx(tc::smem_u32(&s_mbar[B_TAB]), (uint32_t)TAB_B);
        tc::bulk_g2s(tc::smem_u32(s_tab), tables, (uint32_t)TAB_B, tc::smem_u32(&s_mbar[B_TAB]));
        load_wt(0);
    }
    // B2 rows and columns past the halo stay zero (A2 is zero there too, but 0 x garbage could be NaN)
    for (int i = tid; i < (int)(B2_B / 16); i += kThreads)
        reinterpret_cast<uint4*>(s_b2)[i] = make_uint4(0u, 0u, 0u, 0u);

    __shared__ int s_gt[N];   // the planes of the taps
    if (warp == 1) s_gt[lane] = ext_index(t0 - N / 2 + lane, T, bnd);
    // ---- the brick's maximum, over the planes' -----------------------------------------------------------
    if (warp == 0) {
        const int gt = ext_index(t0 - N / 2 + lane, T, bnd);
        float vmax = gt >= 0 ? __ldg(pmax + ((size_t)gt * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
        if (lane == 0) *s_max = vmax;
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *s_tmem;
    const float bmax = *s_max;
    const float scale = bmax > 0.f ? bmax : 1.f;
    const float inv_scale = 1.f / scale;

    const size_t plane = (size_t)X * Y;
    const bool t_in = t0 - N / 2 >= 0 && t0 + N / 2 <= T;
    // ---- stage 1: every k_t of a halo position at once ---------------------------------------------------
    for (int it = tid; it < POS; it += kThreads) {
        // the 32 samples of the column along t, all loads in flight; lanes along y
        const int x = it / YH, y = it - x * YH;
        const int gx = ext_index(xb - N / 2 + x, X, bnd), gy = ext_index(yb - N / 2 + y, Y, bnd);
        const bool in = (gx | gy) >= 0;
        const float* p = V + (in ? (size_t)gx * Y + gy : 0);
        float v[N];
        if (t_in) {
            p += (size_t)(t0 - N / 2) * plane;
#pragma unroll
            for (int u = 0; u < N; ++u) v[u] = in ? __ldg(p + u * plane) : 0.f;
        } else {
#pragma unroll
            for (int u = 0; u < N; ++u) {
                const int gt = s_gt[u];
                v[u] = in && gt >= 0 ? __ldg(p + gt * plane) : 0.f;
            }
        }
#pragma unroll
        for (int u = 0; u < N; u += 2) {
            const float2 r = __half22float2(__floats2half2_rn(v[u] * inv_scale, v[u + 1] * inv_scale));
            v[u] = taper.h[u] * r.x;
            v[u + 1] = taper.h[u + 1] * r.y;
        }
        float2 o[N / 2];
        f32::rfft<N>(v, o);
#pragma unroll
        for (int k = 0; k < N / 2; ++k)
            s_g1[k * POS + it] = Pack<FMT>::two(o[k].x, o[k].y);
    }
    __syncthreads();

    const int q = warp & 3, out = (warp >> 2) & 1, grp = warp >> 3;   // lane quarter (x0); output of a pass; group
    const int kx = lane, x0l = q, m = 32 * q + lane;
    const uint32_t lane_base = (uint32_t)(32 * q) << 16;
    volatile int* v_fail = s_fail;
    // warp-uniform bounded wait for the given phase of a barrier; a give-up stops all further issue
    auto wait = [&](int b, int phase) -> bool {
        bool ok = !*v_fail && tc::mbar_wait(tc::smem_u32(&s_mbar[b]), (uint32_t)phase & 1u, kWaitLimit);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok && lane == 0 && !*v_fail) {
            atomicOr(err, 1);
            atomicExch(s_fail, 1);
        }
        tc::fence_after_sync();
        return ok;
    };
    auto arrive = [&](int b) {
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(tc::smem_u32(&s_mbar[b]));
    };
    // stage-2 B of tile kt: item = (y, 8 x): 8 (re, im) pairs -> four 16-byte rows parts.
    // K-major: byte(ncol, k2) = (ncol/8) SBO_K2 + (k2/8) 128 + (ncol%8) 16 + (k2%8) 2; ncol = y (re) or YP + y (im),
    // k2 = x (cos) or XHP + x (sin)
    auto layout_b2 = [&](int kt) {
        unsigned char* b2 = s_b2;
        const uint32_t* g1 = s_g1 + (kt == N / 2 ? 0 : kt) * POS;
        if (tid < YH * (XHP / 8)) {
            const int y = tid % YH, xg = tid / YH;
            uint32_t re[4], im[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int x = 8 * xg + 2 * i;
                const uint32_t a = x < XH ? g1[x * YH + y] : 0u, b = x + 1 < XH ? g1[(x + 1) * YH + y] : 0u;
                const uint32_t lo = __byte_perm(a, b, 0x5410), hi = __byte_perm(a, b, 0x7632);
                re[i] = kt == N / 2 ? hi : lo;
                im[i] = kt == 0 || kt == N / 2 ? 0u : hi;
            }
            unsigned char* o_re = b2 + (size_t)(y / 8) * SBO_K2 + (y % 8) * 16;
            unsigned char* o_im = b2 + (size_t)((YP + y) / 8) * SBO_K2 + ((YP + y) % 8) * 16;
            const size_t k_c = (size_t)xg * 128, k_s = (size_t)(XHP / 8 + xg) * 128;
            const uint4 r4 = make_uint4(re[0], re[1], re[2], re[3]), i4 = make_uint4(im[0], im[1], im[2], im[3]);
            *reinterpret_cast<uint4*>(o_re + k_c) = r4;
            *reinterpret_cast<uint4*>(o_re + k_s) = i4;
            *reinterpret_cast<uint4*>(o_im + k_c) = i4;
            *reinterpret_cast<uint4*>(o_im + k_s) = make_uint4(r4.x ^ 0x80008000u, r4.y ^ 0x80008000u,
                                                               r4.z ^ 0x80008000u, r4.w ^ 0x80008000u);
        }
        tc::fence_async_smem();
        arrive(B_B2);
    };
    // D2 -> the stage-3 A operands of tile kt (row m at K row y): the four warps of a lane quarter take y 0..31 and 32.. of
    // the real part (columns [0, YP)) and of the imaginary part ([YP, 2 YP))
    auto d2_to_a3 = [&](int kt) {
        if (wait(B_D2, kt)) {
            unsigned char* dst = s_a3 + (size_t)(2 * (kt & 1) + grp) * A_B + (m / 8) * SBO_A + (m % 8) * 2;
            const uint32_t col = tmem + lane_base + kColD2 + (grp ? YP : 0);
            if (out) {
                float v[16];
                tc::tmem_ld16(col + 32, v);
#pragma unroll
                for (int i = 0; i < YH - 32; ++i) *reinterpret_cast<uint16_t*>(dst + (32 + i) * 16) = Pack<FMT>::one(v[i]);
            } else {
                uint32_t r[32];   // 8 (rows) x 8 (y) blocks, stored transposed
                tc::tmem_ld32_blocks(col, r);
                const uint32_t d = tc::smem_u32(s_a3 + (size_t)(2 * (kt & 1) + grp) * A_B) + (uint32_t)(4 * q * SBO_A + lane * 16);
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    uint32_t b[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int i = 16 * (g / 2) + 4 * c + 2 * (g % 2);
                        b[c] = Pack<FMT>::two(__uint_as_float(r[i]), __uint_as_float(r[i + 1]));
                    }
                    tc::store_blocks_trans(d + (uint32_t)(g * SBO_A), b[0], b[1], b[2], b[3]);
                }
            }
            tc::fence_async_smem();
        }
        arrive(B_A3 + (kt & 1));
    };
    const uint32_t idesc2 = tc::idesc_f16(FMT, 128, N2, 0, 0), idesc3 = tc::idesc_f16(FMT, 128, 32, 1, 0);
    auto issue_s2 = [&]() {
        const uint64_t a2d = tc::desc_noswizzle(tc::smem_u32(s_tab), 128, SBO_K2);
        const uint64_t b2d = tc::desc_noswizzle(tc::smem_u32(s_b2), 128, SBO_K2);
        if (tc::elect_one()) {
#pragma unroll
            for (int ks = 0; ks < K2 / 16; ++ks)
                tc::mma_f16(tmem + kColD2, tc::desc_add(a2d, 256 * ks), tc::desc_add(b2d, 256 * ks), idesc2,
                            ks > 0 ? 1u : 0u);
            tc::mma_commit(tc::smem_u32(&s_mbar[B_D2]));
        }
        __syncwarp();
    };
    auto issue_s3 = [&](int P) {   // pass P of the brick (8 per tile)
        const uint32_t a3 = tc::smem_u32(s_a3) + (uint32_t)(2 * ((P / kPasses) & 1) * A_B);
        const uint64_t ared = tc::desc_noswizzle(a3, 128, SBO_A), aimd = tc::desc_noswizzle(a3 + (uint32_t)A_B, 128, SBO_A);
        const uint64_t bd = tc::desc_noswizzle(tc::smem_u32(s_tab) + (uint32_t)A2_B, 128, 512);
        const uint32_t buf = (uint32_t)(P % kBufs), col = tmem + kOuts * 64 * buf;
        if (tc::elect_one()) {
#pragma unroll
            for (int j = 0; j < kOuts; ++j) {
                const uint32_t y0 = (P % kPasses) * kOuts + j;
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                    tc::mma_f16(col + j * 64, tc::desc_add(ared, (y0 + 16 * ks) * 16), tc::desc_add(bd, 256 * ks), idesc3,
                                ks);
                    tc::mma_f16(col + j * 64 + 32, tc::desc_add(aimd, (y0 + 16 * ks) * 16), tc::desc_add(bd, 256 * ks),
                                idesc3, ks);
                }
            }
            tc::mma_commit(tc::smem_u32(&s_mbar[B_FULL + P % (2 * kBufs)]));
        }
        __syncwarp();
    };

    float acc[kOwn][3];
#pragma unroll
    for (int i = 0; i < kOwn; ++i) acc[i][0] = acc[i][1] = acc[i][2] = 0.f;
    layout_b2(0);
    if (warp == 0 && wait(B_TAB, 0) && wait(B_B2, 0)) issue_s2();
    d2_to_a3(0);
    if (warp == 0 && wait(B_A3, 0))
        for (int P = 0; P < kBufs; ++P) issue_s3(P);
    for (int kt = 0; kt < H; ++kt) {
        const bool more = kt + 1 < H;
        float wt[3][H];   // this lane's Eq. 1 weights for (k_t, k_x), |k_y| = 0 .. n/2
        wait(B_WT + (kt & 1), kt / 2);
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int k = 0; k < H; ++k) wt[c][k] = s_wt[(kt & 1) * (WT_B / 4) + (c * H + k) * H + min(kx, N - kx)];
#pragma unroll
        for (int i = 0; i < kOwn; ++i) {
            const int P = kt * kPasses + 2 * i + grp, buf = P % kBufs;
            // the next tile's operands: stage-2 B after the first pass, its MMAs in the second, A3 before the third
            if (i == 2 && more) d2_to_a3(kt + 1);
            const bool full = wait(B_FULL + P % (2 * kBufs), P / (2 * kBufs));
            float e0 = 0.f, e1 = 0.f, e2 = 0.f;
#pragma unroll
            for (int h = 0; h < 2; ++h) {   // columns 16 h .. 16 h + 15: bins k = 8 h .. 8 h + 7
                float vr[16], vi[16];
                if (full) tc::tmem_ld16x2(tmem + lane_base + (uint32_t)(kOuts * 64 * buf + 64 * out + 16 * h), 32u, vr, vi);
                if (h == 1) {
                    arrive(B_READ + buf);
                    // the buffer's next pass, once all eight warps have read it
                    const int Q = P + kBufs;
                    if ((warp & 7) == i && Q < H * kPasses && wait(B_READ + buf, P / kBufs) &&
                        (Q / kPasses == kt || wait(B_A3 + ((kt + 1) & 1), (kt + 1) / 2)))
                        issue_s3(Q);
                    // every warp has laid out its part of B2 (and is past the head of this tile: the other weight buffer
                    // is free); D2 was read when A3 was written
                    if (i == 1 && more && warp == 4 && wait(B_B2, kt + 1)) {
                        issue_s2();
                        if (lane == 0) load_wt(kt + 1);
                    }
                }
                if (!full) continue;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int k = 8 * h + c;
                    const float pr = vr[2 * c], pi = vi[2 * c], qr = vr[2 * c + 1], qi = vi[2 * c + 1];
                    if (k == 0) {   // columns 0, 1: the self-paired bins 0 and n/2
                        const float a0 = bin_mag<EN>(fmaf(pr, pr, pi * pi));
                        const float a1 = bin_mag<EN>(fmaf(qr, qr, qi * qi));
                        e0 = fmaf(wt[0][0], a0, fmaf(wt[0][H - 1], a1, e0));
                        e1 = fmaf(wt[1][0], a0, fmaf(wt[1][H - 1], a1, e1));
                        e2 = fmaf(wt[2][0], a0, fmaf(wt[2][H - 1], a1, e2));
                    } else {        // bins k and n - k: P = pr + i pi, Q = qr + i qi
                        const float ar = pr + qi, ai = pi - qr, br = pr - qi, bi = pi + qr;
                        const float a = bin_mag<EN>(fmaf(ar, ar, ai * ai)) + bin_mag<EN>(fmaf(br, br, bi * bi));
                        e0 = fmaf(wt[0][k], a, e0);
                        e1 = fmaf(wt[1][k], a, e1);
                        e2 = fmaf(wt[2][k], a, e2);
                    }
                }
            }
            acc[i][0] += e0;
            acc[i][1] += e1;
            acc[i][2] += e2;
            if (i == 0 && more) layout_b2(kt + 1);   // (the stage-2 MMAs of kt have completed: D2 was waited for)
        }
    }
    tc::fence_before_sync();
    __syncthreads();

    // E: [3][T][X][Y], or the lattice [3][Tc][Xc][Yc] (ceil(T / s) ...) for stride s > 1
    const int Xc = (X + stride - 1) / stride, Yc = (Y + stride - 1) / stride;
    const size_t NV = (size_t)((T + stride - 1) / stride) * Xc * Yc;
    const int x = xb + x0l;
    const float out_scale = EN ? scale * scale : scale;   // the features of the unscaled brick
#pragma unroll
    for (int i = 0; i < kOwn; ++i) {
        const int y0 = (2 * i + grp) * kOuts + out;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float s = acc[i][c];
#pragma unroll
            for (int o = 1; o < N; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            const int y = yb + y0;
            if (kx == 0 && x < X && y < Y && !*s_fail) {
                if (stride == 1)
                    E[c * NV + ((size_t)t0 * X + x) * Y + y] = s * out_scale;
                else if (x % stride == 0 && y % stride == 0)   // the lattice (a rare path)
                    E[c * NV + ((size_t)(t0 / stride) * Xc + x / stride) * Yc + y / stride] = s * out_scale;
            }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, kTmemCols);
}

template <int FMT, bool EN>
cudaError_t prepare32() {
    return cudaFuncSetAttribute(k1_spectra_tc32<FMT, EN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
}

constexpr size_t kWtOff = (TAB_B + 255) / 256 * 256;   // the weight table behind the operands

}  // namespace

cudaError_t spectra_tc32_prepare(int fmt) {
    cudaError_t e = fmt == 1 ? prepare32<1, false>() : prepare32<0, false>();
    if (e != cudaSuccess) return e;
    return fmt == 1 ? prepare32<1, true>() : prepare32<0, true>();
}

size_t spectra_tc32_tables_bytes() { return kWtOff + WT_FLOATS * sizeof(float); }

cudaError_t spectra_tc32_tables_build(int fmt, const TwiddleTable& t, int feat, void* dst, cudaStream_t s) {
    static_assert(WT_FLOATS * sizeof(float) < (1u << 20), "a host copy");
    unsigned char* out = static_cast<unsigned char*>(dst);
    const Tw<N> tw = f32::make_tw<N>(t);
    if (fmt == 1) k1_tc32_tables<1><<<1, 256, 0, s>>>(tw, out);
    else k1_tc32_tables<0><<<1, 256, 0, s>>>(tw, out);
    note_launches(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    float* wt = new float[WT_FLOATS]();
    for (int kt = 0; kt < H; ++kt)
        for (int k = 0; k < H; ++k)
            for (int j = 0; j < H; ++j) {
                const float mult = (kt == 0 || 2 * kt == N) ? 1.f : 2.f;
                float w[3];
                if (feat == 1) f32::bin_weights<true>(kt, j, k, mult / (float)(N * N * N), w[0], w[1], w[2]);
                else f32::bin_weights<false>(kt, j, k, mult / (float)(N * N * N), w[0], w[1], w[2]);
                for (int c = 0; c < 3; ++c) wt[(size_t)kt * (WT_B / 4) + (c * H + k) * H + j] = w[c];
            }
    e = cudaMemcpyAsync(out + kWtOff, wt, WT_FLOATS * sizeof(float), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);   // wt is pageable and leaves
    delete[] wt;
    return e;
}

cudaError_t spectra_tc32_launch(int fmt, const TwiddleTable& t, const void* tables, float* pmax, const float* V,
                                float* E, int T, int X, int Y, int bnd, int feat, int stride, int* err,
                                cudaStream_t s) {
    if (stride < 1) return cudaErrorInvalidConfiguration;
    dim3 grid((Y + BY - 1) / BY, (X + P - 1) / P, (T + stride - 1) / stride);
    const unsigned char* tab = static_cast<const unsigned char*>(tables);
    const float* wt = reinterpret_cast<const float*>(tab + kWtOff);
    Taper32 tp;
    for (int u = 0; u < N; ++u) tp.h[u] = t.c[0][u];
    const int st = stride;
    const long long rows = (long long)T * grid.x * grid.y;
    k1_tc32_max<<<(unsigned)((rows + 7) / 8), 256, 0, s>>>(V, pmax, T, X, Y, bnd, grid.x, grid.y);
    if (fmt == 1 && feat == 1)
        k1_spectra_tc32<1, true><<<grid, kThreads, SMEM, s>>>(V, E, T, X, Y, bnd, st, tab, wt, pmax, tp, err);
    else if (fmt == 1) k1_spectra_tc32<1, false><<<grid, kThreads, SMEM, s>>>(V, E, T, X, Y, bnd, st, tab, wt, pmax, tp, err);
    else if (feat == 1) k1_spectra_tc32<0, true><<<grid, kThreads, SMEM, s>>>(V, E, T, X, Y, bnd, st, tab, wt, pmax, tp, err);
    else k1_spectra_tc32<0, false><<<grid, kThreads, SMEM, s>>>(V, E, T, X, Y, bnd, st, tab, wt, pmax, tp, err);
    note_launches(2);
    return cudaGetLastError();
}

}  // namespace sal

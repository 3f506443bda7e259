// K1-F32, sliding form (rect cube, stride 1, n = 8, 16, 32): local 3D DFT around every voxel, spectral
// projection and feature, in FP32 on the SIMT pipes (Sec. 2 steps 1-3; Eq. 2 separable DFT, Eq. 1 projection).
//
// A CTA takes one t0, RX positions x0 and 16 to 32 outputs y0 and goes through the half spectrum in n/2 tiles
// (spectra_f32_fft.cuh):
//   stage 1 (t): a thread per halo position (x, y): its n samples straight from global memory (border extension
//            at load), a real FFT, every tile's G1[x][y] kept in shared memory (n = 32: four tiles at a time);
//   stage 2 (x): a thread per (x0, y): an n-point FFT of G1 -> G2[x0][k_x][y] of the tile;
//   stage 3 (y): a thread per (x0, k_x) and run of 16 outputs (n = 32: two threads, the even and the odd k_y):
//            the first window by an FFT (n = 8, 32: and the ninth), each later one by the sliding DFT anchored there,
//              F_{j+1}[k] = F_j[k] + (G2[j + n] - G2[j]) w^(k j),   w = e^(-2 pi i / n),
//            whose phase differs from that of the window itself by w^(k j): |F| is the same.  The products d w^m
//            need one complex multiply per distinct octant angle, the rest are sign changes and swaps, so a
//            bin costs two additions.  |F| (MUFU square root) weighted by Eq. 1 goes into 48 sums in registers (16
//            outputs, 3 maps) across all tiles; the lanes' sums over k_x meet in one shuffle tree at the end.
// Bound: the MUFU pipe, n^3/2 + n^2/2 roots per voxel at 16 per clock and SM (n = 16: 0.90 ms at 128^3), with about
// 110 issue slots per thread and output for its 16 bins beside 128 MUFU cycles.  The 48 sums, 16 bins and 27 weights
// take 168 registers a thread: 12 warps per SM, whose 16 independent bins each hide the latencies.
// 128^3: n = 16 7.23 -> 2.07 ms, n = 8 1.07 -> 0.28 ms; 48 x 64 x 64, n = 32: 21.2 -> 2.3 ms (before: direct DFTs in
// stages 1 and 2 and for each run's first output, a halo for every row of 32 outputs, a six-operation rotation
// per bin and output).  Error against FP64, relative L2 of E: 7e-8, 6e-8 and 8e-8 (before 1.3e-7, 7e-8 and 1.3e-7).
// The brick is staged minus one of its voxels (brick_shift): only the DC bin of a rect cube moves, which Eq. 1 leaves out, so a
// constant volume is exactly zero.
#include "spectra_f32_fft.cuh"

namespace sal {
namespace {

using f32::bin_mag;
using f32::Bins;


// Eq. 1 weights of the tiles, [tile][map][k][row] (k = |k_y|), then those of the packed rows' second signal
// (k_t = n/2), [map][k][row], 0 elsewhere.
template <int N> struct WGeo {
    static constexpr int H = N / 2 + 1, TILES = N / 2;
    static constexpr size_t TILE = (size_t)3 * H * N;
    static constexpr size_t FLOATS = (TILES + 1) * TILE;
};

// One tile of one thread: RUN outputs along the row g, |F| weighted into acc[output][map].  The recursion starts anew from an
// FFT every 16 outputs for n = 16 and every 8 for the others, no further than an extreme sample's rounding, or a NaN, may
// reach behind its windows (16 at n = 8 and 32 made features up to 15 outputs away lose what 8 keep).  The two halves of a run
// as one loop that is not unrolled, which also keeps n = 32 in the instruction cache: 48 x 64 x 64 2.75 -> 2.29 ms; n = 8,
// 128^3: 273 -> 277 us.
template <int N, int M, bool ODD, bool EN, int RUN>
__device__ __forceinline__ void slide_tile(const float2* __restrict__ g, const float* __restrict__ wtab, int tile,
                                           int row, float (&acc)[RUN][3]) {
    using W = WGeo<N>;
    using B = Bins<M, ODD>;
    constexpr int NW = B::NW, PART = RUN < 8 || N == 16 ? RUN : 8;
    static_assert(PART == RUN || 2 * PART == RUN, "two halves");
    float wt[3][NW];
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
        for (int w = 0; w < NW; ++w)
            wt[m][w] = __ldg(wtab + tile * W::TILE + (m * W::H + B::ky(w, N)) * N + row);
    B f;
    const float* wb = wtab + W::TILES * W::TILE + row;
    const float pk = (row == 0 || row == N / 2) ? 1.f : 0.f;   // tile 0: a packed row
#pragma unroll 1
    for (int h = 0; h < RUN; h += PART, g += PART) {
        f.template first<N>(g);
#pragma unroll
        for (int j = 0; j < PART; ++j) {
            if (j > 0) {
                const float2 a = g[j - 1], b = g[j - 1 + N];   // sample leaving, sample entering
                float2 d = make_float2(b.x - a.x, b.y - a.y);
                if (ODD) d = f32::rot32(d, j - 1);
                f.slide(d, j - 1);
            }
            float s[NW];
            if (tile != 0) {
#pragma unroll
                for (int q = 0; q < M / 2; ++q) {
                    const float2 m2 = __ffma2_rn(f.i[q], f.i[q], __fmul2_rn(f.r[q], f.r[q]));
                    const float a = bin_mag<EN>(m2.x), b = bin_mag<EN>(m2.y);
                    if (!ODD && q == 0) {
                        s[0] = a;
                        s[M / 2] = b;
                    } else {
                        s[q] = a + b;
                    }
                }
            } else {
                // tile 0: packed rows give F_0 + conj.. (x2) and F_{n/2} (x2) from the pair, the others their two bins
#pragma unroll
                for (int q = 0; q < M / 2; ++q) {
                    const float2 R = f.r[q], I = f.i[q];
                    float a, b, c = 0.f, e = 0.f;   // first signal (a, c), second signal (b, e)
                    if (!ODD && q == 0) {
                        a = bin_mag<EN>(fmaf(R.x, R.x, (1.f - pk) * I.x * I.x));   // bin 0
                        b = bin_mag<EN>(pk * I.x * I.x);
                        c = bin_mag<EN>(fmaf(R.y, R.y, (1.f - pk) * I.y * I.y));   // bin n/2
                        e = bin_mag<EN>(pk * I.y * I.y);
                        s[0] = a;
                        s[M / 2] = c;
#pragma unroll
                        for (int m = 0; m < 3; ++m) {
                            acc[j][m] = fmaf(__ldg(wb + m * W::H * N), b, acc[j][m]);
                            acc[j][m] = fmaf(__ldg(wb + (m * W::H + N / 2) * N), e, acc[j][m]);
                        }
                    } else {
                        const float r1 = fmaf(pk, R.y, R.x), i1 = fmaf(-pk, I.y, I.x);
                        const float r2 = fmaf(pk, R.x, (1.f - 2.f * pk) * R.y), i2 = fmaf(pk, I.x, I.y);
                        a = bin_mag<EN>(fmaf(r1, r1, i1 * i1));
                        b = bin_mag<EN>(fmaf(r2, r2, i2 * i2));
                        s[q] = a;
#pragma unroll
                        for (int m = 0; m < 3; ++m)
                            acc[j][m] = fmaf(__ldg(wb + (m * W::H + B::ky(q, N)) * N), b, acc[j][m]);
                    }
                }
            }
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                float2 e = make_float2(0.f, 0.f);
#pragma unroll
                for (int w = 0; w + 1 < NW; w += 2)
                    e = __ffma2_rn(make_float2(wt[m][w], wt[m][w + 1]), make_float2(s[w], s[w + 1]), e);
                float t = e.x + e.y;
                if (NW & 1) t = fmaf(wt[m][NW - 1], s[NW - 1], t);
                acc[j][m] += t;
            }
        }
        if (PART < RUN)   // the other half's sums where this half's were: the loop is not unrolled
#pragma unroll
            for (int j = 0; j < PART; ++j)
#pragma unroll
                for (int m = 0; m < 3; ++m) {
                    const float t = acc[j][m];
                    acc[j][m] = acc[RUN - PART + j][m];
                    acc[RUN - PART + j][m] = t;
                }
    }
}

// Sums of the RUN x 3 values over groups of L lanes, each step halving the values a lane keeps as long as they
// are whole outputs: lane l of the group ends with the kOuts outputs from kOuts (l / kShare) on, in v[0 .. 3 kOuts).
template <int L, int RUN> struct LaneSums {
    static constexpr int kShare = L > RUN ? L / RUN : 1;   // lanes that hold the same outputs
    static constexpr int kOuts = RUN * kShare / L;
    __device__ __forceinline__ static void run(const float (&acc)[RUN][3], int lane, float (&v)[3 * RUN]) {
#pragma unroll
        for (int i = 0; i < 3 * RUN; ++i) v[i] = acc[i / 3][i % 3];
        int cnt = 3 * RUN;
#pragma unroll
        for (int w = L / 2; w >= 1; w /= 2) {
            if (w >= kShare) {
                cnt /= 2;
                const bool up = lane & w;
#pragma unroll
                for (int i = 0; i < 3 * RUN / 2; ++i)
                    if (i < cnt) {
                        const float keep = up ? v[i + cnt] : v[i], send = up ? v[i] : v[i + cnt];
                        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, w);
                    }
            } else {
#pragma unroll
                for (int i = 0; i < 3 * kOuts; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], w);
            }
        }
    }
};

// A CTA's threads in groups that share G1 and meet at barriers of their own, so that the FFTs of one group's
// stage 2 fill the pipes under the square roots of the other's stage 3.  Whole multiples of four warps, the
// granule of register allocation.
//   n = 8: one group of 128 threads, 8 x0 and two runs; 39 KB and 128 registers, four CTAs per SM.
//   n = 16: two groups of 192 threads, 12 x0 and one run each; 176 KB and 168 registers, one CTA per SM.
// RUN = 16 outputs per run, or 4: four times the CTAs, each a third as long, for volumes that leave SMs idle (see
// short_runs).
template <int N> struct SGeo;
template <> struct SGeo<8> { static constexpr int RX = 8, RUNS = 2, GROUPS = 1, CTAS = 4; };
template <> struct SGeo<16> { static constexpr int RX = 12, RUNS = 1, GROUPS = 2, CTAS = 1; };
template <int N, int RUN> struct Slide : SGeo<N> {
    using S = SGeo<N>;
    static constexpr int GT = S::RX * N * S::RUNS, NT = GT * S::GROUPS, TILES = N / 2;
    static constexpr int BYG = S::RUNS * RUN, BY = BYG * S::GROUPS;
    static constexpr int XH = S::RX + N - 1, YH = BY + N - 1;   // halo
    static constexpr int YG = BYG + N - 1;   // odd: rows YG float2 apart meet no bank conflict
    static constexpr size_t G1 = (size_t)TILES * XH * YH, G2 = (size_t)S::RX * N * YG;
    static constexpr size_t SMEM = (G1 + S::GROUPS * G2) * sizeof(float2);
    static_assert(NT % 128 == 0 && GT % 32 == 0 && SMEM * S::CTAS <= 227 * 1024, "geometry");
};

// The value a brick of RX x BY outputs is staged minus: the smallest finite one in magnitude of a few voxels of which every
// window of the brick holds one.  (The brick's first voxel where all windows hold that; else, since RX <= n, one n/2 - 1
// past its first x0 and past every n-th output along y, clamped into the volume.)  The value is then never larger than the
// window's own largest sample, and an outlier costs no precision to the windows that do not hold it: a first voxel of 1e6
// in unit noise moved features up to 12 positions away by 1e-2.  0 where none is finite: then every window holds one that
// is not.
template <int N, int RX, int BY>
__device__ __forceinline__ float brick_shift(const float* __restrict__ V, int X, int Y, int t0, int xb, int yb) {
    static_assert(RX <= N, "a voxel of each window");
    constexpr int OX = RX - 1 <= N / 2 ? 0 : N / 2 - 1, OY = BY - 1 <= N / 2 ? 0 : N / 2 - 1;
    const float* row = V + ((size_t)t0 * X + min(X - 1, xb + OX)) * Y;
    float s = 0.f, least = INFINITY;
#pragma unroll
    for (int i = 0; i < BY; i += N) {
        const float v = yb + i < Y ? __ldg(row + min(Y - 1, yb + i + OY)) : INFINITY;
        if (fabsf(v) < least) {   // (false for a NaN)
            s = v;
            least = fabsf(v);
        }
    }
    return s;
}

// Halo position (x, y) of the brick: the n samples of its column along t, minus vshift.  s_gt: the planes of the n taps by
// the border extension (each column of a brick at the volume's first or last planes would find them again).
template <int N>
__device__ __forceinline__ void load_column(const float* __restrict__ V, int T, int X, int Y, int t0,
                                            const int* __restrict__ s_gt, int gx, int gy, float vshift, float (&v)[N]) {
    const bool in = (gx | gy) >= 0;
    const float* p = V + (in ? (size_t)gx * Y + gy : 0);
    const size_t plane = (size_t)X * Y;
    if (t0 - N / 2 >= 0 && t0 + N / 2 <= T) {
        p += (size_t)(t0 - N / 2) * plane;
#pragma unroll
        for (int u = 0; u < N; ++u) v[u] = (in ? __ldg(p + u * plane) : 0.f) - vshift;
    } else {
#pragma unroll
        for (int u = 0; u < N; ++u) {
            const int gt = s_gt[u];
            v[u] = (in && gt >= 0 ? __ldg(p + gt * plane) : 0.f) - vshift;
        }
    }
}

template <int N, bool EN, int RUN>
__global__ void __launch_bounds__(Slide<N, RUN>::NT, SGeo<N>::CTAS)
k1_slide(const float* __restrict__ V, float* __restrict__ E, int T, int X, int Y, int bnd,
         const float* __restrict__ wtab) {
    using G = Slide<N, RUN>;
    constexpr int RX = G::RX, XH = G::XH, YH = G::YH, YG = G::YG;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, grp = tid / G::GT, gt = tid % G::GT;
    float2* s_g1 = reinterpret_cast<float2*>(smem_raw);   // [tile][x][y]
    float2* s_g2 = s_g1 + G::G1 + grp * G::G2;            // [x0][k_x][y] of the group's current tile
    auto group_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(G::GT) : "memory"); };
    const int yb = blockIdx.x * G::BY, xb = blockIdx.y * RX, t0 = blockIdx.z;
    __shared__ int s_gt[N];
    if (tid < N) s_gt[tid] = ext_index(t0 - N / 2 + tid, T, bnd);
    __syncthreads();
    const float vshift = brick_shift<N, RX, G::BY>(V, X, Y, t0, xb, yb);

    for (int it = tid; it < XH * YH; it += G::NT) {
        const int x = it / YH, y = it - x * YH;
        float v[N];
        float2 o[N / 2];
        load_column<N>(V, T, X, Y, t0, s_gt, ext_index(xb - N / 2 + x, X, bnd), ext_index(yb - N / 2 + y, Y, bnd),
                       vshift, v);
        f32::rfft<N>(v, o);
#pragma unroll
        for (int k = 0; k < N / 2; ++k) s_g1[(size_t)k * XH * YH + it] = o[k];
    }

    __syncthreads();
    const int kx = gt % N, x0l = (gt / N) % RX, run = gt / (N * RX);
    float acc[RUN][3];
#pragma unroll
    for (int j = 0; j < RUN; ++j) acc[j][0] = acc[j][1] = acc[j][2] = 0.f;
    for (int tile = 0; tile < G::TILES; ++tile) {
        for (int it = gt; it < RX * YG; it += G::GT) {
            const int x = it / YG, y = it - x * YG;
            const float2* src = s_g1 + ((size_t)tile * XH + x) * YH + grp * G::BYG + y;
            float2 v[N];
#pragma unroll
            for (int u = 0; u < N; ++u) v[u] = src[u * YH];
            f32::fft<N>(v);
            float2* dst = s_g2 + (size_t)x * N * YG + y;
            if (tile != 0) {
#pragma unroll
                for (int k = 0; k < N; ++k) dst[k * YG] = v[f32::fft_pos<N>(k)];
            } else {
#pragma unroll
                for (int k = 0; k < N; ++k) dst[k * YG] = f32::tile0_row<N>(v, k);
            }
        }
        group_sync();
        slide_tile<N, N, false, EN, RUN>(s_g2 + ((size_t)x0l * N + kx) * YG + run * RUN, wtab, tile, kx, acc);
        if (tile + 1 < G::TILES) group_sync();   // the group's G2 is read
    }
    using LS = LaneSums<N, RUN>;
    float v[3 * RUN];
    LS::run(acc, kx, v);
    const size_t NV = (size_t)T * X * Y;
    const int x = xb + x0l;
#pragma unroll
    for (int i = 0; i < LS::kOuts; ++i) {
        const int y = yb + grp * G::BYG + run * RUN + LS::kOuts * (kx / LS::kShare) + i;
        if (kx % LS::kShare == 0 && x < X && y < Y) {
            float* e = E + ((size_t)t0 * X + x) * Y + y;
#pragma unroll
            for (int m = 0; m < 3; ++m) e[m * NV] = v[3 * i + m];
        }
    }
}

// ---- n = 32 --------------------------------------------------------------------------------------
// One CTA of 12 warps per SM: 6 x0, 16 outputs; warp = (x0, parity of k_y), lane = k_x.  G1 holds four of the 16
// tiles at a time (all of them would take 223 KB), so the columns are read from L2 four times and their bins formed as
// direct sums over the samples folded about the window's middle (32 multiplies a bin).  G2 is double-buffered: between two
// barriers every warp runs stage 3 of one tile and stage 2 of the next, half of the warps in either order, so that
// the FFTs of some fill the pipes under the square roots of the others.
namespace w32 {
constexpr int N = 32, RUN = 16, RX = 6, BY = RUN, XH = RX + N - 1, YH = BY + N - 1, NT = 384, GT = 4;
constexpr size_t G1 = (size_t)GT * XH * YH, G2 = (size_t)RX * N * YH;
constexpr size_t SMEM = (G1 + 2 * G2) * sizeof(float2);
static_assert(RX * N * 2 == NT && SMEM <= 226 * 1024, "geometry");

// G1 of tiles T0 .. T0 + 3 at one position from its samples: with s_u = v_u + v_{32-u}, d_u = v_u - v_{32-u},
// bin k = sum_u s_u cos(2 pi k u / 32) - i sum_u d_u sin(2 pi k u / 32).  Tile 0: (bin 0, bin 16).
template <int T0>
__device__ __forceinline__ void tiles4(const float (&v)[N], float2* dst, int plane) {
    float s[17], d[16];
    s[0] = v[0];
    s[16] = v[16];
#pragma unroll
    for (int u = 1; u < 16; ++u) {
        s[u] = v[u] + v[N - u];
        d[u] = v[u] - v[N - u];
    }
#pragma unroll
    for (int i = 0; i < GT; ++i) {
        const int k = T0 + i;
        float re = 0.f, im = 0.f;
        if (k == 0) {
            float a = s[0] + s[16], b = 0.f;   // even and odd samples
#pragma unroll
            for (int u = 2; u < 16; u += 2) a += s[u];
#pragma unroll
            for (int u = 1; u < 16; u += 2) b += s[u];
            re = a + b;
            im = a - b;
        } else {
            re = (k & 1) ? s[0] - s[16] : s[0] + s[16];
#pragma unroll
            for (int u = 1; u < 16; ++u) {
                re = fmaf(s[u], f32::cos32(k * u), re);
                im = fmaf(d[u], -f32::sin32(k * u), im);
            }
        }
        dst[i * plane] = make_float2(re, im);
    }
}
}  // namespace w32

template <bool EN>
__global__ void __launch_bounds__(w32::NT, 1)
k1_slide32(const float* __restrict__ V, float* __restrict__ E, int T, int X, int Y, int bnd,
           const float* __restrict__ wtab) {
    using namespace w32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* s_g1 = reinterpret_cast<float2*>(smem_raw);   // [4 tiles][x][y]
    float2* s_g2 = s_g1 + G1;                             // [2][x0][k_x][y]
    __shared__ float s_odd[RX][3][RUN];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int yb = blockIdx.x * BY, xb = blockIdx.y * RX, t0 = blockIdx.z;
    __shared__ int s_gt[N];
    if (tid < N) s_gt[tid] = ext_index(t0 - N / 2 + tid, T, bnd);
    __syncthreads();
    const float vshift = brick_shift<N, RX, BY>(V, X, Y, t0, xb, yb);
    const int x0l = warp >> 1, odd = warp & 1;

    auto stage1 = [&](int g) {
        for (int it = tid; it < XH * YH; it += NT) {
            const int x = it / YH, y = it - x * YH;
            float v[N];
            load_column<N>(V, T, X, Y, t0, s_gt, ext_index(xb - N / 2 + x, X, bnd), ext_index(yb - N / 2 + y, Y, bnd),
                           vshift, v);
            if (g == 0) tiles4<0>(v, s_g1 + it, XH * YH);
            else if (g == 1) tiles4<4>(v, s_g1 + it, XH * YH);
            else if (g == 2) tiles4<8>(v, s_g1 + it, XH * YH);
            else tiles4<12>(v, s_g1 + it, XH * YH);
        }
    };
    auto stage2 = [&](int tile) {
        float2* out = s_g2 + (size_t)(tile & 1) * G2;
        for (int it = tid; it < RX * YH; it += NT) {
            const int x = it / YH, y = it - x * YH;
            const float2* src = s_g1 + ((size_t)(tile % GT) * XH + x) * YH + y;
            float2 v[N];
#pragma unroll
            for (int u = 0; u < N; ++u) v[u] = src[u * YH];
            f32::fft<N>(v);
            float2* dst = out + (size_t)x * N * YH + y;
            if (tile != 0) {
#pragma unroll
                for (int k = 0; k < N; ++k) dst[k * YH] = v[f32::fft_pos<N>(k)];
            } else {
#pragma unroll
                for (int k = 0; k < N; ++k) dst[k * YH] = f32::tile0_row<N>(v, k);
            }
        }
    };
    float acc[RUN][3];
#pragma unroll
    for (int j = 0; j < RUN; ++j) acc[j][0] = acc[j][1] = acc[j][2] = 0.f;
    auto stage3 = [&](int tile) {
        const float2* g = s_g2 + (size_t)(tile & 1) * G2 + ((size_t)x0l * N + lane) * YH;
        if (odd) slide_tile<N, 16, true, EN, RUN>(g, wtab, tile, lane, acc);
        else slide_tile<N, 16, false, EN, RUN>(g, wtab, tile, lane, acc);
    };

    stage1(0);
    __syncthreads();
    stage2(0);
    __syncthreads();
    for (int tile = 0; tile < N / 2; ++tile) {
        const bool more = tile + 1 < N / 2;
        if (more && (tile + 1) % GT == 0) {   // the next four tiles' G1 (their predecessors' stage 2 is done)
            stage1((tile + 1) / GT);
            __syncthreads();
        }
        const bool early = (warp >> 2) & 1;   // per scheduler, warps of both orders
        if (more && early) stage2(tile + 1);
        stage3(tile);
        if (more && !early) stage2(tile + 1);
        __syncthreads();
    }
    using LS = LaneSums<16, RUN>;
    static_assert(LS::kOuts == 1, "an output per lane");
    float v[3 * RUN];
    LS::run(acc, lane & 15, v);
    const int o = (lane & 15) / LS::kShare;
#pragma unroll
    for (int m = 0; m < 3; ++m) v[m] += __shfl_xor_sync(0xffffffffu, v[m], 16);
    const bool writer = lane < 16 && lane % LS::kShare == 0;
    if (odd && writer)
#pragma unroll
        for (int m = 0; m < 3; ++m) s_odd[x0l][m][o] = v[m];
    __syncthreads();
    const size_t NV = (size_t)T * X * Y;
    const int x = xb + x0l, y = yb + o;
    if (!odd && writer && x < X && y < Y) {
        float* e = E + ((size_t)t0 * X + x) * Y + y;
#pragma unroll
        for (int m = 0; m < 3; ++m) e[m * NV] = v[m] + s_odd[x0l][m][o];
    }
}

constexpr int kLong = 16, kShort = 4;   // outputs per run

// Runs of 4 where runs of 16 would fill less than half of the GPU's resident CTAs: a CTA is then a chain of
// dependent stages with nothing beside it, and a short run's takes less than half of the time: n = 8, 10 x 9 x 37
// 18.7 us long, 9.3 short, 32^3 18.9 and 12.5; n = 16, 24^3 71.9 and 28.9 (from 28^3 on the long runs, 72.0 us for one
// wave of either size; n = 32, whose first stage does not shrink with the run, 12 x 16 x 20 235 and 243: it keeps the long runs).
bool short_runs(long long ctas, int per_sm) { return 2 * ctas <= (long long)per_sm * device_sms(); }

template <int N, bool EN, int RUN> cudaError_t prepare_one() {
    return cudaFuncSetAttribute(k1_slide<N, EN, RUN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)Slide<N, RUN>::SMEM);
}
template <int N> cudaError_t prepare_n() {
    cudaError_t e = prepare_one<N, false, kLong>();
    if (e == cudaSuccess) e = prepare_one<N, true, kLong>();
    if (e == cudaSuccess) e = prepare_one<N, false, kShort>();
    if (e == cudaSuccess) e = prepare_one<N, true, kShort>();
    return e;
}

template <int N, int RUN>
void launch_run(const float* wtab, const float* V, float* E, int T, int X, int Y, int bnd, int feat, cudaStream_t s) {
    using G = Slide<N, RUN>;
    const dim3 grid((Y + G::BY - 1) / G::BY, (X + G::RX - 1) / G::RX, T);
    if (feat == 1) k1_slide<N, true, RUN><<<grid, G::NT, G::SMEM, s>>>(V, E, T, X, Y, bnd, wtab);
    else k1_slide<N, false, RUN><<<grid, G::NT, G::SMEM, s>>>(V, E, T, X, Y, bnd, wtab);
}
template <int N>
void launch_n(const float* wtab, const float* V, float* E, int T, int X, int Y, int bnd, int feat, cudaStream_t s) {
    using G = Slide<N, kLong>;
    const long long ctas = (long long)((Y + G::BY - 1) / G::BY) * ((X + G::RX - 1) / G::RX) * T;
    if (short_runs(ctas, G::CTAS)) launch_run<N, kShort>(wtab, V, E, T, X, Y, bnd, feat, s);
    else launch_run<N, kLong>(wtab, V, E, T, X, Y, bnd, feat, s);
}

// Weights of the tiles' rows (spectra_f32_fft.cuh): multiplicity and 1/n^3 folded in.
template <int N, bool EN> void fill_table(float* out) {
    using W = WGeo<N>;
    constexpr int H = W::H;
    const float inv = 1.f / (float)(N * N * N);
    for (size_t i = 0; i < W::FLOATS; ++i) out[i] = 0.f;
    for (int tile = 0; tile < W::TILES; ++tile)
        for (int row = 0; row < N; ++row) {
            const bool packed = tile == 0 && (row == 0 || row == N / 2);
            const int i = tile == 0 && row > N / 2 ? N / 2 : tile;
            const int j = row <= N / 2 ? row : N - row;   // |k_x|
            for (int k = 0; k < H; ++k) {
                // packed rows: the pair gives twice F of each signal, standing for the bins k and n - k
                const float mult = !packed ? 2.f : (EN && k != 0 && k != N / 2 ? 0.5f : 1.f);
                float w[3];
                f32::bin_weights<EN>(i, j, k, mult * inv, w[0], w[1], w[2]);
                for (int m = 0; m < 3; ++m) out[tile * W::TILE + (m * H + k) * N + row] = w[m];
                if (tile == 0) {   // the second value of the pair: the packed rows' k_t = n/2, else the bin n - k
                    f32::bin_weights<EN>(packed ? N / 2 : i, j, k, mult * inv, w[0], w[1], w[2]);
                    for (int m = 0; m < 3; ++m) out[W::TILES * W::TILE + (m * H + k) * N + row] = w[m];
                }
            }
        }
}

}  // namespace

bool f32_slide_supported(int n) { return n == 8 || n == 16 || n == 32; }

size_t f32_slide_table_floats(int n) {
    return n == 8 ? WGeo<8>::FLOATS : n == 16 ? WGeo<16>::FLOATS : n == 32 ? WGeo<32>::FLOATS : 0;
}

void f32_slide_table_fill(int n, int feat, float* out) {
    if (n == 8) feat == 1 ? fill_table<8, true>(out) : fill_table<8, false>(out);
    if (n == 16) feat == 1 ? fill_table<16, true>(out) : fill_table<16, false>(out);
    if (n == 32) feat == 1 ? fill_table<32, true>(out) : fill_table<32, false>(out);
}

cudaError_t spectra_f32_slide_prepare(int n) {
    if (n == 8) return prepare_n<8>();
    if (n == 16) return prepare_n<16>();
    if (n != 32) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(k1_slide32<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)w32::SMEM);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k1_slide32<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)w32::SMEM);
}

cudaError_t spectra_f32_slide_launch(int n, const float* wtab, const float* V, float* E, int T, int X, int Y, int bnd,
                                     int feat, cudaStream_t s) {
    if (T > 65535 || X > 65535) return cudaErrorInvalidConfiguration;
    if (n == 8) {
        launch_n<8>(wtab, V, E, T, X, Y, bnd, feat, s);
    } else if (n == 16) {
        launch_n<16>(wtab, V, E, T, X, Y, bnd, feat, s);
    } else if (n == 32) {
        const dim3 grid((Y + w32::BY - 1) / w32::BY, (X + w32::RX - 1) / w32::RX, T);
        if (feat == 1) k1_slide32<true><<<grid, w32::NT, w32::SMEM, s>>>(V, E, T, X, Y, bnd, wtab);
        else k1_slide32<false><<<grid, w32::NT, w32::SMEM, s>>>(V, E, T, X, Y, bnd, wtab);
    } else {
        return cudaErrorInvalidValue;
    }
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace sal

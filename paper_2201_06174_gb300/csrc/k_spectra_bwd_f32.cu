// K5-F32: adjoint of the local-spectrum feature step (the backward of Sec. 2 steps 1-3).
//
// For L = sum_p sum_m gE_m[p] E_m[p] with E_m[p] = sum_{k in half} wt_m(k) |F_p[k]| (wt holds
// r_m of Eq. 1, the Hermitian multiplicity of k_t and 1/n^3), the gradient with respect to the
// (extended) input is
//   gVext[p + u - n/2] += Re sum_{k in half} h(u) exp(+2 pi i k.u / n) Gamma_p[k],
//   Gamma_p[k] = (sum_m gE_m[p] wt_m(k)) F_p[k] / |F_p[k]|,
// with Gamma = 0 at DC and where F_p[k] = 0 (|F| has no direction there: the zero subgradient), i.e. the
// transposes of the three sliding DFT stages applied to Gamma in reverse order.
//
// The direction F / |F| is ill-conditioned for small |F|: FP32 computes F to about 2^-26 of the window's
// L1 norm A_p = sum_u |h(u) Vext[p + u - n/2]| (which bounds every |F_p[k]|), so a bin with |F| near that
// level has no usable FP32 direction.  Such bins are resolved exactly:
//   - bins that vanish for every input, because the border extension makes the coefficient of every
//     source sample of one axis vanish (a mirror-symmetric window along an axis zeroes its Nyquist bin,
//     a window folded onto few samples zeroes more), are found on the host by integer arithmetic on the
//     window's index map (axis_vanish_mask) and take Gamma = 0;
//   - every other bin with FP32 |F| <= 2^-16 A_p and a non-zero weight is recomputed by one warp as a
//     direct sum over its cube in float-float arithmetic (pairs of FP32 values, error about 2^-46 A_p;
//     resolve_small_bins), and takes Gamma = 0 if |F| <= 2^-36 A_p, else its float-float direction.
// Bins above 2^-16 A_p carry an FP32 direction error of at most about 2^-10.
// Spectra are recomputed brick by brick (the forward stages of K1), never stored.
//
// One CTA = one brick (t0, x0, y_start .. y_start+BY-1), same mapping as K1:
//   1. stage brick, forward stages 1 and 2 (shared with K1);
//   2. per (row, y0): forward stage 3 -> Gamma -> inverse DFT along y (pairing k, n-k), added
//      into a private accumulation window of the thread (thread-interleaved shared memory);
//   3. windows of the y-chunks summed into Gamma_G2[k_t][k_x][y];
//   4. adjoint of stage 2 (x) -> Gamma_G1[k_t][u_x][y];
//   5. adjoint of stage 1 (t), real part -> the brick's block [u_t][u_x][y] of gVext, written to
//      scratch; a separate gather kernel sums the overlapping blocks in a fixed order.
#include <cooperative_groups.h>

#include <algorithm>

#include "spectra_f32_exact.cuh"

namespace sal {
namespace {

using f32::Exact2f;
using f32::FF;
using f32::ff_add;
using f32::ff_gather;
using f32::ff_mul;
using f32::ff_mul1;
using f32::kSmallBin;
using f32::kZeroBin;
using f32::make_exact2f;
using f32::make_vanish_tab;
using f32::Tw;
using f32::vanish_mask;
using f32::VanishTab;

constexpr int kListQ = 32;   // small bins a CTA may hand to the listed-bin passes (more: it resolves them itself)
// Layout of the listed-bin scratch of one launch of ncta CTAs (ints): [0] the number of listed bins, [4 ..)
// the work list (cta << 5 | entry, in no particular order), then per CTA kListStride ints: [0] its count,
// [1 .. Q] its entries (owner | output << 10 | bin << 14, in the in-kernel resolve's order), [1 + Q ..) the
// (Re, Im) of each entry's Gamma, written by the exact pass.
constexpr int kListStride = 1 + 3 * kListQ;
__host__ __device__ constexpr size_t list_cta_offset(long long ncta) { return 4 + (size_t)ncta * kListQ; }

template <int N> struct BCfg;
template <> struct BCfg<2>  { static constexpr int BY = 32, YC = 1, MINB = 4; };
template <> struct BCfg<4>  { static constexpr int BY = 32, YC = 2, MINB = 4; };
template <> struct BCfg<8>  { static constexpr int BY = 32, YC = 4, MINB = 2; };
template <> struct BCfg<16> { static constexpr int BY = 16, YC = 8, MINB = 2; };

template <int N> struct BGeo {
    static constexpr int H = N / 2 + 1;
    static constexpr int BY = BCfg<N>::BY;
    static constexpr int YC = BCfg<N>::YC;
    static constexpr int ROWS = H * N;
    static constexpr int NT = ROWS * (BY / YC);
    using B = f32::Brick<N, BY, NT>;
    static constexpr int YH = B::YH;
    static constexpr int WIN = YC + N - 1;                       // private window (complex values)
    static constexpr size_t IN_BYTES = (size_t)B::IN_FLOATS * 4;
    static constexpr size_t G_BYTES = (size_t)B::G_FLOAT2 * 8;
    static constexpr size_t WIN_BYTES = (size_t)NT * WIN * 8;
    static constexpr size_t A0 = IN_BYTES + G_BYTES;
    static constexpr size_t A_BYTES = A0 > WIN_BYTES ? A0 : WIN_BYTES;   // s_in+s_g1 | windows | Gamma_G1
    static constexpr size_t SMALL_OFF = A_BYTES + G_BYTES + (size_t)4 * BY * 4 + (size_t)YH * 4;
    // [YC][NT] uint16 masks of the small bins each thread leaves to the exact recompute, then the source
    // rows of the cube along t and x ([N] + [N] ints, -1 outside a zero-extended volume)
    static constexpr size_t IDX_OFF = (SMALL_OFF + (size_t)YC * NT * 2 + 15) / 16 * 16;
    static constexpr size_t WB_OFF = IDX_OFF + (size_t)2 * N * 4;   // [NT / 32] owners of small bins, per warp
    static constexpr size_t SMEM = WB_OFF + (size_t)(NT / 32 + 1) * 4;   // + the CTA's list decision
    static_assert(N <= 16, "16-bit masks of small bins");
    static constexpr int SLICE = (N * YH + 3) / 4 * 4;           // u_t slices of the block, 16-byte aligned
    static constexpr int BLOCK_FLOATS = N * SLICE;               // scratch block per CTA
    static_assert(BY % YC == 0 && NT <= 1024, "geometry");
};

// The small bins left by step 2 (s_small[yi][owner] bit k_y: output yi of the owner's run, bin k_y of its
// (k_t, k_x) row), each owner's bins by one warp (the owners dealt round-robin to the CTA's warps in thread
// order): the lanes split the n^3 terms of the direct sum
// F = sum_u h(u) Vext[p + u - n/2] w^(k.u) (each lane a fixed u_y, four independent float-float
// accumulators, the loads of four terms issued before their arithmetic) and reduce it; Gamma = rho F / |F|
// (0 if max(|Re F|, |Im F|) <= 2^-36 A_p) and its inverse DFT along y, h(u) Gamma exp(+2 pi i k_y u / n),
// go into the owner's private window.
template <int N, int NT, int YC, int BY, int H, int ROWS>
__device__ __noinline__ void resolve_small_bins(const float* __restrict__ V, int X, int Y, int bnd, int y_start,
                                                int taper, const uint16_t* s_small, const int* s_src, float2* s_win,
                                                const float* s_ge, const float* s_l1,
                                                const float* __restrict__ wtab, const Tw<N>& tw,
                                                const Exact2f<N>& ex, unsigned* s_wbits) {
    constexpr int N3 = N * N * N, PER = N3 >= 32 ? N3 / 32 : 1, STEP = 32 / N;   // terms per lane, (ut, ux) step
    constexpr int U = PER >= 4 ? 4 : PER;                                          // independent accumulators
    const int tid = threadIdx.x, lane = tid & 31;
    // lane's fixed u_y and its first (u_t, u_x) pair: term e = lane + 32 i has u_y = lane % N and
    // (u_t, u_x) = divmod(lane / N + STEP i, N)
    const int uy = lane % N, r0 = lane / N;
    const bool live = lane < N3;   // n = 2: 8 terms, lanes 8.. idle
    // the owners (threads with small bins) in thread order, dealt round-robin to the CTA's warps: an owner's bins
    // are processed by one warp in a fixed order (the same sums in the same order whichever warp it is), and
    // owners that cluster in one warp no longer hold the rest of the CTA at the next barrier
    constexpr int NW = NT / 32;
    const int warp = tid >> 5;
    bool mine = false;
    for (int yi = 0; yi < YC; ++yi) mine = mine || s_small[yi * NT + tid] != 0;
    const unsigned wb = __ballot_sync(0xffffffffu, mine);
    if (lane == 0) s_wbits[warp] = wb;
    __syncthreads();   // every owner's masks and every warp's owner bits visible
    int idx = 0;   // index of the next owner in thread order
    for (int w = 0; w < NW; ++w) {
        unsigned todo = s_wbits[w];
        while (todo) {
            const int o = 32 * w + __ffs(todo) - 1;
            todo &= todo - 1;
            if (idx++ % NW != warp) continue;
            const int row = o % ROWS, kt = row / N, kx = row % N, ych = o / ROWS;
            for (int yi = 0; yi < YC; ++yi) {
                unsigned msk = s_small[yi * NT + o];
                const int yl = ych * YC + yi;
                const int gy = ext_index(y_start + yl - N / 2 + uy, Y, bnd);
                while (msk) {
                    const int ky = __ffs(msk) - 1;
                    msk &= msk - 1;
                    FF re[U], im[U];
    #pragma unroll
                    for (int a = 0; a < U; ++a) re[a] = im[a] = FF{0.f, 0.f};
                    const FF hy = {ex.hh[uy], ex.hl[uy]};
                    for (int i0 = 0; i0 < PER; i0 += U) {
                        float v[U];
                        int ph[U];
                        FF h2[U];
    #pragma unroll
                        for (int a = 0; a < U; ++a) {   // loads first, then the arithmetic
                            const int rr = live ? r0 + STEP * (i0 + a) : 0, ut = rr / N, ux = rr % N;
                            const int gt = s_src[ut], gx = s_src[N + ux];
                            v[a] = (live && (gt | gx | gy) >= 0) ? __ldg(V + ((size_t)gt * X + gx) * Y + gy) : 0.f;
                            ph[a] = (kt * ut + kx * ux + ky * uy) % N;
                            h2[a] = taper ? ff_mul(FF{ex.hh[ut], ex.hl[ut]}, FF{ex.hh[ux], ex.hl[ux]}) : FF{1.f, 0.f};
                        }
    #pragma unroll
                        for (int a = 0; a < U; ++a) {
                            FF c = {ex.ch[ph[a]], ex.cl[ph[a]]}, sn = {-ex.sh[ph[a]], -ex.sl[ph[a]]};
                            if (taper) {
                                const FF h3 = ff_mul(h2[a], hy);
                                c = ff_mul(h3, c);
                                sn = ff_mul(h3, sn);
                            }
                            re[a] = ff_add(re[a], ff_mul1(v[a], c));
                            im[a] = ff_add(im[a], ff_mul1(v[a], sn));
                        }
                    }
    #pragma unroll
                    for (int a = 1; a < U; ++a) {
                        re[0] = ff_add(re[0], re[a]);
                        im[0] = ff_add(im[0], im[a]);
                    }
                    FF fre = re[0], fim = im[0];
    #pragma unroll
                    for (int d = 16; d > 0; d >>= 1) {
                        const FF r2 = {__shfl_xor_sync(0xffffffffu, fre.hi, d), __shfl_xor_sync(0xffffffffu, fre.lo, d)};
                        const FF i2 = {__shfl_xor_sync(0xffffffffu, fim.hi, d), __shfl_xor_sync(0xffffffffu, fim.lo, d)};
                        fre = ff_add(fre, r2);
                        fim = ff_add(fim, i2);
                    }
                    const float mx = fmaxf(fabsf(fre.hi), fabsf(fim.hi));
                    if (mx > kZeroBin * s_l1[yl] && lane < N) {
                        const int k = ky <= N / 2 ? ky : N - ky;
                        const float rho = fmaf(s_ge[yl], __ldg(wtab + k * ROWS + row),
                                               fmaf(s_ge[BY + yl], __ldg(wtab + (H + k) * ROWS + row),
                                                    s_ge[2 * BY + yl] * __ldg(wtab + (2 * H + k) * ROWS + row)));
                        const float fr = fre.hi / mx, fi = fim.hi / mx;      // scaled first: no underflow
                        const float sc = rho / sqrtf(fmaf(fr, fr, fi * fi));
                        const float gr = sc * fr, gi = sc * fi;
                        const int u = lane;
                        const float c = tw.c[k][u], sn = ky <= N / 2 ? tw.s[k][u] : -tw.s[k][u];
                        float2* w = s_win + (yi + u) * NT + o;
                        float2 acc = *w;
                        acc.x += gr * c - gi * sn;
                        acc.y += gr * sn + gi * c;
                        *w = acc;
                    }
                    __syncwarp();
                }
            }
        }
    }
}

// The CTA's small bins as a list for the listed-bin pass: entries (owner, output, bin) in the order the
// in-kernel resolve would take them (owners in thread order, then outputs, then bins), list[0] = their
// count.  Returns (CTA-uniform) whether the list holds them all; a CTA with more than kListQ writes a count
// of 0 and resolves its bins itself.  Contains one __syncthreads.
template <int NT, int YC>
__device__ bool list_small_bins(const uint16_t* s_small, unsigned* s_wbits, int* __restrict__ list,
                                int* __restrict__ work, int* __restrict__ nwork, long long cta) {
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    bool mine = false;
    for (int yi = 0; yi < YC; ++yi) mine = mine || s_small[yi * NT + tid] != 0;
    const unsigned wb = __ballot_sync(0xffffffffu, mine);
    if (lane == 0) s_wbits[warp] = wb;
    __syncthreads();
    if (tid == 0) {
        int cnt = 0;
        for (int w = 0; w < NW; ++w) {
            for (unsigned todo = s_wbits[w]; todo; todo &= todo - 1) {
                const int o = 32 * w + __ffs(todo) - 1;
                for (int yi = 0; yi < YC; ++yi)
                    for (unsigned msk = s_small[yi * NT + o]; msk; msk &= msk - 1) {
                        if (cnt < kListQ) list[1 + cnt] = o | (yi << 10) | ((__ffs(msk) - 1) << 14);
                        ++cnt;
                    }
            }
        }
        const bool fits = cnt <= kListQ;
        list[0] = fits ? cnt : 0;
        s_wbits[NW] = fits ? 1u : 0u;
        if (fits && cnt > 0) {   // the exact pass takes the bins in any order: each writes its own slot
            const int base = atomicAdd(nwork, cnt);
            for (int e = 0; e < cnt; ++e) work[base + e] = (int)(cta << 5) | e;
        }
    }
    __syncthreads();
    return s_wbits[NW] != 0u;
}

// The listed bins' exact pass: one warp per listed bin (a grid-stride loop over the work list).  Each is
// recomputed exactly as the in-kernel resolve does (the direct sum F = sum_u h(u) Vext[...] w^(k.u) in
// float-float arithmetic, lanes splitting the n^3 terms; A_p = sum_u h(u) |Vext| alongside), and its
// Gamma = rho F / |F| (0 if max(|Re F|, |Im F|) <= 2^-36 A_p) is written to the bin's slot of its CTA's list.
template <int N>
__global__ void __launch_bounds__(256)
k5_listed_exact_f32(const float* __restrict__ V, const float* __restrict__ gE, int* __restrict__ lists,
                    long long ncta, int T, int X, int Y, int bnd, int t_begin, int t_step,
                    const float* __restrict__ wtab, int taper, const __grid_constant__ Exact2f<N> ex) {
    using G = BGeo<N>;
    constexpr int H = G::H, BY = G::BY, YC = G::YC, ROWS = G::ROWS;
    constexpr int N3 = N * N * N, PER = N3 >= 32 ? N3 / 32 : 1, STEP = 32 / N;
    constexpr int U = PER >= 4 ? 4 : PER;   // terms whose loads are issued together
    // the float-float constants in shared memory: the lanes index them by their own phase, which the
    // parameter space would serve one distinct address at a time
    __shared__ float s_ex[6][N];
    __shared__ int s_rows[8][2][N];   // per warp: the cube's source rows along t and x of its current bin
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < 6 * N; i += blockDim.x) {
        const int a = i / N, m = i % N;
        s_ex[a][m] = a == 0 ? ex.ch[m] : a == 1 ? ex.cl[m] : a == 2 ? ex.sh[m] : a == 3 ? ex.sl[m]
                   : a == 4 ? ex.hh[m] : ex.hl[m];
    }
    __syncthreads();
    const int nw = lists[0];
    const int* work = lists + 4;
    int* ctal = lists + list_cta_offset(ncta);
    const int nseg = (Y + BY - 1) / BY;
    const size_t NV = (size_t)T * X * Y;
    const int uy = lane % N, r0 = lane / N;
    const bool live = lane < N3;
    const int wstride = gridDim.x * (blockDim.x / 32);
    for (int w = blockIdx.x * (blockDim.x / 32) + wib; w < nw; w += wstride) {
        const int item = work[w];
        const long long cta = item >> 5;
        const int e = item & 31;
        int* L = ctal + cta * kListStride;
        const int ent = L[1 + e];
        const int y_start = (int)(cta % nseg) * BY;
        const int x0 = (int)((cta / nseg) % X);
        const int t0 = t_begin + (int)(cta / ((long long)nseg * X)) * t_step;
        const int o = ent & 1023, yi = (ent >> 10) & 15, ky = (ent >> 14) & 15;
        const int row = o % ROWS, kt = row / N, kx = row % N, ych = o / ROWS;
        const int yl = ych * YC + yi;
        const int gy = ext_index(y_start + yl - N / 2 + uy, Y, bnd);
        if (lane < 2 * N)
            s_rows[wib][lane / N][lane % N] = lane < N ? ext_index(t0 - N / 2 + lane, T, bnd)
                                                       : ext_index(x0 - N / 2 + lane - N, X, bnd);
        __syncwarp();
        const FF hy = {s_ex[4][uy], s_ex[5][uy]};
        FF re = {0.f, 0.f}, im = {0.f, 0.f};
        float a1 = 0.f;   // the window's L1 norm, FP32 (it only places the 2^-36 band)
        for (int i0 = 0; i0 < PER; i0 += U) {
            float v[U];
            int tx[U];
#pragma unroll
            for (int a = 0; a < U; ++a) {   // loads first
                const int rr = live ? r0 + STEP * (i0 + a) : 0, ut = rr / N, ux = rr % N;
                const int gt = s_rows[wib][0][ut], gx = s_rows[wib][1][ux];
                v[a] = (live && (gt | gx | gy) >= 0) ? __ldg(V + ((size_t)gt * X + gx) * Y + gy) : 0.f;
                tx[a] = rr;
            }
#pragma unroll
            for (int a = 0; a < U; ++a) {
                const int ut = tx[a] / N, ux = tx[a] % N;
                const int ph = (kt * ut + kx * ux + ky * uy) % N;
                FF c = {s_ex[0][ph], s_ex[1][ph]}, sn = {-s_ex[2][ph], -s_ex[3][ph]};
                if (taper) {
                    const FF h3 = ff_mul(ff_mul(FF{s_ex[4][ut], s_ex[5][ut]}, FF{s_ex[4][ux], s_ex[5][ux]}), hy);
                    c = ff_mul(h3, c);
                    sn = ff_mul(h3, sn);
                    a1 = fmaf(h3.hi, fabsf(v[a]), a1);
                } else {
                    a1 += fabsf(v[a]);
                }
                re = ff_add(re, ff_mul1(v[a], c));
                im = ff_add(im, ff_mul1(v[a], sn));
            }
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            const FF r2 = {__shfl_xor_sync(0xffffffffu, re.hi, d), __shfl_xor_sync(0xffffffffu, re.lo, d)};
            const FF i2 = {__shfl_xor_sync(0xffffffffu, im.hi, d), __shfl_xor_sync(0xffffffffu, im.lo, d)};
            re = ff_add(re, r2);
            im = ff_add(im, i2);
            a1 += __shfl_xor_sync(0xffffffffu, a1, d);
        }
        float gr = 0.f, gim = 0.f;
        const float mx = fmaxf(fabsf(re.hi), fabsf(im.hi));
        if (mx > kZeroBin * a1) {
            const int k = ky <= N / 2 ? ky : N - ky;
            const size_t gi = ((size_t)t0 * X + x0) * Y + y_start + yl;
            const float rho = fmaf(__ldg(gE + gi), __ldg(wtab + k * ROWS + row),
                                   fmaf(__ldg(gE + NV + gi), __ldg(wtab + (H + k) * ROWS + row),
                                        __ldg(gE + 2 * NV + gi) * __ldg(wtab + (2 * H + k) * ROWS + row)));
            const float fr = re.hi / mx, fi = im.hi / mx;      // scaled first: no underflow
            const float sc = rho / sqrtf(fmaf(fr, fr, fi * fi));
            gr = sc * fr;
            gim = sc * fi;
        }
        if (lane == 0) {
            float* gam = reinterpret_cast<float*>(L + 1 + kListQ);
            gam[2 * e] = gr;
            gam[2 * e + 1] = gim;
        }
        __syncwarp();   // the next bin rewrites this warp's source rows
    }
}

// The listed bins' apply pass: one warp per CTA of the main kernel's launch adds its listed bins, in list
// order, to the brick's block; the three adjoint stages of one bin are the outer product
//   block[u_t][u_x][y_l + u_y] += Re( Gamma h(u_t) h(u_x) h(u_y) e^{+2 pi i (k_t u_t + k_x u_x + k_y u_y) / n} ).
// Each block element is owned by one lane per bin; the warp syncs between bins (they overlap along y).
template <int N>
__global__ void __launch_bounds__(256)
k5_listed_apply_f32(float* __restrict__ blocks, const int* __restrict__ lists, long long ncta,
                    const __grid_constant__ Tw<N> tw) {
    using G = BGeo<N>;
    constexpr int YC = G::YC, YH = G::YH, ROWS = G::ROWS;
    constexpr int N3 = N * N * N, PER = N3 >= 32 ? N3 / 32 : 1, STEP = 32 / N;
    __shared__ float s_c[N / 2 + 1][N], s_s[N / 2 + 1][N];   // the lanes index them by their own taps
    for (int i = threadIdx.x; i < (N / 2 + 1) * N; i += blockDim.x) {
        s_c[i / N][i % N] = tw.c[i / N][i % N];
        s_s[i / N][i % N] = tw.s[i / N][i % N];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const long long cta = (long long)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    if (cta >= ncta) return;
    const int* L = lists + list_cta_offset(ncta) + cta * kListStride;
    const int cnt = L[0];
    if (cnt <= 0) return;
    const float* gam = reinterpret_cast<const float*>(L + 1 + kListQ);
    float* blk = blocks + cta * G::BLOCK_FLOATS;
    const int uy = lane % N, r0 = lane / N;
    const bool live = lane < N3;
    for (int e = 0; e < cnt; ++e) {
        const float gr = gam[2 * e], gim = gam[2 * e + 1];
        if (gr != 0.f || gim != 0.f) {   // warp-uniform
            const int ent = L[1 + e];
            const int o = ent & 1023, yi = (ent >> 10) & 15, ky = (ent >> 14) & 15;
            const int row = o % ROWS, kt = row / N, kx = row % N, ych = o / ROWS;
            const int yl = ych * YC + yi;
            // h(u) e^{+i theta} of each axis from the twiddle table (the taper is in it): bins above n/2 take the
            // conjugate of their mirror
            const int kxa = kx <= N / 2 ? kx : N - kx, kya = ky <= N / 2 ? ky : N - ky;
            const float sx = kx <= N / 2 ? 1.f : -1.f, sy = ky <= N / 2 ? 1.f : -1.f;
            const float eyr = s_c[kya][uy], eyi = sy * s_s[kya][uy];
            const float gyr = gr * eyr - gim * eyi, gyi = gr * eyi + gim * eyr;   // Gamma e_y
            constexpr int UB = PER >= 8 ? 8 : PER;   // block elements read, then written, together
            for (int i0 = 0; i0 < PER; i0 += UB) {
                float cur[UB];
                size_t off[UB];
#pragma unroll
                for (int a = 0; a < UB; ++a) {
                    const int rr = r0 + STEP * (i0 + a);
                    off[a] = (size_t)(rr / N) * G::SLICE + (rr % N) * YH + yl + uy;
                    cur[a] = (live && rr < N * N) ? blk[off[a]] : 0.f;
                }
#pragma unroll
                for (int a = 0; a < UB; ++a) {
                    const int rr = r0 + STEP * (i0 + a);
                    if (!live || rr >= N * N) continue;
                    const int ut = rr / N, ux = rr % N;
                    const float etr = s_c[kt][ut], eti = s_s[kt][ut];
                    const float exr = s_c[kxa][ux], exi = sx * s_s[kxa][ux];
                    const float txr = etr * exr - eti * exi, txi = etr * exi + eti * exr;
                    blk[off[a]] = cur[a] + (gyr * txr - gyi * txi);
                }
            }
        }
        __syncwarp();   // the next bin's window overlaps this one's along y
    }
}

// ---- Bricks of the sliding form with more small bins than it lists -------------------------------------------------
// Every small bin of such a brick from float-float spectra formed separably, as the FP32 ones are: G1 of four k_t at a time
// and G2 of all rows in shared memory, then 16 terms a bin instead of the direct sum's 4096 (n = 16).  The x0 of a brick are
// dealt to the CTAs of a cluster, which add their parts to the brick's block in the order of x0.
constexpr int kDenseRun = 16;      // outputs of a sliding brick along y
template <int N> struct DGeo {
    using G = BGeo<N>;
    static constexpr int XY = kDenseRun + N - 1;   // odd: rows XY float4 apart meet no bank conflict
    static constexpr int KG = 4;                   // k_t a group, in the FP32 G1's place
    static constexpr int CLUSTER = N == 8 ? 8 : 4;   // CTAs a brick's 16 (n = 16: 12) x0 are dealt to
    static constexpr size_t X2_OFF = (G::SMEM + 15) / 16 * 16;
    static constexpr size_t EX_OFF = X2_OFF + (size_t)G::ROWS * XY * 16;
    static constexpr size_t SMEM = EX_OFF + (size_t)4 * N * 4;
    static constexpr int CTAS = SMEM <= 100 * 1024 ? 2 : 1;   // per SM
    static_assert((size_t)KG * N * XY * 16 <= G::G_BYTES && G::IN_BYTES % 16 == 0 && SMEM <= 227 * 1024, "geometry");
};

// The float-float G2 of a staged brick (rect cube), [row][XY] as (re hi, re lo, im hi, im lo).  s_t: KG N XY float4.
template <int N>
__device__ void exact_rows(const float* s_in, float4* s_t, float4* s_x2, const float (*s_ex)[N]) {
    using G = BGeo<N>;
    using D = DGeo<N>;
    constexpr int XY = D::XY, NT = G::NT;
    for (int k0 = 0; k0 < G::H; k0 += D::KG) {
        const int items = min(D::KG, G::H - k0) * N * XY;
        for (int it = threadIdx.x; it < items; it += NT) {
            const int y = it % XY, ux = it / XY % N, kt = k0 + it / (XY * N);
            FF re = {0.f, 0.f}, im = {0.f, 0.f};
#pragma unroll
            for (int ut = 0; ut < N; ++ut) {
                const float v = s_in[(ut * N + ux) * G::YH + y];
                const int ph = (kt * ut) % N;
                ff_gather(re, v, s_ex[0][ph], s_ex[1][ph]);
                ff_gather(im, v, -s_ex[2][ph], -s_ex[3][ph]);
            }
            re = f32::ff_fast_two_sum(re.hi, re.lo);
            im = f32::ff_fast_two_sum(im.hi, im.lo);
            s_t[it] = make_float4(re.hi, re.lo, im.hi, im.lo);
        }
        __syncthreads();
        for (int it = threadIdx.x; it < items; it += NT) {
            const int y = it % XY, kx = it / XY % N, kl = it / (XY * N);
            FF re = {0.f, 0.f}, im = {0.f, 0.f};
#pragma unroll 4
            for (int ux = 0; ux < N; ++ux) {
                const float4 g = s_t[(kl * N + ux) * XY + y];
                const int ph = (kx * ux) % N;
                const FF c = {s_ex[0][ph], s_ex[1][ph]}, sn = {s_ex[2][ph], s_ex[3][ph]}, ns = {-sn.hi, -sn.lo};
                re = ff_add(re, ff_add(ff_mul(FF{g.x, g.y}, c), ff_mul(FF{g.z, g.w}, sn)));
                im = ff_add(im, ff_add(ff_mul(FF{g.z, g.w}, c), ff_mul(FF{g.x, g.y}, ns)));
            }
            s_x2[((k0 + kl) * N + kx) * XY + y] = make_float4(re.hi, re.lo, im.hi, im.lo);
        }
        __syncthreads();
    }
}

// F / |F| of bin k_y of the window whose n samples of G2 start at g; 0 where F is 0 in float-float arithmetic.
template <int N>
__device__ __noinline__ float2 exact_direction(const float4* g, int ky, float l1, const float (*s_ex)[N]) {
    FF re = {0.f, 0.f}, im = {0.f, 0.f};
#pragma unroll 4
    for (int u = 0; u < N; ++u) {
        const float4 v = g[u];
        const int ph = (ky * u) % N;
        const FF c = {s_ex[0][ph], s_ex[1][ph]}, sn = {s_ex[2][ph], s_ex[3][ph]}, ns = {-sn.hi, -sn.lo};
        re = ff_add(re, ff_add(ff_mul(FF{v.x, v.y}, c), ff_mul(FF{v.z, v.w}, sn)));
        im = ff_add(im, ff_add(ff_mul(FF{v.z, v.w}, c), ff_mul(FF{v.x, v.y}, ns)));
    }
    const float mx = fmaxf(fabsf(re.hi), fabsf(im.hi));
    if (!(mx > kZeroBin * l1)) return make_float2(0.f, 0.f);
    const float fr = re.hi / mx, fi = im.hi / mx;   // scaled first: no underflow
    const float s = 1.f / sqrtf(fmaf(fr, fr, fi * fi));
    return make_float2(s * fr, s * fi);
}

// Adjoint of stage 1 (t), real part, of the brick's Gamma_G1 [H][N][YH]: the block [u_t][u_x][y], slices `slice` and rows
// `pitch` floats apart, the first `ny` positions of each row; written, or added (ADD).
template <int N, bool ADD>
__device__ __forceinline__ void write_block(float* blk, size_t slice, int pitch, int ny, const Tw<N>& tw) {
    using G = BGeo<N>;
    constexpr int H = G::H, YH = G::YH;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const float2* s_gg1 = reinterpret_cast<const float2*>(smem_raw);
    for (int it = threadIdx.x; it < N * YH; it += G::NT) {
        const int ux = it / YH, y = it % YH;
        float2 g[H];
#pragma unroll
        for (int k = 0; k < H; ++k) g[k] = s_gg1[(size_t)(k * N + ux) * YH + y];
        float had[N];   // all loads first
        if (ADD) {
#pragma unroll
            for (int u = 0; u < N; ++u) had[u] = y < ny ? blk[u * slice + ux * pitch + y] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < N; ++u) {
            float z = 0.f;
#pragma unroll
            for (int k = 0; k < H; ++k) {
                z = fmaf(g[k].x, tw.c[k][u], z);
                if (k != 0 && 2 * k != N) z = fmaf(-g[k].y, tw.s[k][u], z);
            }
            if (!ADD) blk[u * slice + ux * pitch + y] = z;
            else if (y < ny) blk[u * slice + ux * pitch + y] = had[u] + z;
        }
    }
}

// One brick (t0, x0, y_start ..), cta its index among the launch's: Gamma_G1 [H][N][YH] at the start of shared memory (after a
// barrier).  EN: the energy reading of the feature (Gamma = 2 rho F, no kink band).  DENSE: one x0 of a brick of the sliding
// form: outputs past kDenseRun are none of its own, and small bins are resolved as above.
template <int N, bool EN, bool DENSE>
__device__ __forceinline__ void adjoint_brick(const float* __restrict__ V, const float* __restrict__ gE, int T, int X, int Y,
                                              int bnd, int t0, int x0, int y_start, const float* __restrict__ wtab,
                                              int taper, const Tw<N>& tw, const Exact2f<N>& ex, const VanishTab& vt,
                                              int* __restrict__ lists, long long cta, long long ncta) {
    using G = BGeo<N>;
    using B = typename G::B;
    constexpr int H = G::H, BY = G::BY, YC = G::YC, YH = G::YH, ROWS = G::ROWS, NT = G::NT, WIN = G::WIN;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* s_in = reinterpret_cast<float*>(smem_raw);
    float2* s_g1 = reinterpret_cast<float2*>(smem_raw + G::IN_BYTES);
    float2* s_win = reinterpret_cast<float2*>(smem_raw);                 // [WIN][NT] after stage 2
    float2* s_gg1 = reinterpret_cast<float2*>(smem_raw);                 // Gamma_G1 [H][N][YH] after step 3
    float2* s_g2 = reinterpret_cast<float2*>(smem_raw + G::A_BYTES);     // G2, then Gamma_G2 [H][N][YH]
    float* s_ge = reinterpret_cast<float*>(smem_raw + G::A_BYTES + G::G_BYTES);  // [3][BY]
    float* s_l1 = s_ge + 3 * BY;                                                 // [BY] window L1 norms
    float* s_col = s_l1 + BY;                                                    // [YH] column sums
    uint16_t* s_small = reinterpret_cast<uint16_t*>(smem_raw + G::SMALL_OFF);    // [YC][NT]
    int* s_src = reinterpret_cast<int*>(smem_raw + G::IDX_OFF);                   // [2][N] cube rows along t, x

    const int tid = threadIdx.x;
    const size_t NV = (size_t)T * X * Y;
    using D = DGeo<N < 8 ? 8 : N>;   // (DENSE: the windows that slide)
    const float4* s_x2 = reinterpret_cast<const float4*>(smem_raw + D::X2_OFF);       // [ROWS][XY]
    const float(*s_ex)[N] = reinterpret_cast<const float(*)[N]>(smem_raw + D::EX_OFF);   // [4][N], the kernel's

    if (!EN && !DENSE)
        for (int i = tid; i < 2 * N; i += NT)
            s_src[i] = i < N ? ext_index(t0 - N / 2 + i, T, bnd) : ext_index(x0 - N / 2 + i - N, X, bnd);
    B::stage_brick(V, s_in, T, X, Y, bnd, t0, x0, y_start);
    for (int i = tid; i < 3 * BY; i += NT) {
        const int m = i / BY, yl = i % BY, y = y_start + yl;
        s_ge[i] = y < Y && (!DENSE || yl < kDenseRun) ? __ldg(gE + m * NV + ((size_t)t0 * X + x0) * Y + y) : 0.f;
    }
    __syncthreads();
    // window L1 norms A[y0] = sum_u h(u_t) h(u_x) h(u_y) |V|, as column sums then a y box sum
    for (int yy = tid; yy < YH; yy += NT) {
        float a = 0.f;
        for (int r = 0; r < N * N; ++r) a = fmaf(tw.c[0][r / N] * tw.c[0][r % N], fabsf(s_in[r * YH + yy]), a);
        s_col[yy] = a;
    }
    B::stage1(s_in, s_g1, tw);
    __syncthreads();
    for (int yl = tid; yl < BY; yl += NT) {
        float a = 0.f;
#pragma unroll
        for (int u = 0; u < N; ++u) a = fmaf(tw.c[0][u], s_col[yl + u], a);
        s_l1[yl] = a;
    }
    B::stage2(s_g1, s_g2, tw);
    __syncthreads();
    if constexpr (DENSE)
        exact_rows<N>(s_in, reinterpret_cast<float4*>(s_g1), reinterpret_cast<float4*>(smem_raw + D::X2_OFF), s_ex);

    // ---- step 2: forward stage 3, Gamma, inverse along y into the private window -------------
    const int row = tid % ROWS;
    const int ych = tid / ROWS;
    float wt[3][H];
    B::row_weights(wtab, row, wt);
#pragma unroll
    for (int j = 0; j < WIN; ++j) s_win[j * NT + tid] = make_float2(0.f, 0.f);
    const float2* grow = s_g2 + (size_t)row * YH;
    float fr[N], fi[N];   // F[k_y] of the current output, all n bins
    // the whole row vanishes when its k_t or its k_x does
    const bool row_vanishes =
        !EN && (((vanish_mask(vt, 0, t0, N) >> (row / N)) | (vanish_mask(vt, 1, x0, N) >> (row % N))) & 1u);
    for (int yi = 0; yi < YC; ++yi) {
        const int yl = ych * YC + yi;
        if (DENSE && yl >= kDenseRun) break;
        {
            float pr[H], pi[H], qr[H], qi[H];
#pragma unroll
            for (int k = 0; k < H; ++k) pr[k] = pi[k] = qr[k] = qi[k] = 0.f;
#pragma unroll
            for (int u = 0; u < N; ++u) {
                const float2 g = grow[yl + u];
#pragma unroll
                for (int k = 0; k < H; ++k) {
                    pr[k] = fmaf(g.x, tw.c[k][u], pr[k]);
                    pi[k] = fmaf(g.y, tw.c[k][u], pi[k]);
                    if (k != 0 && 2 * k != N) {
                        qr[k] = fmaf(g.x, tw.s[k][u], qr[k]);
                        qi[k] = fmaf(g.y, tw.s[k][u], qi[k]);
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < H; ++k) {
                if (k == 0 || 2 * k == N) {
                    fr[k] = pr[k];
                    fi[k] = pi[k];
                } else {
                    fr[k] = pr[k] + qi[k];       // F[k]   = P - iQ
                    fi[k] = pi[k] - qr[k];
                    fr[N - k] = pr[k] - qi[k];   // F[n-k] = P + iQ
                    fi[N - k] = pi[k] + qr[k];
                }
            }
        }
        const float g0 = s_ge[yl], g1 = s_ge[BY + yl], g2 = s_ge[2 * BY + yl];
        const float thr = kSmallBin * s_l1[yl];
        const float thr2 = fmaxf(thr * thr, 1e-30f);   // also keeps subnormal |F|^2 away from rsqrt
        unsigned small = 0u;                            // bins at or below thr: Gamma left to the FP64 recompute
        // A_k = Gamma[k] + Gamma[n-k], B_k = i (Gamma[k] - Gamma[n-k]); self-paired bins: A_k = Gamma[k]
        float ar[H], ai[H], br[H], bi[H];
#pragma unroll
        for (int k = 0; k < H; ++k) {
            const float rho = fmaf(g0, wt[0][k], fmaf(g1, wt[1][k], g2 * wt[2][k]));
            if (k == 0 || 2 * k == N) {
                const float m2 = fmaf(fr[k], fr[k], fi[k] * fi[k]);
                const float sc = f32::bin_adjoint_scale<EN>(rho, m2, thr2);
                if (!EN && m2 <= thr2 && rho != 0.f) small |= 1u << k;
                ar[k] = sc * fr[k];
                ai[k] = sc * fi[k];
                br[k] = bi[k] = 0.f;
            } else {
                const float far = fr[k], fai = fi[k];            // F[k]
                const float hr = fr[N - k], hi = fi[N - k];      // F[n-k]
                const float m2a = fmaf(far, far, fai * fai), m2b = fmaf(hr, hr, hi * hi);
                const float sa = f32::bin_adjoint_scale<EN>(rho, m2a, thr2);
                const float sb = f32::bin_adjoint_scale<EN>(rho, m2b, thr2);
                if (!EN && rho != 0.f) {
                    if (m2a <= thr2) small |= 1u << k;
                    if (m2b <= thr2) small |= 1u << (N - k);
                }
                const float gar = sa * far, gai = sa * fai, gbr = sb * hr, gbi = sb * hi;
                ar[k] = gar + gbr;
                ai[k] = gai + gbi;
                br[k] = gbi - gai;        // i * (Gamma_a - Gamma_b)
                bi[k] = gar - gbr;
            }
        }
        if (!EN) {
            // bins that vanish for every input keep Gamma = 0; so does an all-zero cube (A_p = 0)
            if (small != 0u && (row_vanishes || !(s_l1[yl] > 0.f))) small = 0u;
            if (small != 0u) small &= ~vanish_mask(vt, 2, y_start + yl, N);
            if (!DENSE) s_small[yi * NT + tid] = (uint16_t)small;
        }
        if constexpr (DENSE) {
            const float4* xrow = s_x2 + row * D::XY + yl;
#pragma unroll
            for (int q = 0; q < N; ++q) {
                const int k = q <= N / 2 ? q : N - q;
                if ((small >> q) & 1u) {
                    const float2 d = exact_direction<N>(xrow, q, s_l1[yl], s_ex);
                    const float rho = fmaf(g0, wt[0][k], fmaf(g1, wt[1][k], g2 * wt[2][k]));
                    ar[k] = fmaf(rho, d.x, ar[k]);
                    ai[k] = fmaf(rho, d.y, ai[k]);
                    if (k != 0 && 2 * k != N) {
                        const float sg = q < N / 2 ? rho : -rho;
                        br[k] = fmaf(-sg, d.y, br[k]);
                        bi[k] = fmaf(sg, d.x, bi[k]);
                    }
                }
            }
        }
#pragma unroll
        for (int u = 0; u < N; ++u) {
            float zr = 0.f, zi = 0.f;
#pragma unroll
            for (int k = 0; k < H; ++k) {
                zr = fmaf(ar[k], tw.c[k][u], zr);
                zi = fmaf(ai[k], tw.c[k][u], zi);
                if (k != 0 && 2 * k != N) {
                    zr = fmaf(br[k], tw.s[k][u], zr);
                    zi = fmaf(bi[k], tw.s[k][u], zi);
                }
            }
            float2* w = s_win + (yi + u) * NT + tid;
            float2 acc = *w;
            acc.x += zr;
            acc.y += zi;
            *w = acc;
        }
    }
    if constexpr (!EN && !DENSE) {
        // the small bins go to the listed-bin pass when a list is given and they fit in it
        unsigned* s_wbits = reinterpret_cast<unsigned*>(smem_raw + G::WB_OFF);
        const bool listed = lists && list_small_bins<NT, YC>(s_small, s_wbits,
                                                             lists + list_cta_offset(ncta) + cta * kListStride,
                                                             lists + 4, lists, cta);
        if (!listed)
            resolve_small_bins<N, NT, YC, BY, H, ROWS>(V, X, Y, bnd, y_start, taper, s_small, s_src, s_win, s_ge,
                                                       s_l1, wtab, tw, ex, s_wbits);
    }
    __syncthreads();

    // ---- step 3: sum the y-chunk windows into Gamma_G2[row][y] ---------------------------------
    for (int it = tid; it < ROWS * YH; it += NT) {
        const int r = it % ROWS, y = it / ROWS;   // rows fastest: window reads are consecutive
        float sr = 0.f, si = 0.f;
#pragma unroll
        for (int c = 0; c < BY / YC; ++c) {
            const int j = y - c * YC;
            if (j >= 0 && j < WIN) {
                const float2 v = s_win[j * NT + c * ROWS + r];
                sr += v.x;
                si += v.y;
            }
        }
        s_g2[(size_t)r * YH + y] = make_float2(sr, si);
    }
    __syncthreads();

    // ---- step 4: adjoint of stage 2 (x): Gamma_G1[k_t][u][y] ----------------------------------
    for (int it = tid; it < H * YH; it += NT) {
        const int kt = it / YH, y = it % YH;
        float ar[H], ai[H], br[H], bi[H];
#pragma unroll
        for (int k = 0; k < H; ++k) {
            const float2 a = s_g2[(size_t)(kt * N + k) * YH + y];
            if (k == 0 || 2 * k == N) {
                ar[k] = a.x; ai[k] = a.y; br[k] = bi[k] = 0.f;
            } else {
                const float2 b = s_g2[(size_t)(kt * N + (N - k)) * YH + y];
                ar[k] = a.x + b.x;
                ai[k] = a.y + b.y;
                br[k] = b.y - a.y;
                bi[k] = a.x - b.x;
            }
        }
#pragma unroll
        for (int u = 0; u < N; ++u) {
            float zr = 0.f, zi = 0.f;
#pragma unroll
            for (int k = 0; k < H; ++k) {
                zr = fmaf(ar[k], tw.c[k][u], zr);
                zi = fmaf(ai[k], tw.c[k][u], zi);
                if (k != 0 && 2 * k != N) {
                    zr = fmaf(br[k], tw.s[k][u], zr);
                    zi = fmaf(bi[k], tw.s[k][u], zi);
                }
            }
            s_gg1[(size_t)(kt * N + u) * YH + y] = make_float2(zr, zi);
        }
    }
    __syncthreads();
}

// A CTA per brick (one x0).  The rect cube at n = 8, 16 takes the sliding form (k_spectra_bwd_f32_slide.cu).
template <int N, bool EN>
__global__ void __launch_bounds__(BGeo<N>::NT, BCfg<N>::MINB)
k5_spectra_adjoint_f32(const float* __restrict__ V, const float* __restrict__ gE, float* __restrict__ blocks,
                       int T, int X, int Y, int bnd, int t_begin, int t_step, const float* __restrict__ wtab,
                       int taper, const __grid_constant__ Tw<N> tw, const __grid_constant__ Exact2f<N> ex,
                       const __grid_constant__ VanishTab vt, int* __restrict__ lists) {
    const long long cta = ((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    using G = BGeo<N>;
    // t_step s > 1: the lattice planes of stride-s windows
    adjoint_brick<N, EN, false>(V, gE, T, X, Y, bnd, t_begin + blockIdx.z * t_step, blockIdx.y, blockIdx.x * G::BY, wtab,
                                taper, tw, ex, vt, lists, cta, (long long)gridDim.x * gridDim.y * gridDim.z);
    // ---- step 5: adjoint of stage 1 (t), real part -> scratch block [u_t][u_x][y] -------------
    write_block<N, false>(blocks + cta * G::BLOCK_FLOATS, G::SLICE, G::YH, G::YH, tw);
}

// The bricks the sliding form leaves (dense[brick] set: more small bins than it lists): cluster c looks through the marks of
// bricks c, c + C, .. 32 at a time.  Constant volumes, n = 16: 48^3 42 ms (a direct sum per bin, a CTA per brick: 3.87 s),
// 6 x 8 x 10 1.1 ms (409 ms); n = 8: 3.0 ms (70 ms) and 0.15 ms (5.8 ms).  Bound: the latency of float-float chains.
template <int N>
__global__ void __cluster_dims__(DGeo<N>::CLUSTER, 1, 1) __launch_bounds__(BGeo<N>::NT, DGeo<N>::CTAS)
k5_dense_f32(const float* __restrict__ V, const float* __restrict__ gE, float* __restrict__ blocks, int T, int X, int Y,
             int bnd, int t_begin, int t_step, int t_count, const float* __restrict__ wtab,
             const __grid_constant__ Tw<N> tw, const __grid_constant__ Exact2f<N> ex,
             const __grid_constant__ VanishTab vt, const SpectraAdjointGeometry dg, const int* __restrict__ dense) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int kDenseCluster = DGeo<N>::CLUSTER;
    const auto cluster = cooperative_groups::this_cluster();
    float* s_ex = reinterpret_cast<float*>(smem_raw + DGeo<N>::EX_OFF);
    for (int i = threadIdx.x; i < 4 * N; i += BGeo<N>::NT) {
        const int a = i / N, m = i % N;
        s_ex[i] = a == 0 ? ex.ch[m] : a == 1 ? ex.cl[m] : a == 2 ? ex.sh[m] : ex.sl[m];
    }
    const int rank = blockIdx.x % kDenseCluster, lane = threadIdx.x & 31;
    const long long c = blockIdx.x / kDenseCluster, C = gridDim.x / kDenseCluster;
    const int nseg = (Y + dg.BY - 1) / dg.BY, nxs = (X + dg.BX - 1) / dg.BX;
    const long long total = (long long)nseg * nxs * t_count;
    for (long long b0 = c; b0 < total; b0 += 32 * C) {
        const long long mine = b0 + lane * C;
        unsigned todo = __ballot_sync(0xffffffffu, mine < total && dense[mine] != 0);   // the same in the whole cluster
        for (; todo; todo &= todo - 1) {
            const long long b = b0 + (__ffs(todo) - 1) * C;
            const int sg = (int)(b % nseg), xs = (int)(b / nseg % nxs);
            const int t0 = t_begin + (int)(b / ((long long)nseg * nxs)) * t_step;
            float* blk = blocks + b * dg.block_floats;
            for (int i = rank * BGeo<N>::NT + threadIdx.x; i < dg.block_floats; i += kDenseCluster * BGeo<N>::NT) blk[i] = 0.f;
            const int xl = xs * dg.BX, nx = min(X - xl, dg.BX);
            cluster.sync();   // the block is zeroed
            for (int x = rank; x - rank < nx; x += kDenseCluster) {
                if (x < nx)
                    adjoint_brick<N, false, true>(V, gE, T, X, Y, bnd, t0, xl + x, sg * dg.BY, wtab, 0, tw, ex, vt, nullptr,
                                                  0, 1);
                for (int r = 0; r < kDenseCluster; ++r) {
                    if (r == rank && x < nx) write_block<N, true>(blk + (size_t)x * dg.YH, dg.slice, dg.YH, dg.YH, tw);
                    cluster.sync();
                }
            }
        }
    }
}

template <int N> constexpr bool kHasSliding = N >= 8;   // the rect cube takes k_spectra_bwd_f32_slide.cu

template <int N>
cudaError_t prepare_n() {
    constexpr int smem = (int)BGeo<N>::SMEM;
    cudaError_t e = cudaFuncSetAttribute(k5_spectra_adjoint_f32<N, false>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k5_spectra_adjoint_f32<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if constexpr (kHasSliding<N>) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k5_dense_f32<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DGeo<N>::SMEM);
    }
    return e;
}

template <int N>
cudaError_t launch_n(const TwiddleTable& t, const float* wtab, const float* V, const float* gE, float* blocks, int T,
                     int X, int Y, int bnd, int feat, int t_begin, int t_step, int t_count, int taper, int* lists,
                     cudaStream_t s) {
    using G = BGeo<N>;
    dim3 grid((Y + G::BY - 1) / G::BY, X, t_count);
    note_launches(1);
    if (feat == 1) {
        k5_spectra_adjoint_f32<N, true><<<grid, G::NT, G::SMEM, s>>>(
            V, gE, blocks, T, X, Y, bnd, t_begin, t_step, wtab, taper, f32::make_tw<N>(t), make_exact2f<N>(taper),
            VanishTab{}, nullptr);
        return cudaGetLastError();
    }
    if (lists) {   // the work-list counter starts at zero
        const cudaError_t e = cudaMemsetAsync(lists, 0, sizeof(int), s);
        if (e != cudaSuccess) return e;
    }
    k5_spectra_adjoint_f32<N, false><<<grid, G::NT, G::SMEM, s>>>(
        V, gE, blocks, T, X, Y, bnd, t_begin, t_step, wtab, taper, f32::make_tw<N>(t), make_exact2f<N>(taper),
        make_vanish_tab(N, T, X, Y, bnd, taper), lists);
    if (lists) {
        const long long ncta = (long long)grid.x * grid.y * grid.z;
        k5_listed_exact_f32<N><<<8 * device_sms(), 256, 0, s>>>(V, gE, lists, ncta, T, X, Y, bnd, t_begin, t_step,
                                                                 wtab, taper, make_exact2f<N>(taper));
        k5_listed_apply_f32<N><<<(unsigned)((ncta + 7) / 8), 256, 0, s>>>(blocks, lists, ncta, f32::make_tw<N>(t));
        note_launches(2);
    }
    return cudaGetLastError();
}

template <int N>
cudaError_t launch_dense(const TwiddleTable& t, const float* wtab, const float* V, const float* gE, float* blocks,
                         int T, int X, int Y, int bnd, int t_begin, int t_step, int t_count, const int* dense,
                         cudaStream_t s) {
    using G = BGeo<N>;
    const SpectraAdjointGeometry g = spectra_adjoint_f32_slide_geometry(N);
    const long long total = (long long)((Y + g.BY - 1) / g.BY) * ((X + g.BX - 1) / g.BX) * t_count;
    if (g.BY != kDenseRun || g.YH != DGeo<N>::XY) return cudaErrorInvalidValue;
    const long long clusters = std::max(1, DGeo<N>::CTAS * device_sms() / DGeo<N>::CLUSTER);
    const int grid = (int)std::min(total, clusters) * DGeo<N>::CLUSTER;
    k5_dense_f32<N><<<grid, G::NT, DGeo<N>::SMEM, s>>>(V, gE, blocks, T, X, Y, bnd, t_begin, t_step, t_count, wtab,
                                                 f32::make_tw<N>(t), make_exact2f<N>(0),
                                                 make_vanish_tab(N, T, X, Y, bnd, 0), g, dense);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace

cudaError_t spectra_adjoint_f32_prepare(int n) {
    switch (n) {
        case 2: return prepare_n<2>();
        case 4: return prepare_n<4>();
        case 8: return prepare_n<8>();
        case 16: return prepare_n<16>();
        default: return cudaErrorInvalidValue;
    }
}

SpectraAdjointGeometry spectra_adjoint_f32_geometry(int n) {
    switch (n) {
        case 2: return {BGeo<2>::BY, BGeo<2>::YH, 1, 2, BGeo<2>::BLOCK_FLOATS, BGeo<2>::SLICE};
        case 4: return {BGeo<4>::BY, BGeo<4>::YH, 1, 4, BGeo<4>::BLOCK_FLOATS, BGeo<4>::SLICE};
        case 8: return {BGeo<8>::BY, BGeo<8>::YH, 1, 8, BGeo<8>::BLOCK_FLOATS, BGeo<8>::SLICE};
        case 16: return {BGeo<16>::BY, BGeo<16>::YH, 1, 16, BGeo<16>::BLOCK_FLOATS, BGeo<16>::SLICE};
        default: return {0, 0, 0, 0, 0, 0};
    }
}

cudaError_t spectra_adjoint_f32_dense_launch(int n, const TwiddleTable& tw, const float* wtab, const float* V,
                                             const float* gE, float* blocks, int T, int X, int Y, int bnd,
                                             int t_begin, int t_step, int t_count, const int* dense, cudaStream_t s) {
    if (t_step < 1) return cudaErrorInvalidValue;
    if (n == 8) return launch_dense<8>(tw, wtab, V, gE, blocks, T, X, Y, bnd, t_begin, t_step, t_count, dense, s);
    if (n == 16) return launch_dense<16>(tw, wtab, V, gE, blocks, T, X, Y, bnd, t_begin, t_step, t_count, dense, s);
    return cudaErrorInvalidValue;
}

size_t spectra_adjoint_f32_list_bytes(int n, int X, int Y, int t_count) {
    const int by = n == 16 ? BGeo<16>::BY : BGeo<8>::BY;   // 32 for n <= 8
    const long long ncta = (long long)((Y + by - 1) / by) * X * t_count;
    return (list_cta_offset(ncta) + (size_t)ncta * kListStride) * sizeof(int);
}

cudaError_t spectra_adjoint_f32_launch(int n, const TwiddleTable& tw, const float* wtab, const float* V,
                                       const float* gE, float* blocks, int T, int X, int Y, int bnd, int feat,
                                       int t_begin, int t_step, int t_count, int taper, int* lists, cudaStream_t s) {
    if (t_step < 1 || taper < 0 || taper > 1) return cudaErrorInvalidValue;
    switch (n) {
        case 2:
            return launch_n<2>(tw, wtab, V, gE, blocks, T, X, Y, bnd, feat, t_begin, t_step, t_count, taper, lists, s);
        case 4:
            return launch_n<4>(tw, wtab, V, gE, blocks, T, X, Y, bnd, feat, t_begin, t_step, t_count, taper, lists, s);
        case 8:
            return launch_n<8>(tw, wtab, V, gE, blocks, T, X, Y, bnd, feat, t_begin, t_step, t_count, taper, lists, s);
        case 16:
            return launch_n<16>(tw, wtab, V, gE, blocks, T, X, Y, bnd, feat, t_begin, t_step, t_count, taper, lists,
                                s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace sal

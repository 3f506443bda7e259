// K5-F32, sliding form (rect cube, n = 8, 16): adjoint of the local-spectrum feature step in FP32, as
// k_spectra_bwd_f32.cu defines it (Gamma, small bins), over the tiles and register FFTs of the sliding forward
// (spectra_f32_fft.cuh).  One group of threads takes one brick: one t0, RX positions x0, 16 outputs y0.
//   stages 1 and 2 as in K1; per tile, a thread per (x0, k_x) then follows its row along y in runs of R outputs (4 for
//   n = 8, 8 for n = 16): a run's first window by an FFT, the others by the anchored recursion F_{j+1}[k] = F_j[k] +
//   d_j w^(k j).  |F| does not see the phase, and with Gamma_j the gradient of F_j in the same phase and P_j = sum_{i <= j}
//   Gamma_i the run's part of the row's gradient is
//     e_p (p < n),   e_p - e_{p-n} (p >= n),   e_j = sum_k P_j[k] w^(-k j)  (j < R-1),   e_p = sum_k P_{R-1}[k] w^(-k p) after,
//   one evaluation at a point per output (two additions a bin, the adjoint of the recursion) and one inverse FFT per
//   run; the n - 1 positions a run shares with the next stay in registers, and the gradient replaces G2 in the thread's
//   own row.  The sums P run over R outputs and no more: what is left of a strong output where its windows have ended (the
//   differences e_p - e_{p-n}), and a NaN, reach R - 1 outputs on (runs of all 16: up to 15, and 2 to 4 times the error
//   beside an output of 1e5 times the others' gradient; at n = 16 that took 6.2 instead of 6.9 ms on 128^3);
//   adjoint of stage 2: an inverse FFT per (x0, y), then per halo position the sum of the x0 whose cubes hold it,
//   which replaces the tile's G1; after all tiles the adjoint of stage 1 writes the brick's block.
// Small bins (|F| <= 2^-16 of the window's L1 norm) take Gamma = 0 in the tile loop and go to the brick's list; at the
// end, in the order of their codes, its warps recompute them as direct float-float sums, and their rank-one gradients
// are added to the gradient of G1 (256 terms each; at the block they would be 4096).  A brick with more than
// list_max such bins (constant regions: every bin) is marked and left to k5_dense_f32.
// The instruction cache sets how far the loop over outputs is unrolled: by R, and not at all in tile 0, whose packed rows
// need the most code for an eighth of the work (there every window is an FFT).
// Bound: issue slots, about 500 per thread and output of 16 bins with the FFTs and the small bins (128 MUFU cycles), by 12
// warps an SM at 168 registers.  The adjoint call, 128^3: n = 16 25.0 -> 6.9 ms, n = 8 2.54 -> 0.91
// (before: one x0 per brick, direct DFTs in stages 1 and 2 and both of their adjoints, 31 point evaluations of 32
// multiply-adds per run of 8 outputs, and two passes over the grid for the small bins, 0.1 per voxel here); 24^3, n = 16:
// 353 -> 186 us.  Error against FP64 9.8e-7 -> 9.7e-7 (n = 16), 7.9e-7 -> 7.6e-7 (n = 8), most of it in the directions
// of the weak bins just above the small-bin level.
#include "spectra_f32_exact.cuh"
#include "spectra_f32_fft.cuh"

namespace sal {
namespace {

using f32::Bins;
using f32::Exact2f;
using f32::fast_rsqrt;
using f32::FF;
using f32::ff_add;
using f32::ff_gather;
using f32::ff_mul;
using f32::kSmallBin;
using f32::kZeroBin;
using f32::vanish_mask;
using f32::VanishTab;

constexpr int kRun = 16;     // outputs of a brick along y
constexpr int kList = 1024;  // small bins a brick can list at most
constexpr int kChunk = 64;   // small bins whose Gamma is held at a time

// n = 8: a brick of 16 x0 per CTA of 128 threads, four CTAs an SM.  n = 16: bricks of 12 x0 in groups of 192 threads,
// two in a CTA of 384 (whole multiples of four warps, the granule of register allocation), one CTA an SM; the groups
// meet at barriers of their own.  With no more bricks than SMs a CTA takes one (12 x 16 x 20: 248 -> 205 us a call).
template <int N> struct AGeo;
template <> struct AGeo<8> { static constexpr int RX = 16, R = 4, GROUPS = 1, CTAS = 4; };
template <> struct AGeo<16> { static constexpr int RX = 12, R = 8, GROUPS = 2, CTAS = 1; };
template <int N, int GROUPS_ = AGeo<N>::GROUPS> struct Adj {
    static constexpr int GROUPS = GROUPS_, CTAS = AGeo<N>::CTAS;
    static constexpr int RX = AGeo<N>::RX, GT = RX * N, NT = GT * GROUPS, TILES = N / 2, H = N / 2 + 1;
    static constexpr int XH = RX + N - 1, YH = kRun + N - 1;   // YH odd: rows YH float2 apart meet no bank conflict
    static constexpr int SLICE = (XH * YH + 3) / 4 * 4;        // u_t slices of the block, 16-byte aligned
    static constexpr int BLOCK_FLOATS = N * SLICE;
    static constexpr size_t G1 = (size_t)TILES * XH * YH, G2 = (size_t)RX * N * YH;   // float2
    static constexpr size_t FLOATS = 2 * (G1 + G2) + kList + 4 * RX * kRun + 2 * kChunk + 4 + N + XH + 1 + RX + kRun;
    static constexpr size_t GROUP_B = (FLOATS * 4 + 15) / 16 * 16;
    static constexpr size_t SMEM = GROUPS * GROUP_B;
    static_assert((SMEM + 1024) * CTAS <= 228 * 1024, "geometry");
    static_assert((size_t)XH * YH + XH * kRun <= 2 * G2 && kList <= 2 * G2, "L1 sums and the sorted list fit in G2");
};

// A small bin: x0 within the brick (5 bits), output (4), k_t (4), k_x (4), k_y (4).
__device__ __forceinline__ int small_code(int x0l, int j, int kt, int kx, int ky) {
    return x0l | (j << 5) | (kt << 9) | (kx << 13) | (ky << 17);
}

// The small bins of one thread's output onto the brick's list (past kList they are only counted).  small_a: bit k_y of
// tiles above 0; tile 0: bit q of the pairs' first values, small_b of their second ones.  mx, my: the vanishing bins of
// the output's x0 and y0; mt of t0.
template <int N>
__device__ __noinline__ void note_small(uint32_t mt, uint32_t mx, uint32_t my, int tile, int tid, int j, unsigned small_a,
                                        unsigned small_b, int* s_small, int* s_count) {
    const int kx = tid % N, x0l = tid / N;
    const bool upper = tile == 0 && kx > N / 2, packed = tile == 0 && (kx == 0 || kx == N / 2);
    for (int second = 0; second < 2; ++second)
        for (unsigned m = second ? small_b : small_a; m; m &= m - 1) {
            const int q = __ffs(m) - 1;
            const int kt = tile != 0 ? tile : (upper || (packed && second) ? N / 2 : 0);
            const int kxs = upper ? N - kx : kx, ky = second && !packed ? N - q : q;
            if ((kt | kxs | ky) == 0 || (((mt >> kt) | (mx >> kxs) | (my >> ky)) & 1u)) continue;   // DC, vanishing
            const int at = atomicAdd(s_count, 1);
            if (at < kList) s_small[at] = small_code(x0l, j, kt, kxs, ky);
        }
}

template <int N, bool EN, int GROUPS>
__global__ void __launch_bounds__(Adj<N, GROUPS>::NT, AGeo<N>::CTAS)
k5_slide(const float* __restrict__ V, const float* __restrict__ gE, float* __restrict__ blocks, int T, int X, int Y,
         int bnd, int t_begin, int t_step, const float* __restrict__ wtab, const __grid_constant__ Exact2f<N> ex,
         const __grid_constant__ VanishTab vt, int* __restrict__ dense, int list_max) {
    using G = Adj<N, GROUPS>;
    using B = Bins<N, false>;
    constexpr int RX = G::RX, R = AGeo<N>::R, XH = G::XH, YH = G::YH, GT = G::GT, H = G::H, TILES = G::TILES, NW = B::NW;
    constexpr size_t TILE_W = (size_t)3 * H * N;   // weights of a tile, [map][k][row] (f32_slide_table_fill)
    constexpr bool ALT = N == 8;                   // the directions of weak bins (at n = 16 no further off than direct sums)
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float s_ex[4][N];   // cos, sin (2 pi m / n) as float-float pairs, indexed by the lanes' own phases
    const int grp = threadIdx.x / GT, tid = threadIdx.x % GT, lane = threadIdx.x & 31, warp = tid >> 5;
    float2* s_g1 = reinterpret_cast<float2*>(smem_raw + grp * G::GROUP_B);   // [tile][x][y], then its gradient
    float2* s_g2 = s_g1 + G::G1;                                             // [x0][k_x][y], then its gradient
    int* s_small = reinterpret_cast<int*>(s_g2 + G::G2);                     // [kList] codes
    float* s_ge = reinterpret_cast<float*>(s_small + kList);                 // [3][x0][j]
    float* s_l1 = s_ge + 3 * RX * kRun;                                      // [x0][j] window L1 norms
    float2* s_gam = reinterpret_cast<float2*>(s_l1 + RX * kRun);             // [kChunk]
    int* s_count = reinterpret_cast<int*>(s_gam + kChunk);                   // small bins so far
    int* s_src = s_count + 4;                                                // [n] source planes, [XH] source rows
    uint32_t* s_van = reinterpret_cast<uint32_t*>(s_src + N + XH);           // vanishing bins of t0, of each x0, of each y0
    auto group_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(GT) : "memory"); };
    for (int i = threadIdx.x; i < 4 * N; i += G::NT) {
        const int a = i / N, m = i % N;
        s_ex[a][m] = a == 0 ? ex.ch[m] : a == 1 ? ex.cl[m] : a == 2 ? ex.sh[m] : ex.sl[m];
    }
    __syncthreads();

    const int nseg = (Y + kRun - 1) / kRun, nxs = (X + RX - 1) / RX;
    const int brick = blockIdx.x * GROUPS + grp;   // within the plane: x brick, y segment
    if (brick >= nseg * nxs) return;                  // whole group: only its own barriers follow
    const int yb = (brick % nseg) * kRun, xb = (brick / nseg) * RX, t0 = t_begin + blockIdx.z * t_step;
    const size_t NV = (size_t)T * X * Y, plane = (size_t)X * Y;
    const size_t id = (size_t)blockIdx.z * nseg * nxs + brick;

    // ---- gE of the outputs, stage 1, column sums of |V| ------------------------------------------------
    if (tid == 0) *s_count = 0;
    if (!EN)
        for (int i = tid; i < 1 + RX + kRun; i += GT) {   // (outputs past the volume have no gradient and note nothing)
            const int x = min(X - 1, xb + i - 1), y = min(Y - 1, yb + i - 1 - RX);
            s_van[i] = i == 0 ? vanish_mask(vt, 0, t0, N) : i <= RX ? vanish_mask(vt, 1, x, N) : vanish_mask(vt, 2, y, N);
        }
    for (int i = tid; i < N + XH; i += GT)
        s_src[i] = i < N ? ext_index(t0 - N / 2 + i, T, bnd) : ext_index(xb - N / 2 + i - N, X, bnd);
    for (int i = tid; i < 3 * RX * kRun; i += GT) {
        const int m = i / (RX * kRun), x = xb + (i / kRun) % RX, y = yb + i % kRun;
        s_ge[i] = x < X && y < Y ? __ldg(gE + m * NV + ((size_t)t0 * X + x) * Y + y) : 0.f;
    }
    group_sync();   // s_src
    float* s_col = reinterpret_cast<float*>(s_g2);   // [x][y], before the first tile's G2
    float* s_row = s_col + XH * YH;                  // [x][j]
    const bool t_in = t0 - N / 2 >= 0 && t0 + N / 2 <= T;
    for (int it = tid; it < XH * YH; it += GT) {
        const int x = it / YH, y = it - x * YH;
        const int gx = s_src[N + x], gy = ext_index(yb - N / 2 + y, Y, bnd);
        const bool in = (gx | gy) >= 0;
        const float* p = V + (in ? (size_t)gx * Y + gy : 0);
        float v[N], a = 0.f;
        float2 o[N / 2];
        if (t_in) {
            p += (size_t)(t0 - N / 2) * plane;
#pragma unroll
            for (int u = 0; u < N; ++u) v[u] = in ? __ldg(p + u * plane) : 0.f;
        } else {
#pragma unroll
            for (int u = 0; u < N; ++u) {
                const int gt = s_src[u];
                v[u] = in && gt >= 0 ? __ldg(p + gt * plane) : 0.f;
            }
        }
        if (!EN) {
#pragma unroll
            for (int u = 0; u < N; ++u) a += fabsf(v[u]);
            s_col[it] = a;
        }
        f32::rfft<N, ALT>(v, o);
#pragma unroll
        for (int k = 0; k < TILES; ++k) s_g1[(size_t)k * XH * YH + it] = o[k];
    }
    group_sync();
    if (!EN) {
        for (int i = tid; i < XH * kRun; i += GT) {
            float a = 0.f;
#pragma unroll
            for (int u = 0; u < N; ++u) a += s_col[(i / kRun) * YH + i % kRun + u];
            s_row[i] = a;
        }
        group_sync();
        for (int i = tid; i < RX * kRun; i += GT) {
            float a = 0.f;
#pragma unroll
            for (int u = 0; u < N; ++u) a += s_row[(i / kRun + u) * kRun + i % kRun];
            s_l1[i] = a;
        }
        group_sync();
    }

    // ---- tiles -----------------------------------------------------------------------------------------
    const int kx = tid % N, x0l = tid / N;
    float2* row = s_g2 + (size_t)tid * YH;
    const float* l1 = s_l1 + x0l * kRun;
    const float* ge = s_ge + x0l * kRun;
    for (int tile = 0; tile < TILES; ++tile) {
        // stage 2 (x)
        for (int it = tid; it < RX * YH; it += GT) {
            const int x = it / YH, y = it - x * YH;
            const float2* src = s_g1 + ((size_t)tile * XH + x) * YH + y;
            float2 v[N];
#pragma unroll
            for (int u = 0; u < N; ++u) v[u] = src[u * YH];
            f32::fft<N, ALT>(v);
            float2* dst = s_g2 + (size_t)x * N * YH + y;
            if (tile != 0) {
#pragma unroll
                for (int k = 0; k < N; ++k) dst[k * YH] = v[f32::fft_pos<N>(k)];
            } else {
#pragma unroll
                for (int k = 0; k < N; ++k) dst[k * YH] = f32::tile0_row<N>(v, k);
            }
        }
        group_sync();
        // stage 3 (y), Gamma, adjoint of stage 3
        {
            float wt[3][NW];
#pragma unroll
            for (int m = 0; m < 3; ++m)
#pragma unroll
                for (int w = 0; w < NW; ++w) wt[m][w] = __ldg(wtab + tile * TILE_W + (m * H + w) * N + kx);
            B f, P;
            float2 c[N - 1];   // what the runs so far give to positions h .. h + n - 2
#pragma unroll
            for (int i = 0; i < N - 1; ++i) c[i] = make_float2(0.f, 0.f);
            // rho per |k_y| of output j: sum_m gE_m w_m
            auto weights = [&](int j, float (&rho)[NW]) {
                const float g0 = ge[j], g1 = ge[RX * kRun + j], g2 = ge[2 * RX * kRun + j];
#pragma unroll
                for (int w = 0; w + 1 < NW; w += 2) {
                    const float2 r2 = __ffma2_rn(make_float2(g0, g0), make_float2(wt[0][w], wt[0][w + 1]),
                                                 __ffma2_rn(make_float2(g1, g1), make_float2(wt[1][w], wt[1][w + 1]),
                                                            __fmul2_rn(make_float2(g2, g2),
                                                                       make_float2(wt[2][w], wt[2][w + 1]))));
                    rho[w] = r2.x;
                    rho[w + 1] = r2.y;
                }
                rho[NW - 1] = fmaf(g0, wt[0][NW - 1], fmaf(g1, wt[1][NW - 1], g2 * wt[2][NW - 1]));
            };
            // the small-bin level of output j, squared; it also keeps subnormal |F|^2 away from rsqrt.  A window of zeros has no
            // direction: what the recursion leaves there is the rounding of samples that have left it
            auto level = [&](int j) {
                const float a = kSmallBin * l1[j];
                return l1[j] == 0.f ? 3.4e38f : fmaxf(a * a, 1e-30f);
            };
            // small bins at output j (bit k_y; tile 0: bit q of the pairs' first and second values) onto the list
            auto note = [&](int j, unsigned small_a, unsigned small_b) {
                const uint32_t my = s_van[1 + RX + j];
                if (tile != 0) small_a = ((s_van[0] >> tile) | (s_van[1 + x0l] >> kx)) & 1u ? 0u : small_a & ~my;
                if ((small_a | small_b) && l1[j] > 0.f &&
                    (ge[j] != 0.f || ge[RX * kRun + j] != 0.f || ge[2 * RX * kRun + j] != 0.f))
                    note_small<N>(s_van[0], s_van[1 + x0l], my, tile, tid, j, small_a, small_b, s_small, s_count);
            };
            // tile 0: packed rows hold two signals (k_t = 0 and n/2) in each pair.  Every window anew, in its own phase
            // (the sums P turn with it)
            const float* wb = wtab + TILES * TILE_W + kx;
            const bool packed = kx == 0 || kx == N / 2;
            const float pk = packed ? 1.f : 0.f, qk = 1.f - 2.f * pk;
#pragma unroll 1
            for (int h = 0; h < kRun; h += R) {
                f.template first<N, ALT>(row + h);   // phases are those of the run's first window
#pragma unroll
                for (int q = 0; q < N / 2; ++q) P.r[q] = P.i[q] = make_float2(0.f, 0.f);
                if (tile != 0) {
#pragma unroll
                    for (int b = 0; b < R; ++b) {
                        const int j = h + b;
                        float2 d = make_float2(0.f, 0.f);
                        if (b + 1 < R) {   // before row[j] becomes the gradient's
                            const float2 u = row[j], v = row[j + N];
                            d = make_float2(v.x - u.x, v.y - u.y);
                        }
                        float rho[NW];
                        weights(j, rho);
                        const float thr2 = level(j);
                        float2 sc[N / 2];
                        float lo = 3.4e38f;
#pragma unroll
                        for (int q = 0; q < N / 2; ++q) {
                            const float2 r = q == 0 ? make_float2(rho[0], rho[N / 2]) : make_float2(rho[q], rho[q]);
                            if (EN) {
                                sc[q] = make_float2(2.f * r.x, 2.f * r.y);
                            } else {
                                const float2 m2 = __ffma2_rn(f.i[q], f.i[q], __fmul2_rn(f.r[q], f.r[q]));
                                sc[q] = __fmul2_rn(r, make_float2(fast_rsqrt(m2.x), fast_rsqrt(m2.y)));
                                lo = fminf(lo, fminf(m2.x, m2.y));
                            }
                        }
                        if (!EN && !(lo > thr2)) {   // rare: a bin at or below the level takes Gamma = 0 here
                            unsigned small = 0u;
#pragma unroll
                            for (int q = 0; q < N; ++q) {
                                const float2 F = f.get(q);
                                if (!(fmaf(F.y, F.y, F.x * F.x) > thr2)) {
                                    if (B::second(q)) sc[B::slot(q)].y = 0.f;
                                    else sc[B::slot(q)].x = 0.f;
                                    small |= 1u << q;
                                }
                            }
                            note(j, small, 0u);
                        }
#pragma unroll
                        for (int q = 0; q < N / 2; ++q) {
                            P.r[q] = __ffma2_rn(sc[q], f.r[q], P.r[q]);
                            P.i[q] = __ffma2_rn(sc[q], f.i[q], P.i[q]);
                        }
                        if (b + 1 < R) {
                            const float2 e = P.at(b);
                            row[j] = make_float2(e.x + c[b].x, e.y + c[b].y);
                            c[b] = e;
                            f.slide(d, b);
                        }
                    }
                } else {
#pragma unroll 1
                    for (int b = 0; b < R; ++b) {
                        const int j = h + b;
                        if (b > 0) f.template first<N, ALT>(row + j);
                        float rho[NW];
                        weights(j, rho);
                        const float g0 = ge[j], g1 = ge[RX * kRun + j], g2 = ge[2 * RX * kRun + j];
                        const float thr2 = level(j), thr2p = packed ? 4.f * thr2 : thr2;   // a packed pair holds 2 F
                        unsigned small_a = 0u, small_b = 0u;
                        auto scale = [&](float m2, float r, float lim, unsigned& small, int bit) -> float {
                            if (EN) return 2.f * r;
                            if (m2 > lim) return r * fast_rsqrt(m2);
                            small |= 1u << bit;
                            return 0.f;
                        };
                        auto rho_b = [&](int w) -> float {   // the second value of the pair
                            return fmaf(g0, __ldg(wb + w * N),
                                        fmaf(g1, __ldg(wb + (H + w) * N), g2 * __ldg(wb + (2 * H + w) * N)));
                        };
#pragma unroll
                        for (int k = 0; k <= N / 2; k += N / 2) {   // the self-paired bins 0 and n/2
                            const float re = k ? f.r[0].y : f.r[0].x, im = k ? f.i[0].y : f.i[0].x;
                            const float sa = scale(fmaf(re, re, (1.f - pk) * im * im), rho[k], thr2, small_a, k);
                            const float ga = sa * re;
                            float gb = sa * im;
                            if (packed) gb = scale(im * im, rho_b(k), thr2, small_b, k) * im;
                            if (k) {
                                P.r[0].y += ga;
                                P.i[0].y += gb;
                            } else {
                                P.r[0].x += ga;
                                P.i[0].x += gb;
                            }
                        }
#pragma unroll
                        for (int q = 1; q < N / 2; ++q) {
                            const float2 Rr = f.r[q], Ii = f.i[q];
                            const float r1 = fmaf(pk, Rr.y, Rr.x), i1 = fmaf(-pk, Ii.y, Ii.x);
                            const float r2 = fmaf(pk, Rr.x, qk * Rr.y), i2 = fmaf(pk, Ii.x, Ii.y);
                            const float sa = scale(fmaf(r1, r1, i1 * i1), rho[q], thr2p, small_a, q);
                            const float sb = scale(fmaf(r2, r2, i2 * i2), rho_b(q), thr2p, small_b, q);
                            const float ur = sa * r1, ui = sa * i1, vr = sb * r2, vi = sb * i2;
                            P.r[q].x += fmaf(pk, vr, ur);
                            P.i[q].x += fmaf(pk, vi, ui);
                            P.r[q].y += fmaf(pk, ur, qk * vr);
                            P.i[q].y += fmaf(-pk, ui, vi);
                        }
                        if (!EN && (small_a | small_b)) note(j, small_a, small_b);
                        if (b + 1 < R) {
                            const float2 e = P.sum();
                            row[j] = make_float2(e.x + c[0].x, e.y + c[0].y);
#pragma unroll
                            for (int i = 0; i + 1 < N - 1; ++i) c[i] = c[i + 1];   // (a loop that is not unrolled: by turns)
                            c[N - 2] = e;
                            P.turn();
                        }
                    }
                    float2 o[N - 1];
#pragma unroll
                    for (int i = 0; i < N - 1; ++i) o[(i + R - 1) % (N - 1)] = c[i];
#pragma unroll
                    for (int i = 0; i < N - 1; ++i) c[i] = o[i];
                }
                // c: e_0 .. e_{R-2} of this run, then what is left of the runs before.  z: sum_k P_{R-1}[k] w^(-k i) at position
                // h + i, of period n; in tile 0 P is in the phase of the last window, w^(-(R-1) k) ahead
                float2 z[N];
#pragma unroll
                for (int q = 0; q < N; ++q) z[q] = P.get(q);
                f32::ifft<N>(z);
                auto at = [&](int i) -> float2 {
                    return tile == 0 ? z[f32::fft_pos<N>((i + N - (R - 1)) % N)] : z[f32::fft_pos<N>(i % N)];
                };
                {
                    const float2 e = at(R - 1);
                    row[h + R - 1] = make_float2(e.x + c[R - 1].x, e.y + c[R - 1].y);
                }
                float2 o[N - 1];
#pragma unroll
                for (int i = R; i < R + N - 1; ++i) {
                    const float2 e = at(i % N);
                    o[i - R] = i < N - 1    ? make_float2(e.x + c[i].x, e.y + c[i].y)
                               : i == N - 1 ? e
                                            : make_float2(e.x - c[i % N].x, e.y - c[i % N].y);
                }
#pragma unroll
                for (int i = 0; i < N - 1; ++i) c[i] = o[i];
            }
#pragma unroll
            for (int i = 0; i < N - 1; ++i) row[kRun + i] = c[i];
        }
        group_sync();
        // adjoint of stage 2: inverse FFT over k_x of each (x0, y), in place as [x0][u][y]
        for (int it = tid; it < RX * YH; it += GT) {
            const int x = it / YH, y = it - x * YH;
            float2* dst = s_g2 + (size_t)x * N * YH + y;
            float2 v[N];
#pragma unroll
            for (int k = 0; k < N; ++k) v[k] = dst[k * YH];
            if (tile == 0) f32::tile0_adjoint<N>(v);
            f32::ifft<N>(v);
#pragma unroll
            for (int u = 0; u < N; ++u) dst[u * YH] = v[f32::fft_pos<N>(u)];
        }
        group_sync();
        // halo position (x, y): the sum over the x0 whose cubes hold it replaces the tile's G1
        for (int it = tid; it < XH * YH; it += GT) {
            const int x = it / YH, y = it - x * YH;
            float sr = 0.f, si = 0.f;
#pragma unroll
            for (int a = 0; a < RX; ++a) {
                const int u = x - a;
                if (u >= 0 && u < N) {
                    const float2 g = s_g2[(size_t)(a * N + u) * YH + y];
                    sr += g.x;
                    si += g.y;
                }
            }
            s_g1[(size_t)tile * XH * YH + it] = make_float2(sr, si);
        }
        if (tile + 1 < TILES) group_sync();   // G2 is rewritten
    }

    // ---- small bins ------------------------------------------------------------------------------------
    if (!EN) {
        group_sync();
        const int total = *s_count;
        if (tid == 0) dense[id] = total > list_max;
        if (total > list_max) return;   // whole group: this brick's block comes from k5_dense_f32
        int* s_list = reinterpret_cast<int*>(s_g2);   // the codes in increasing order (G2 is free)
        for (int i = tid; i < total; i += GT) {
            const int c = s_small[i];
            int rank = 0;
            for (int k = 0; k < total; ++k) rank += s_small[k] < c;
            s_list[rank] = c;
        }
        group_sync();
        // a lane's terms: its u_y = lane % n, the NU u_x = lane / n + i STEP, every u_t
        constexpr int N3 = N * N * N, STEP = 32 / N, NU = N / STEP;
        const int uy = lane % N, ux0 = lane / N;
        for (int c0 = 0; c0 < total; c0 += kChunk) {
            const int c1 = min(total, c0 + kChunk);
            for (int e = c0 + warp; e < c1; e += GT / 32) {
                // F = sum_u V[p + u - n/2] w^(k.u) by one warp, float-float: over u_t for each (u_x, u_y), the
                // low parts gathered without renormalising (16 terms), then the phases of (u_x, u_y)
                const int code = s_list[e];
                const int xl = code & 31, j = (code >> 5) & 15, kt = (code >> 9) & 15, kxs = (code >> 13) & 15,
                          ky = (code >> 17) & 15;
                const int gy = ext_index(yb + j - N / 2 + uy, Y, bnd);
                FF re[NU], im[NU];
                long long col[NU];   // gx Y + gy, or -1
#pragma unroll
                for (int a = 0; a < NU; ++a) {
                    const int gx = s_src[N + xl + ux0 + a * STEP];
                    col[a] = (gx | gy) >= 0 ? (long long)gx * Y + gy : -1;
                    re[a] = im[a] = FF{0.f, 0.f};
                }
#pragma unroll (N == 8 ? 8 : 2)
                for (int ut = 0; ut < N; ++ut) {   // 16 loads in flight
                    const int gt = s_src[ut], ph = (kt * ut) % N;
                    const float* p = V + (size_t)(gt < 0 ? 0 : gt) * plane;
                    const float ch = s_ex[0][ph], cl = s_ex[1][ph], sh = -s_ex[2][ph], sl = -s_ex[3][ph];
                    float v[NU];
#pragma unroll
                    for (int a = 0; a < NU; ++a) v[a] = gt >= 0 && col[a] >= 0 ? __ldg(p + col[a]) : 0.f;
#pragma unroll
                    for (int a = 0; a < NU; ++a) {
                        ff_gather(re[a], v[a], ch, cl);
                        ff_gather(im[a], v[a], sh, sl);
                    }
                }
                FF fre = {0.f, 0.f}, fim = {0.f, 0.f};
#pragma unroll
                for (int a = 0; a < NU; ++a) {
                    const FF x = f32::ff_fast_two_sum(re[a].hi, re[a].lo), y = f32::ff_fast_two_sum(im[a].hi, im[a].lo);
                    const int ph = (kxs * (ux0 + a * STEP) + ky * uy) % N;
                    const FF c = {s_ex[0][ph], s_ex[1][ph]}, sn = {s_ex[2][ph], s_ex[3][ph]}, ns = {-sn.hi, -sn.lo};
                    fre = ff_add(fre, ff_add(ff_mul(x, c), ff_mul(y, sn)));
                    fim = ff_add(fim, ff_add(ff_mul(y, c), ff_mul(x, ns)));
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    fre = ff_add(fre, FF{__shfl_xor_sync(0xffffffffu, fre.hi, o), __shfl_xor_sync(0xffffffffu, fre.lo, o)});
                    fim = ff_add(fim, FF{__shfl_xor_sync(0xffffffffu, fim.hi, o), __shfl_xor_sync(0xffffffffu, fim.lo, o)});
                }
                if (lane == 0) {
                    const int gi = xl * kRun + j;
                    float2 gam = make_float2(0.f, 0.f);
                    const float mx = fmaxf(fabsf(fre.hi), fabsf(fim.hi));
                    if (mx > kZeroBin * s_l1[gi]) {
                        // the bins of the half spectrum this one stands for: itself and its mirror, unless they coincide
                        const bool self = (2 * kt) % N == 0 && (2 * kxs) % N == 0 && (2 * ky) % N == 0;
                        float w0, w1, w2;
                        f32::bin_weights<false>(kt, kxs <= N / 2 ? kxs : N - kxs, ky <= N / 2 ? ky : N - ky,
                                                (self ? 1.f : 2.f) / (float)N3, w0, w1, w2);
                        const float r = fmaf(s_ge[gi], w0, fmaf(s_ge[RX * kRun + gi], w1, s_ge[2 * RX * kRun + gi] * w2));
                        const float fr = fre.hi / mx, fi = fim.hi / mx;   // scaled first: no underflow
                        const float sc = r / sqrtf(fmaf(fr, fr, fi * fi));
                        gam = make_float2(sc * fr, sc * fi);
                    }
                    s_gam[e - c0] = gam;
                }
            }
            group_sync();
            // Gamma e^(+2 pi i (k_x u_x + k_y u_y) / n) added to the gradient of G1 of its k_t (tile 0: the real part
            // of bin k_t = 0 or n/2 in the real or the imaginary part)
            for (int e = c0; e < c1; ++e) {
                const int code = s_list[e];
                const int xl = code & 31, j = (code >> 5) & 15, kt = (code >> 9) & 15, kxs = (code >> 13) & 15,
                          ky = (code >> 17) & 15;
                const float2 gam = s_gam[e - c0];
                for (int i = tid; i < N * N; i += GT) {
                    const int ux = i / N, vy = i % N, ph = (kxs * ux + ky * vy) % N;
                    const float c = s_ex[0][ph], sn = s_ex[2][ph];
                    float2* g = s_g1 + ((size_t)(kt == N / 2 ? 0 : kt) * XH + xl + ux) * YH + j + vy;
                    const float gr = gam.x * c - gam.y * sn;
                    if (kt == 0) g->x += gr;
                    else if (kt == N / 2) g->y += gr;
                    else {
                        g->x += gr;
                        g->y += gam.x * sn + gam.y * c;
                    }
                }
                group_sync();
            }
        }
    }
    group_sync();

    // ---- adjoint of stage 1 (t), real part -> the block [u_t][x][y] ------------------------------------------
    float* blk = blocks + id * G::BLOCK_FLOATS;
    for (int it = tid; it < XH * YH; it += GT) {
        float2 g[N / 2];
        float v[N];
#pragma unroll
        for (int k = 0; k < TILES; ++k) g[k] = s_g1[(size_t)k * XH * YH + it];
        f32::rfft_adjoint<N>(g, v);
#pragma unroll
        for (int u = 0; u < N; ++u) blk[(size_t)u * G::SLICE + it] = v[u];
    }
}

template <int N, int GROUPS> cudaError_t prepare_g() {
    cudaError_t e = cudaFuncSetAttribute(k5_slide<N, false, GROUPS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)Adj<N, GROUPS>::SMEM);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k5_slide<N, true, GROUPS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)Adj<N, GROUPS>::SMEM);
}

template <int N, int GROUPS>
void launch_g(const float* wtab, const float* V, const float* gE, float* blocks, int T, int X, int Y, int bnd, int feat,
              int t_begin, int t_step, int t_count, int bricks, int* dense, int list_max, cudaStream_t s) {
    using G = Adj<N, GROUPS>;
    const dim3 grid((bricks + GROUPS - 1) / GROUPS, 1, t_count);
    const Exact2f<N> ex = f32::make_exact2f<N>(0);
    if (feat == 1)
        k5_slide<N, true, GROUPS><<<grid, G::NT, G::SMEM, s>>>(V, gE, blocks, T, X, Y, bnd, t_begin, t_step, wtab, ex,
                                                               VanishTab{}, dense, list_max);
    else
        k5_slide<N, false, GROUPS><<<grid, G::NT, G::SMEM, s>>>(V, gE, blocks, T, X, Y, bnd, t_begin, t_step, wtab, ex,
                                                                f32::make_vanish_tab(N, T, X, Y, bnd, 0), dense,
                                                                list_max);
}

template <int N>
cudaError_t launch_n(const float* wtab, const float* V, const float* gE, float* blocks, int T, int X, int Y, int bnd,
                     int feat, int t_begin, int t_step, int t_count, int* dense, cudaStream_t s) {
    const int bricks = ((Y + kRun - 1) / kRun) * ((X + AGeo<N>::RX - 1) / AGeo<N>::RX);
    // n = 8: a listed bin takes 0.4 us of its brick's time, k5_dense_f32 about 100 us for all of them, but many bricks side by
    // side 6.6 us each against 0.4 for a full list.  So the list ends early where the bricks leave SMs idle (one sample set
    // in 12 x 16 x 20: 590 -> 140 us; 5 % of them 440 -> 195), and at half in larger launches (a lone spike in 64^3
    // 640 -> 207 us, 1 % of the samples 1170 -> 1114).  n = 16, k5_dense_f32 about 1 ms: at its end.
    const bool few = (long long)bricks * t_count <= device_sms();
    const int list_max = N == 8 ? (few ? 128 : 512) : kList;
    if (few)
        launch_g<N, 1>(wtab, V, gE, blocks, T, X, Y, bnd, feat, t_begin, t_step, t_count, bricks, dense, list_max, s);
    else
        launch_g<N, AGeo<N>::GROUPS>(wtab, V, gE, blocks, T, X, Y, bnd, feat, t_begin, t_step, t_count, bricks, dense,
                                     list_max, s);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace

cudaError_t spectra_adjoint_f32_slide_prepare(int n) {
    cudaError_t e = cudaErrorInvalidValue;
    if (n == 8) e = prepare_g<8, 1>();
    if (n == 16 && (e = prepare_g<16, 1>()) == cudaSuccess) e = prepare_g<16, 2>();
    return e;
}

SpectraAdjointGeometry spectra_adjoint_f32_slide_geometry(int n) {
    if (n == 8) return {kRun, Adj<8>::YH, Adj<8>::RX, Adj<8>::XH, Adj<8>::BLOCK_FLOATS, Adj<8>::SLICE};
    if (n == 16) return {kRun, Adj<16>::YH, Adj<16>::RX, Adj<16>::XH, Adj<16>::BLOCK_FLOATS, Adj<16>::SLICE};
    return {0, 0, 0, 0, 0, 0};
}

cudaError_t spectra_adjoint_f32_slide_launch(int n, const float* wtab, const float* V, const float* gE, float* blocks,
                                             int T, int X, int Y, int bnd, int feat, int t_begin, int t_step,
                                             int t_count, int* dense, cudaStream_t s) {
    if (t_step < 1 || t_count > 65535) return cudaErrorInvalidValue;
    if (n == 8) return launch_n<8>(wtab, V, gE, blocks, T, X, Y, bnd, feat, t_begin, t_step, t_count, dense, s);
    if (n == 16) return launch_n<16>(wtab, V, gE, blocks, T, X, Y, bnd, feat, t_begin, t_step, t_count, dense, s);
    return cudaErrorInvalidValue;
}

}  // namespace sal

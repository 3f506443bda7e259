// Register-resident pieces of the FP32 sliding-DFT kernels (rect cube, stride 1): short complex FFTs, the
// real DFT along t, and the sliding DFT along y with its |F| / Eq. 1 epilogue.
//
// Half spectrum in n/2 tiles instead of n/2 + 1.  The planes k_t = 0 and n/2 of a real cube are Hermitian in
// (k_x, k_y), so half of each is redundant; tile 0 holds the other halves of both:
//   rows 1 .. n/2-1:     (k_t = 0,   k_x = row)         the mirrored rows n - k_x doubled into the weights,
//   rows n/2+1 .. n-1:   (k_t = n/2, k_x = n - row)     likewise,
//   rows 0 and n/2:      k_x = 0 and n/2, whose y-signals are real: the signal of k_t = 0 as the real part
//                        and that of k_t = n/2 as the imaginary part of one complex row ("packed" row); with Z its
//                        spectrum, F_0[k] = (Z[k] + conj Z[-k]) / 2 and F_{n/2}[k] = (Z[k] - conj Z[-k]) / (2 i).
// Tiles 1 .. n/2 - 1 are k_t = 1 .. n/2 - 1.  n = 16: 8 tiles of 16 rows against 9, an eighth less of everything.
#pragma once

#include "spectra_f32_common.cuh"

namespace sal {
namespace f32 {

// cos and sin of 2 pi m / 32 (any integer m), for arguments the compiler knows.
__host__ __device__ constexpr float cos32q(int m) {   // 0 <= m <= 8
    return m == 0   ? 1.0f
           : m == 1 ? 0.98078528040323044913f
           : m == 2 ? 0.92387953251128675613f
           : m == 3 ? 0.83146961230254523708f
           : m == 4 ? 0.70710678118654752440f
           : m == 5 ? 0.55557023301960222474f
           : m == 6 ? 0.38268343236508977173f
           : m == 7 ? 0.19509032201612826785f
                    : 0.0f;
}
__host__ __device__ constexpr float cos32(int m) {
    m &= 31;
    if (m > 16) m = 32 - m;
    return m <= 8 ? cos32q(m) : -cos32q(16 - m);
}
__host__ __device__ constexpr float sin32(int m) { return cos32(m - 8); }

// a e^(-2 pi i m / 32), m known at compile time after unrolling
__device__ __forceinline__ float2 rot32(float2 a, int m) {
    m &= 31;
    if (m == 0) return a;
    if (m == 8) return make_float2(a.y, -a.x);
    if (m == 16) return make_float2(-a.x, -a.y);
    if (m == 24) return make_float2(-a.y, a.x);
    if (m == 4) return make_float2(cos32q(4) * (a.x + a.y), cos32q(4) * (a.y - a.x));
    if (m == 12) return make_float2(cos32q(4) * (a.y - a.x), -cos32q(4) * (a.x + a.y));
    const float c = cos32(m), s = sin32(m);
    return make_float2(fmaf(a.x, c, a.y * s), fmaf(a.y, c, -a.x * s));
}

// Position of output k of fft<N> (in place on naturally ordered inputs, the outputs bit-reversed).
template <int N> __host__ __device__ constexpr int fft_pos(int k) {
    int r = 0;
    for (int b = 1; b < N; b *= 2) r = 2 * r + ((k & b) ? 1 : 0);
    return r;
}

// X[k] = sum_u v[u] e^(-2 pi i k u / N) in place, X[k] at v[fft_pos<N>(k)].  N = 4 .. 32.  Decimation in time, a + w c and
// a - w c as two multiply-adds per component: no more operations than twiddling the differences, and one rounding less
// per component and level, which the weak bins of a strong cube show.
// ALT: bin N/2, the sum of alternating signs, from the differences of neighbours instead of the sums of the even and of the odd
// samples: on smooth data those are large and their difference is not.  N - 2 additions more; at N = 8, where it is an
// eighth of the bins, without it the error of weak bins is 1.2 times that of direct sums, with it 0.8 times.
template <int N, bool ALT = false> __device__ __forceinline__ void fft(float2 (&v)[N]) {
    float2 alt[N / 2];
    if (ALT) {
#pragma unroll
        for (int i = 0; i < N / 2; ++i) alt[i] = make_float2(v[2 * i].x - v[2 * i + 1].x, v[2 * i].y - v[2 * i + 1].y);
#pragma unroll
        for (int w = N / 4; w > 0; w /= 2)
#pragma unroll
            for (int i = 0; i < w; ++i) alt[i] = make_float2(alt[2 * i].x + alt[2 * i + 1].x, alt[2 * i].y + alt[2 * i + 1].y);
    }
#pragma unroll
    for (int st = 0; st < 5; ++st) {
        const int len = 2 << st;
        if (len > N) continue;
#pragma unroll
        for (int b = 0; b < N / 2; ++b) {
            const int j = b % (len / 2), l0 = (b / (len / 2)) * len + j, m = j * (32 / len);
            const int i0 = fft_pos<N>(l0), i1 = fft_pos<N>(l0 + len / 2);
            const float2 a = v[i0], c = v[i1];
            if (m == 0) {
                v[i0] = make_float2(a.x + c.x, a.y + c.y);
                v[i1] = make_float2(a.x - c.x, a.y - c.y);
            } else if (m == 8) {
                v[i0] = make_float2(a.x + c.y, a.y - c.x);
                v[i1] = make_float2(a.x - c.y, a.y + c.x);
            } else {
                const float wr = cos32(m), wi = sin32(m);   // w = wr - i wi
                v[i0] = make_float2(fmaf(c.x, wr, fmaf(c.y, wi, a.x)), fmaf(c.y, wr, fmaf(-c.x, wi, a.y)));
                v[i1] = make_float2(fmaf(-c.x, wr, fmaf(-c.y, wi, a.x)), fmaf(-c.y, wr, fmaf(c.x, wi, a.y)));
            }
        }
    }
    if (ALT) v[fft_pos<N>(N / 2)] = alt[0];
}

// sum_k X[k] e^(+2 pi i k u / N) (unnormalised inverse), output u at v[fft_pos<N>(u)]: the forward transform of the
// swapped parts, swapped.
template <int N> __device__ __forceinline__ void ifft(float2 (&v)[N]) {
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = make_float2(v[i].y, v[i].x);
    fft<N>(v);
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = make_float2(v[i].y, v[i].x);
}

// Bins 0 .. N/2 of the N real samples v[off], v[off + S], .. : decimation in time as fft, on half spectra (bins 0 and
// N/2 are real).  70 operations for N = 16; packing the samples in pairs into a complex transform takes 120 and mixes
// the rounding of strong bins into weak ones (31 % more error there at n = 8, 16 % at n = 16).
template <int N, int S, int L> __device__ __forceinline__ void half_dft(const float (&v)[L], int off, float2 (&X)[N / 2 + 1]) {
    if constexpr (N == 2) {
        X[0] = make_float2(v[off] + v[off + S], 0.f);
        X[1] = make_float2(v[off] - v[off + S], 0.f);
    } else {
        float2 e[N / 4 + 1], o[N / 4 + 1];
        half_dft<N / 2, 2 * S, L>(v, off, e);
        half_dft<N / 2, 2 * S, L>(v, off + S, o);
        X[0] = make_float2(e[0].x + o[0].x, 0.f);
        X[N / 2] = make_float2(e[0].x - o[0].x, 0.f);
        X[N / 4] = make_float2(e[N / 4].x, -o[N / 4].x);
#pragma unroll
        for (int k = 1; k < N / 4; ++k) {
            const float wr = cos32(k * (32 / N)), wi = sin32(k * (32 / N));   // w = wr - i wi
            X[k] = make_float2(fmaf(o[k].x, wr, fmaf(o[k].y, wi, e[k].x)), fmaf(o[k].y, wr, fmaf(-o[k].x, wi, e[k].y)));
            X[N / 2 - k] = make_float2(fmaf(-o[k].x, wr, fmaf(-o[k].y, wi, e[k].x)),
                                       -fmaf(-o[k].y, wr, fmaf(o[k].x, wi, e[k].y)));
        }
    }
}

// DFT of N real samples: out[0] = (bin 0, bin N/2) (both real), out[k] = bin k.  ALT as for fft.
template <int N, bool ALT = false> __device__ __forceinline__ void rfft(const float (&v)[N], float2 (&out)[N / 2]) {
    float2 X[N / 2 + 1];
    half_dft<N, 1, N>(v, 0, X);
    if (ALT) {
        float alt[N / 2];
#pragma unroll
        for (int i = 0; i < N / 2; ++i) alt[i] = v[2 * i] - v[2 * i + 1];
#pragma unroll
        for (int w = N / 4; w > 0; w /= 2)
#pragma unroll
            for (int i = 0; i < w; ++i) alt[i] = alt[2 * i] + alt[2 * i + 1];
        X[N / 2].x = alt[0];
    }
    out[0] = make_float2(X[0].x, X[N / 2].x);
#pragma unroll
    for (int k = 1; k < N / 2; ++k) out[k] = X[k];
}

// Adjoint of rfft: out[u] = Re sum_k d[k] e^(+2 pi i k u / N) over k = 1 .. N/2-1, plus d[0].x (bin 0) and
// (-1)^u d[0].y (bin N/2), as an N/2-point inverse of the even and odd outputs.
template <int N> __device__ __forceinline__ void rfft_adjoint(const float2 (&d)[N / 2], float (&out)[N]) {
    constexpr int M = N / 2;
    float2 z[M];
    z[0] = make_float2(d[0].x + d[0].y, d[0].x - d[0].y);
#pragma unroll
    for (int k = 1; k < M; ++k) {
        // with Y[k] = d[k] / 2, Z[k] = (Y[k] + conj Y[M-k]) + i e^(2 pi i k / N) (Y[k] - conj Y[M-k])
        const float2 a = d[k], b = d[M - k];
        const float2 e = make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y));
        const float2 o = rot32(make_float2(0.5f * (a.x - b.x), 0.5f * (a.y + b.y)), -k * (32 / N) - 8);
        z[k] = make_float2(e.x + o.x, e.y + o.y);
    }
    ifft<M>(z);
#pragma unroll
    for (int u = 0; u < M; ++u) {
        out[2 * u] = z[fft_pos<M>(u)].x;
        out[2 * u + 1] = z[fft_pos<M>(u)].y;
    }
}

// The stage-2 result of tile 0: Z[k] = spectrum along x of G1[k_t = 0] + i G1[k_t = n/2], v in fft order ->
// row r of the tile (see above).
template <int N> __device__ __forceinline__ float2 tile0_row(const float2 (&v)[N], int r) {
    if (r == 0 || r == N / 2) return v[fft_pos<N>(r)];
    if (r < N / 2) {
        const float2 a = v[fft_pos<N>(r)], b = v[fft_pos<N>(N - r)];
        return make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y));
    }
    const float2 a = v[fft_pos<N>(N - r)], b = v[fft_pos<N>(r)];
    return make_float2(0.5f * (a.y + b.y), 0.5f * (b.x - a.x));
}

// Its adjoint: from the gradients g of the rows to those of Z, in place (index = row, then k).
template <int N> __device__ __forceinline__ void tile0_adjoint(float2 (&g)[N]) {
#pragma unroll
    for (int r = 1; r < N / 2; ++r) {
        const float2 a = g[r], b = g[N - r];   // of F_0's and of F_{n/2}'s row
        g[r] = make_float2(0.5f * (a.x - b.y), 0.5f * (a.y + b.x));
        g[N - r] = make_float2(0.5f * (a.x + b.y), 0.5f * (b.x - a.y));
    }
}

// The bins one thread follows along y: M of them, twiddle index q = 0 .. M - 1, kept in pairs (bin k, bin n - k).
//   ODD = false: k = q n / M; slot 0 = (q = 0, q = M/2) (the self-paired bins), slot q = (q, M - q)
//   ODD = true:  k = 2 q + 1 (n = 32, M = 16); slot q = (q, M - 1 - q)
template <int M, bool ODD> struct Bins {
    static constexpr int NW = ODD ? M / 2 : M / 2 + 1;   // distinct |k_y|
    static constexpr __host__ __device__ int slot(int q) {
        if (ODD) return q < M / 2 ? q : M - 1 - q;
        return q == M / 2 ? 0 : (q < M / 2 ? q : M - q);
    }
    static constexpr __host__ __device__ bool second(int q) { return ODD ? q >= M / 2 : q >= M / 2; }
    static constexpr __host__ __device__ int ky(int w, int n) { return ODD ? 2 * w + 1 : w * (n / M); }   // |k_y| of weight w
    float2 r[M / 2], i[M / 2];   // per slot: (re, re), (im, im)

    __device__ __forceinline__ void set(int q, float2 f) {
        if (second(q)) { r[slot(q)].y = f.x; i[slot(q)].y = f.y; }
        else { r[slot(q)].x = f.x; i[slot(q)].x = f.y; }
    }
    // bin q += the entering minus the leaving sample times w^(k j), anchored at the start of the run:
    // F_{j+1}[k] = F_j[k] + d w^(k j) (d already times w32^j for the odd bins), w^(q j) = (-i)^s w^(m mod 8).
    __device__ __forceinline__ void slide(float2 d, int j) {
        float2 p[8];
#pragma unroll
        for (int m = 0; m < 8; m += 32 / M) p[m] = rot32(d, m);
#pragma unroll
        for (int q = 0; q < M; ++q) {
            const int m = (q * j * (32 / M)) & 31, s = m / 8;
            const float2 a = p[m % 8];
            const float dr = s == 0 ? a.x : s == 1 ? a.y : s == 2 ? -a.x : -a.y;
            const float di = s == 0 ? a.y : s == 1 ? -a.x : s == 2 ? -a.y : a.x;
            if (second(q)) { r[slot(q)].y += dr; i[slot(q)].y += di; }
            else { r[slot(q)].x += dr; i[slot(q)].x += di; }
        }
    }
    // adjoint of slide: sum_q F[q] e^(+2 pi i k j / n)
    __device__ __forceinline__ float2 at(int j) const {
        float2 p[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) p[m] = make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < M; ++q) {
            const int m = (q * j * (32 / M)) & 31, t = m / 8;
            const float2 f = get(q);
            p[m % 8].x += t == 0 ? f.x : t == 1 ? -f.y : t == 2 ? -f.x : f.y;
            p[m % 8].y += t == 0 ? f.y : t == 1 ? f.x : t == 2 ? -f.y : -f.x;
        }
        float2 e = make_float2(0.f, 0.f);
#pragma unroll
        for (int m = 0; m < 8; m += 32 / M) {
            const float2 a = rot32(p[m], -m);
            e.x += a.x;
            e.y += a.y;
        }
        return e;
    }
    // for loops that are not unrolled, sums kept in the phase of the current window: F <- F e^(2 pi i k / n) when the
    // window moves by one, and the sum of all bins
    __device__ __forceinline__ void turn() {
#pragma unroll
        for (int q = 0; q < M; ++q) set(q, rot32(get(q), -q * (32 / M)));
    }
    __device__ __forceinline__ float2 sum() const {
        float2 e = make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < M / 2; ++q) {
            e.x += r[q].x + r[q].y;
            e.y += i[q].x + i[q].y;
        }
        return e;
    }
    __device__ __forceinline__ float2 get(int q) const {
        return second(q) ? make_float2(r[slot(q)].y, i[slot(q)].y) : make_float2(r[slot(q)].x, i[slot(q)].x);
    }
    // the first window of a run, from its n samples g[0 .. n)
    template <int N, bool ALT = false> __device__ __forceinline__ void first(const float2* __restrict__ g) {
        float2 v[M];
        if (N == M) {
#pragma unroll
            for (int u = 0; u < M; ++u) v[u] = g[u];
        } else {
#pragma unroll
            for (int u = 0; u < M; ++u) {
                const float2 a = g[u], b = g[u + M];
                v[u] = ODD ? rot32(make_float2(a.x - b.x, a.y - b.y), u) : make_float2(a.x + b.x, a.y + b.y);
            }
        }
        fft<M, ALT>(v);
#pragma unroll
        for (int q = 0; q < M; ++q) set(q, v[fft_pos<M>(q)]);
    }
};

}  // namespace f32
}  // namespace sal

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

// Position of output k of fft<N> (decimation in frequency leaves the outputs bit-reversed).
template <int N> __host__ __device__ constexpr int fft_pos(int k) {
    int r = 0;
    for (int b = 1; b < N; b *= 2) r = 2 * r + ((k & b) ? 1 : 0);
    return r;
}

// X[k] = sum_u v[u] e^(-2 pi i k u / N) in place, X[k] at v[fft_pos<N>(k)].  N = 4 .. 32.
template <int N> __device__ __forceinline__ void fft(float2 (&v)[N]) {
#pragma unroll
    for (int st = 0; st < 5; ++st) {
        const int len = N >> st;
        if (len < 2) continue;
#pragma unroll
        for (int b = 0; b < N / 2; ++b) {
            const int j = b % (len / 2), i0 = (b / (len / 2)) * len + j, i1 = i0 + len / 2;
            const float2 a = v[i0], c = v[i1];
            v[i0] = make_float2(a.x + c.x, a.y + c.y);
            v[i1] = rot32(make_float2(a.x - c.x, a.y - c.y), j * (32 / len));
        }
    }
}

// DFT of N real samples, bins 0 .. N/2, as an N/2-point complex FFT of (v[2u], v[2u+1]):
// out[0] = (bin 0, bin N/2) (both real), out[k] = bin k.
template <int N> __device__ __forceinline__ void rfft(const float (&v)[N], float2 (&out)[N / 2]) {
    constexpr int M = N / 2;
    float2 z[M];
#pragma unroll
    for (int u = 0; u < M; ++u) z[u] = make_float2(v[2 * u], v[2 * u + 1]);
    fft<M>(z);
    out[0] = make_float2(z[0].x + z[0].y, z[0].x - z[0].y);
#pragma unroll
    for (int k = 1; k < M; ++k) {
        const float2 a = z[fft_pos<M>(k)], b = z[fft_pos<M>(M - k)];
        const float2 e = make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y));          // even samples
        const float2 o = rot32(make_float2(0.5f * (a.y + b.y), 0.5f * (b.x - a.x)), k * (32 / N));   // odd samples
        out[k] = make_float2(e.x + o.x, e.y + o.y);
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
    // F_{j+1}[k] = F_j[k] + d w^(k j) (d already times w32^j for the odd bins), w^(q j) = (-i)^s w^(m mod 8)
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
    // the first window of a run, from its n samples g[0 .. n)
    template <int N> __device__ __forceinline__ void first(const float2* __restrict__ g) {
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
        fft<M>(v);
#pragma unroll
        for (int q = 0; q < M; ++q) set(q, v[fft_pos<M>(q)]);
    }
};

}  // namespace f32
}  // namespace sal

// Small bins of the FP32 spectral adjoint: the bins of a cube whose FP32 spectrum gives no usable direction
// F / |F| (k_spectra_bwd_f32.cu says which and why), resolved exactly.  The integer test for the bins that the
// border extension makes vanish, and the float-float arithmetic of the direct sums of the others.
#pragma once

#include <cmath>

#include "spectra_f32_common.cuh"

namespace sal {
namespace f32 {

constexpr float kSmallBin = 1.0f / 65536.0f;       // FP32 |F| / A_p at or below which a bin is resolved exactly
constexpr float kZeroBin = 1.0f / 68719476736.0f;  // float-float max(|Re F|, |Im F|) / A_p at or below which F = 0

// Float-float constants of the exact recompute: cos, sin of 2 pi m / n and the taper h(u), each as a pair
// (hi, lo) of FP32 values whose sum is the double-precision value.
template <int N> struct Exact2f {
    float ch[N], cl[N], sh[N], sl[N], hh[N], hl[N];
};

// Masks of the bins that vanish for every input, per axis (t, x, y): bit k of the mask of position p
// (the cube's samples p - n/2 .. p + n/2 - 1 of that axis) is set when bin k of that axis vanishes.
// Positions whose cube lies inside the axis never vanish; the others are p < n (entries 0 .. n-1) and
// p >= L - n (entries n .. 2n-1).
struct VanishTab {
    uint16_t m[3][32];
    int L[3];
};

__device__ __forceinline__ uint32_t vanish_mask(const VanishTab& v, int a, int p, int n) {
    const int L = v.L[a];
    if (p - n / 2 >= 0 && p + n / 2 - 1 < L) return 0u;
    return p < n ? v.m[a][p] : v.m[a][n + (p - (L - n))];
}

// Host: does bin k of the one-axis cube at position p (axis length L) vanish for every input?  The bin is
// sum_m h(m) w^(k m) x[src(m)] (w = exp(-2 pi i / n)), so it vanishes for all x iff, for each source
// sample j, the coefficient sum_{m: src(m) = j} h(m) w^(k m) is 0.  With n a power of two, w has minimal
// polynomial w^(n/2) + 1, so the coefficient is zero iff its coordinates on w^0 .. w^(n/2-1)
// (w^(e + n/2) = -w^e) are; they are integers for the rect taper (h = 1) and, scaled by 4, for the
// periodic Hann taper (4 h(m) w^(km) = 2 w^(km) - w^(km+m) - w^(km-m)).  Exact: no rounding enters.
inline bool axis_bin_vanishes(int n, int p, int L, int bnd, int taper, int k) {
    if (p - n / 2 >= 0 && p + n / 2 - 1 < L) return false;
    int src[32];
    for (int m = 0; m < n; ++m) src[m] = ext_index(p - n / 2 + m, L, bnd);
    for (int m = 0; m < n; ++m) {
        if (src[m] < 0) continue;
        bool first = true;
        for (int q = 0; q < m; ++q) first = first && src[q] != src[m];
        if (!first) continue;
        int a[16] = {0};
        for (int q = m; q < n; ++q) {
            if (src[q] != src[m]) continue;
            const int e0 = (k * q) % n;
            const int es[3] = {e0, (e0 + q) % n, (e0 - q + n) % n};
            const int vs[3] = {taper ? 2 : 1, taper ? -1 : 0, taper ? -1 : 0};
            for (int r = 0; r < 3; ++r) {
                if (es[r] < n / 2) a[es[r]] += vs[r];
                else a[es[r] - n / 2] -= vs[r];
            }
        }
        for (int e = 0; e < n / 2; ++e)
            if (a[e] != 0) return false;
    }
    return true;
}

inline uint16_t axis_vanish_mask(int n, int p, int L, int bnd, int taper) {
    uint16_t mk = 0;
    for (int k = 0; k < n; ++k)
        if (axis_bin_vanishes(n, p, L, bnd, taper, k)) mk = (uint16_t)(mk | (1u << k));
    return mk;
}

inline VanishTab make_vanish_tab(int n, int T, int X, int Y, int bnd, int taper) {
    VanishTab v{};
    const int L[3] = {T, X, Y};
    for (int a = 0; a < 3; ++a) {
        v.L[a] = L[a];
        for (int p = 0; p < n && p < L[a]; ++p) v.m[a][p] = axis_vanish_mask(n, p, L[a], bnd, taper);
        for (int p = L[a] - n > 0 ? L[a] - n : 0; p < L[a]; ++p)
            v.m[a][n + (p - (L[a] - n))] = axis_vanish_mask(n, p, L[a], bnd, taper);
    }
    return v;
}

// Float-float arithmetic (an unevaluated sum hi + lo of two FP32 values): the error-free transformations
// two-sum (Knuth) and the FMA product residual, with the usual renormalisation.
struct FF {
    float hi, lo;
};
__device__ __forceinline__ FF ff_fast_two_sum(float a, float b) {   // |a| >= |b|
    const float s = a + b;
    return {s, b - (s - a)};
}
__device__ __forceinline__ FF ff_add(FF a, FF b) {
    const float s = a.hi + b.hi;
    const float bb = s - a.hi;
    const float e = (a.hi - (s - bb)) + (b.hi - bb);
    return ff_fast_two_sum(s, e + a.lo + b.lo);
}
__device__ __forceinline__ FF ff_mul(FF a, FF b) {
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
    return ff_fast_two_sum(p, e);
}
__device__ __forceinline__ FF ff_mul1(float a, FF b) {   // a exact in FP32
    const float p = a * b.hi;
    return ff_fast_two_sum(p, fmaf(a, b.lo, fmaf(a, b.hi, -p)));
}

// s += v (ch + cl): the rounded product by an error-free sum, its residuals into the low part.
__device__ __forceinline__ void ff_gather(FF& s, float v, float ch, float cl) {
    const float p = v * ch, e = fmaf(v, cl, fmaf(v, ch, -p));
    const float t = s.hi + p, b = t - s.hi;
    s.lo += ((s.hi - (t - b)) + (p - b)) + e;
    s.hi = t;
}

// The float-float constants of the exact recompute of small bins: cos, sin (2 pi m / n) and the taper
// (rect, or the periodic Hann window 1/2 - cos(2 pi u / n) / 2), from the host's double-precision libm,
// each split into an FP32 head and the FP32 rounding of the remainder.
template <int N>
inline Exact2f<N> make_exact2f(int taper) {
    Exact2f<N> e;
    auto split = [](double v, float& hi, float& lo) {
        hi = (float)v;
        lo = (float)(v - (double)hi);
    };
    for (int m = 0; m < N; ++m) {
        const double a = 2.0 * 3.14159265358979323846 * m / N;
        split(cos(a), e.ch[m], e.cl[m]);
        split(sin(a), e.sh[m], e.sl[m]);
        split(taper ? 0.5 - 0.5 * cos(a) : 1.0, e.hh[m], e.hl[m]);
    }
    return e;
}

}  // namespace f32
}  // namespace sal

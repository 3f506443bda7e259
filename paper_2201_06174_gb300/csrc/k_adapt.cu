// K3a: the paper's adaptive weight update (LMS, NLMS, RLS; Eq. 4 and the adaptive scheme around it)
// run as the sequential filters they are: one recursion per chain, in FP64, over the voxels in the
// order inline sections (y) outermost, then x, then t.  Chains are independent blocks of `sections`
// inline sections (the re-adaptation after every N sections the paper allows); sections = 0 is one
// chain over the whole volume.  One warp per chain: the lanes stage the normalised maps
// x_m = (S_m - lo_m) / (hi_m - lo_m) and the desired value d of the next 32 steps in shared memory
// while lane 0 runs the FP64 recursion over the current 32 (a single FP64 chain; FP64 throughput on
// this part is low, so no lane repeats it).
//   LMS:  W += mu e x
//   NLMS: W += mu e x / (eps + |x|^2)
//   RLS:  k = P x / (lambda + x'Px);  W += k e;  P = (P - k x'P) / lambda,  P0 = I/delta
// with e = d - W.x; W0 = (1/3, 1/3, 1/3) for LMS and NLMS, 0 for RLS.
//
// One chain is bound by the latency of its dependent FP64 operations (0.80 us a step for NLMS: 709 ms for
// the 884,736 steps of a 96^3 volume, with one lane of the GPU at work).  Its steps can be regrouped,
// since each one is an affine map of the weights (LMS, NLMS: W -> (I - g x x') W + g d x) or adds to a sum
// (RLS with lambda = 1: R += x x', z += x d, with P = R^-1 and W = R^-1 z), and both compose associatively:
//   k3_adapt_segments  a thread per segment of L steps of one section: the segment's map, then by a tree
//                      the map of the block's 32 segments of each section (FP64 throughput: about 40
//                      operations a step at 2 per clock and SM);
//   k3_adapt_chain     a block per chain: the weights at the start of each group of 32 segments, and W_out;
//   k3_adapt_errors    (only for err2) each segment's steps again from its own starting weights, all at once.
// All in FP64; 96^3, NLMS with err2: 708.1 -> 0.25 ms a call.  Chains the regrouping could make less exact than
// the step-by-step filter are marked and left to it (k3_adapt): maps that grow (an entry above kGrow: LMS or NLMS
// with a step size beyond their stability limit, or values that are not finite), and RLS whose R is near singular (kPivot).
#include <algorithm>
#include <cfloat>

#include "reduce_tail.cuh"

namespace sal {
namespace {

enum : int { ADAPT_LMS = 0, ADAPT_NLMS = 1, ADAPT_RLS = 2 };
enum : int { kTodoChain = 1, kTodoErrors = 2 };

__global__ void __launch_bounds__(32)
k3_adapt(const float* __restrict__ S3, const float* __restrict__ D, int T, int X, int Y, int method, double mu,
         double eps, double lambda, double delta, int sec, const float* __restrict__ norm, float* __restrict__ W_out,
         float* __restrict__ err2, const int* __restrict__ todo, unsigned* __restrict__ counter) {
    if (blockIdx.x == 0 && threadIdx.x == 0) counter[tail::C_MAPS] = 0u;   // (reduce_tail.cuh)
    // todo (nullable): per chain, what the regrouped form has left to this kernel: nothing, all (kTodoChain) or only the
    // errors (kTodoErrors: its weights stand, and are the same whether err2 is asked for or not)
    const int left = todo ? todo[blockIdx.x] : kTodoChain;
    if (left == 0) return;
    __shared__ double s_x[2][4][32];   // two chunks of 32 steps: x_t, x_x, x_y, d
    const long long NV = (long long)T * X * Y;
    const int lane = threadIdx.x;
    const int y_begin = blockIdx.x * sec, y_end = min(Y, y_begin + sec);
    const long long steps = (long long)(y_end - y_begin) * X * T;
    const long long first = (long long)y_begin * X * T;   // index of this chain's first step in filter order
    const double lo0 = norm[0], lo1 = norm[1], lo2 = norm[2];
    const double iv0 = norm[3], iv1 = norm[4], iv2 = norm[5];
    const double inv_lambda = 1.0 / lambda;
    // the recursion state lives in lane 0 (one FP64 chain; the other lanes stage the next chunk)
    double w0, w1, w2;
    if (method == ADAPT_RLS) w0 = w1 = w2 = 0.0;
    else w0 = w1 = w2 = 1.0 / 3.0;
    double P[3][3] = {{1.0 / delta, 0.0, 0.0}, {0.0, 1.0 / delta, 0.0}, {0.0, 0.0, 1.0 / delta}};
    auto stage = [&](long long base, int buf) {
        const long long s = base + lane;
        double a0 = 0.0, a1 = 0.0, a2 = 0.0, dv = 0.0;
        if (s < steps) {
            const int t = (int)(s % T), x = (int)((s / T) % X), y = y_begin + (int)(s / ((long long)T * X));
            const long long p = ((long long)t * X + x) * Y + y;
            a0 = ((double)__ldg(S3 + p) - lo0) * iv0;
            a1 = ((double)__ldg(S3 + NV + p) - lo1) * iv1;
            a2 = ((double)__ldg(S3 + 2 * NV + p) - lo2) * iv2;
            dv = (double)__ldg(D + p);
        }
        s_x[buf][0][lane] = a0;
        s_x[buf][1][lane] = a1;
        s_x[buf][2][lane] = a2;
        s_x[buf][3][lane] = dv;
    };
    stage(0, 0);
    __syncwarp();
    int buf = 0;
    for (long long base = 0; base < steps; base += 32, buf ^= 1) {
        if (base + 32 < steps) stage(base + 32, buf ^ 1);   // the next chunk, while lane 0 runs this one
        if (lane == 0) {
            const int cnt = steps - base < 32 ? (int)(steps - base) : 32;
            for (int i = 0; i < cnt; ++i) {
                const double x0 = s_x[buf][0][i], x1 = s_x[buf][1][i], x2 = s_x[buf][2][i], d = s_x[buf][3][i];
                const double e = d - (w0 * x0 + w1 * x1 + w2 * x2);
                if (err2) err2[first + base + i] = (float)(e * e);
                if (method == ADAPT_LMS) {
                    w0 += mu * e * x0;
                    w1 += mu * e * x1;
                    w2 += mu * e * x2;
                } else if (method == ADAPT_NLMS) {
                    const double g = mu * e / (eps + (x0 * x0 + x1 * x1 + x2 * x2));
                    w0 += g * x0;
                    w1 += g * x1;
                    w2 += g * x2;
                } else {
                    double Px[3], xP[3];
#pragma unroll
                    for (int r = 0; r < 3; ++r) {
                        Px[r] = P[r][0] * x0 + P[r][1] * x1 + P[r][2] * x2;
                        xP[r] = x0 * P[0][r] + x1 * P[1][r] + x2 * P[2][r];
                    }
                    const double inv_den = 1.0 / (lambda + x0 * Px[0] + x1 * Px[1] + x2 * Px[2]);
                    const double k0 = Px[0] * inv_den, k1 = Px[1] * inv_den, k2 = Px[2] * inv_den;
                    w0 += k0 * e;
                    w1 += k1 * e;
                    w2 += k2 * e;
                    const double kk[3] = {k0, k1, k2};
#pragma unroll
                    for (int r = 0; r < 3; ++r)
#pragma unroll
                        for (int c = 0; c < 3; ++c) P[r][c] = (P[r][c] - kk[r] * xP[c]) * inv_lambda;
                }
            }
        }
        __syncwarp();
    }
    if (lane == 0 && left == kTodoChain) {
        W_out[blockIdx.x * 3 + 0] = (float)w0;
        W_out[blockIdx.x * 3 + 1] = (float)w1;
        W_out[blockIdx.x * 3 + 2] = (float)w2;
    }
}

// ---- The regrouped form -------------------------------------------------------------------------
constexpr int kSegY = 4;               // sections of a block: with 8 (a whole 32-byte sector of S3 and D) too few blocks to
                                       // share the SMs evenly, NLMS with errors on 48^3, 96^3, 128^3: 139, 255 and 432 us against
                                       // 175, 293 and 528 (200^3 1545 against 1489)
constexpr int kSegS = 32;              // segments of each section in a block
constexpr int kSegThreads = kSegY * kSegS;
constexpr int kMinSeg = 16;            // steps of a segment at least: the maps' composition costs what ~1.5 steps cost
constexpr int kChainThreads = 256;     // chunks of a chain's groups, in kChainRows rows: chunks, then rows, are composed
constexpr int kChainRows = 16;         // side by side (the rows by lanes of one warp: a partly filled warp takes as much of
                                       // the FP64 pipe as a full one), and only the rows' maps one after the other
constexpr double kGrow = 16.0;         // largest entry of a map that counts as stable (a contraction's is at most 1)
constexpr double kPivot = 1e-7;        // smallest Cholesky pivot of R over its trace

// The state one segment contributes: LMS / NLMS the map W -> A W + b, RLS the sums R (6) and z (3).
template <bool RLS> struct SegState;
template <> struct SegState<false> {
    static constexpr int K = 12;
    double v[12];   // A row-major, then b
    __device__ __forceinline__ void identity() {
#pragma unroll
        for (int i = 0; i < 12; ++i) v[i] = i < 9 && i % 4 == 0 ? 1.0 : 0.0;
    }
    // one step: A -= g x (x'A), b += g x (d - x'b)
    __device__ __forceinline__ void step(const double (&x)[3], double d, double g) {
        double xa[4];
#pragma unroll
        for (int c = 0; c < 3; ++c) xa[c] = x[0] * v[c] + x[1] * v[3 + c] + x[2] * v[6 + c];
        xa[3] = d - (x[0] * v[9] + x[1] * v[10] + x[2] * v[11]);
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const double gx = g * x[r];
#pragma unroll
            for (int c = 0; c < 3; ++c) v[3 * r + c] -= gx * xa[c];
            v[9 + r] += gx * xa[3];
        }
    }
    // this, then `later`
    __device__ __forceinline__ void then(const SegState& l) {
        double o[12];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
                o[3 * r + c] = l.v[3 * r] * v[c] + l.v[3 * r + 1] * v[3 + c] + l.v[3 * r + 2] * v[6 + c];
            o[9 + r] = l.v[3 * r] * v[9] + l.v[3 * r + 1] * v[10] + l.v[3 * r + 2] * v[11] + l.v[9 + r];
        }
#pragma unroll
        for (int i = 0; i < 12; ++i) v[i] = o[i];
    }
    __device__ __forceinline__ bool bad() const {
        bool ok = true;
#pragma unroll
        for (int i = 0; i < 12; ++i) ok = ok && fabs(v[i]) <= (i < 9 ? kGrow : DBL_MAX);   // false for NaN
        return !ok;
    }
};
template <> struct SegState<true> {
    static constexpr int K = 9;
    double v[9];   // R00, R01, R02, R11, R12, R22, z
    __device__ __forceinline__ void identity() {
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = 0.0;
    }
    __device__ __forceinline__ void step(const double (&x)[3], double d, double) {
        v[0] += x[0] * x[0]; v[1] += x[0] * x[1]; v[2] += x[0] * x[2];
        v[3] += x[1] * x[1]; v[4] += x[1] * x[2]; v[5] += x[2] * x[2];
#pragma unroll
        for (int r = 0; r < 3; ++r) v[6 + r] += x[r] * d;
    }
    __device__ __forceinline__ void then(const SegState& l) {
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] += l.v[i];
    }
    __device__ __forceinline__ bool bad() const {
        bool ok = true;
#pragma unroll
        for (int i = 0; i < 9; ++i) ok = ok && fabs(v[i]) <= DBL_MAX;
        return !ok;
    }
};

// The weights (and P) a chain starts a segment with.  LMS / NLMS carry W; RLS carries the sums R, z.
template <bool RLS> struct Start;
template <> struct Start<false> {
    static constexpr int K = 3;
    double v[3];
    __device__ __forceinline__ void first(double) { v[0] = v[1] = v[2] = 1.0 / 3.0; }
    __device__ __forceinline__ void advance(const SegState<false>& s) {
        const double a = s.v[0] * v[0] + s.v[1] * v[1] + s.v[2] * v[2] + s.v[9];
        const double b = s.v[3] * v[0] + s.v[4] * v[1] + s.v[5] * v[2] + s.v[10];
        const double c = s.v[6] * v[0] + s.v[7] * v[1] + s.v[8] * v[2] + s.v[11];
        v[0] = a; v[1] = b; v[2] = c;
    }
    __device__ __forceinline__ bool weights(double (&w)[3], double (&)[6]) const {
        w[0] = v[0]; w[1] = v[1]; w[2] = v[2];
        return true;
    }
};
template <> struct Start<true> {
    static constexpr int K = 9;
    double v[9];
    __device__ __forceinline__ void first(double delta) {
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = 0.0;
        v[0] = v[3] = v[5] = delta;
    }
    __device__ __forceinline__ void advance(const SegState<true>& s) {
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] += s.v[i];
    }
    // P = R^-1 by a Cholesky factorisation R = L D L', W = P z; false when R is too near singular for it (the
    // chain's start, R = delta I, is not)
    __device__ __forceinline__ bool weights(double (&w)[3], double (&P)[6]) const {
        const double d0 = v[0], l10 = v[1] / d0, l20 = v[2] / d0;
        const double d1 = v[3] - l10 * v[1], m = v[4] - l10 * v[2], l21 = m / d1;
        const double d2 = v[5] - l20 * v[2] - l21 * m;
        const double lim = kPivot * (v[0] + v[3] + v[5]);
        if (!(d0 > lim && d1 > lim && d2 > lim && d0 <= DBL_MAX)) return false;
        const double i2 = 1.0 / d2, i1 = 1.0 / d1, i0 = 1.0 / d0;
        P[5] = i2;
        P[4] = -l21 * i2;
        P[3] = i1 - l21 * P[4];
        P[2] = -l10 * P[4] - l20 * P[5];
        P[1] = -l10 * P[3] - l20 * P[4];
        P[0] = i0 - l10 * P[1] - l20 * P[2];
        w[0] = P[0] * v[6] + P[1] * v[7] + P[2] * v[8];
        w[1] = P[1] * v[6] + P[3] * v[7] + P[4] * v[8];
        w[2] = P[2] * v[6] + P[4] * v[7] + P[5] * v[8];
        return true;
    }
};

// Segments: section y's steps r = x T + t in [seg L, (seg + 1) L); groups of kSegS of them.
struct SegGeo {
    int T, X, Y, sec, L, nseg, ngroup;   // ngroup = ceil(nseg / kSegS)
    int method;
    double mu, eps, delta;
};

// (double)f on the integer pipe for zeros and normal numbers: the FP64 pipe, which bounds these kernels, also converts.
__device__ __forceinline__ double widen(float f) {
    const unsigned b = __float_as_uint(f), e = (b >> 23) & 255u;
    if (e - 1u >= 254u) return (b << 1) == 0u ? 0.0 : (double)f;
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}

// 1 / d by Newton's iteration from the FP32 reciprocal (2^-22, then 2^-44, then FP64's rounding): 4 multiply-adds of the
// FP64 pipe; outside FP32's range the division.
__device__ __forceinline__ double reciprocal(double d) {
    const float f = (float)d;
    if (!(f >= 1e-30f && f <= 1e30f)) return 1.0 / d;
    double y = widen(__fdividef(1.0f, f));
    y = fma(y, fma(-d, y, 1.0), y);
    return fma(y, fma(-d, y, 1.0), y);
}

// The normalised maps and the desired value of step r of section y (nlo = -lo iv).
__device__ __forceinline__ void seg_load(const float* __restrict__ S3, const float* __restrict__ D, const SegGeo& g,
                                         long long NV, const double (&nlo)[3], const double (&iv)[3], int y, int t, int xi,
                                         double (&x)[3], double& d) {
    const long long p = ((long long)t * g.X + xi) * g.Y + y;
#pragma unroll
    for (int m = 0; m < 3; ++m) x[m] = fma(widen(__ldg(S3 + m * NV + p)), iv[m], nlo[m]);
    d = widen(__ldg(D + p));
}

template <bool RLS>
__global__ void __launch_bounds__(kSegThreads)
k3_adapt_segments(const float* __restrict__ S3, const float* __restrict__ D, SegGeo g, const float* __restrict__ norm,
                  double* __restrict__ segs, double* __restrict__ groups, int* __restrict__ todo) {
    using St = SegState<RLS>;
    __shared__ double s_v[St::K][kSegThreads];
    const long long NV = (long long)g.T * g.X * g.Y;
    const int yl = threadIdx.x % kSegY, sl = threadIdx.x / kSegY;
    const int y = blockIdx.y * kSegY + yl, seg = blockIdx.x * kSegS + sl;
    const double iv[3] = {norm[3], norm[4], norm[5]}, nlo[3] = {-(norm[0] * iv[0]), -(norm[1] * iv[1]), -(norm[2] * iv[2])};
    St s;
    s.identity();
    if (y < g.Y && seg < g.nseg) {
        const long long per = (long long)g.X * g.T, r0 = (long long)seg * g.L;
        const int cnt = (int)(per - r0 < g.L ? per - r0 : g.L);
        int xi = (int)(r0 / g.T), t = (int)(r0 - (long long)xi * g.T);
        double x[3], d;
        seg_load(S3, D, g, NV, nlo, iv, y, t, xi, x, d);
        for (int i = 0; i < cnt; ++i) {
            if (++t == g.T) { t = 0; ++xi; }
            double xn[3] = {0.0, 0.0, 0.0}, dn = 0.0;
            if (i + 1 < cnt) seg_load(S3, D, g, NV, nlo, iv, y, t, xi, xn, dn);   // under this step's arithmetic
            const double gain = RLS ? 0.0
                                : g.method == ADAPT_NLMS
                                    ? g.mu * reciprocal(g.eps + (x[0] * x[0] + x[1] * x[1] + x[2] * x[2]))
                                    : g.mu;
            s.step(x, d, gain);
            x[0] = xn[0]; x[1] = xn[1]; x[2] = xn[2];
            d = dn;
        }
        double* o = segs + ((long long)y * g.nseg + seg) * St::K;
#pragma unroll
        for (int i = 0; i < St::K; ++i) o[i] = s.v[i];
        if (s.bad()) todo[y / g.sec] = kTodoChain;
    }
    // the group's state: a tree over its 32 segments in order (absent ones are the identity)
#pragma unroll
    for (int i = 0; i < St::K; ++i) s_v[i][threadIdx.x] = s.v[i];
    for (int h = 1; h < kSegS; h *= 2) {
        __syncthreads();
        if (sl % (2 * h) == 0) {
            St l;
#pragma unroll
            for (int i = 0; i < St::K; ++i) l.v[i] = s_v[i][threadIdx.x + h * kSegY];
            s.then(l);
#pragma unroll
            for (int i = 0; i < St::K; ++i) s_v[i][threadIdx.x] = s.v[i];
        }
    }
    if (sl == 0 && y < g.Y) {
        double* o = groups + ((long long)y * g.ngroup + blockIdx.x) * St::K;
#pragma unroll
        for (int i = 0; i < St::K; ++i) o[i] = s.v[i];
        if (s.bad()) todo[y / g.sec] = kTodoChain;
    }
}

// One block per chain: its groups (section by section) in kChainThreads contiguous chunks, each composed by one thread; 16
// lanes compose 16 chunks each; thread 0 applies these rows in order; the lanes then walk their chunks, and each thread its
// groups, from their starts.
template <bool RLS>
__global__ void __launch_bounds__(kChainThreads)
k3_adapt_chain(SegGeo g, const double* __restrict__ groups, double* __restrict__ starts, float* __restrict__ W_out,
               int* __restrict__ todo) {
    using St = SegState<RLS>;
    using Sa = Start<RLS>;
    constexpr int kPerRow = kChainThreads / kChainRows, kPitch = kPerRow + 1;   // rows one double apart in the banks
    __shared__ double s_v[St::K][kChainRows * kPitch], s_r[St::K][kChainRows], s_st[Sa::K][kChainRows * kPitch];
    const int y0 = blockIdx.x * g.sec, y1 = min(g.Y, y0 + g.sec), tid = threadIdx.x;
    const int slot = tid / kPerRow * kPitch + tid % kPerRow;
    const long long base = (long long)y0 * g.ngroup, total = (long long)(y1 - y0) * g.ngroup;
    const long long per = (total + kChainThreads - 1) / kChainThreads;
    const long long a = min(total, per * tid), b = min(total, a + per);
    auto group = [&](long long i) {
        St l;
#pragma unroll
        for (int k = 0; k < St::K; ++k) l.v[k] = __ldg(groups + (base + i) * St::K + k);
        return l;
    };
    auto get = [&](St& l, int i) {
#pragma unroll
        for (int k = 0; k < St::K; ++k) l.v[k] = s_v[k][i];
    };
    St s;
    s.identity();
    if (a < b) {
        s = group(a);
        for (long long i = a + 1; i < b; ++i) s.then(group(i));
    }
#pragma unroll
    for (int k = 0; k < St::K; ++k) s_v[k][slot] = s.v[k];
    __syncthreads();
    bool unsound = s.bad();
    if (tid < kChainRows) {
        get(s, tid * kPitch);
        for (int i = 1; i < kPerRow; ++i) {
            St l;
            get(l, tid * kPitch + i);
            s.then(l);
        }
        unsound = unsound || s.bad();
#pragma unroll
        for (int k = 0; k < St::K; ++k) s_r[k][tid] = s.v[k];
    }
    const int bad = __syncthreads_or(unsound);
    if (bad || todo[blockIdx.x]) {
        __syncthreads();
        if (tid == 0) todo[blockIdx.x] = kTodoChain;
        return;   // block-uniform: the step-by-step filter takes this chain
    }
    Sa st;
    if (tid == 0) {
        st.first(g.delta);
        for (int i = 0; i < kChainRows; ++i) {
            St l;
#pragma unroll
            for (int k = 0; k < Sa::K; ++k) s_st[k][i * kPitch] = st.v[k];
#pragma unroll
            for (int k = 0; k < St::K; ++k) l.v[k] = s_r[k][i];
            st.advance(l);
        }
        double w[3], P[6];
        if (st.weights(w, P)) {
#pragma unroll
            for (int m = 0; m < 3; ++m) W_out[blockIdx.x * 3 + m] = (float)w[m];
        } else {
            todo[blockIdx.x] = kTodoChain;
        }
    }
    if (!starts) return;
    __syncthreads();
    if (tid < kChainRows) {
#pragma unroll
        for (int k = 0; k < Sa::K; ++k) st.v[k] = s_st[k][tid * kPitch];
        for (int i = 1; i < kPerRow; ++i) {
            St l;
            get(l, tid * kPitch + i - 1);
            st.advance(l);
#pragma unroll
            for (int k = 0; k < Sa::K; ++k) s_st[k][tid * kPitch + i] = st.v[k];
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < Sa::K; ++k) st.v[k] = s_st[k][slot];
    for (long long i = a; i < b; ++i) {
#pragma unroll
        for (int k = 0; k < Sa::K; ++k) starts[(base + i) * Sa::K + k] = st.v[k];
        st.advance(group(i));
    }
}

// The squared error of every step: each segment's steps again, from the weights its predecessors leave.
template <bool RLS>
__global__ void __launch_bounds__(kSegThreads)
k3_adapt_errors(const float* __restrict__ S3, const float* __restrict__ D, SegGeo g, const float* __restrict__ norm,
                const double* __restrict__ segs, const double* __restrict__ starts, float* __restrict__ err2,
                int* __restrict__ todo) {
    using St = SegState<RLS>;
    using Sa = Start<RLS>;
    __shared__ double s_v[St::K][kSegThreads], s_st[Sa::K][kSegThreads];
    const long long NV = (long long)g.T * g.X * g.Y;
    const int yl = threadIdx.x % kSegY, sl = threadIdx.x / kSegY;
    const int y = blockIdx.y * kSegY + yl, seg = blockIdx.x * kSegS + sl;
    const bool live = y < g.Y && seg < g.nseg;
    if (live) {
        const double* o = segs + ((long long)y * g.nseg + seg) * St::K;
#pragma unroll
        for (int i = 0; i < St::K; ++i) s_v[i][threadIdx.x] = __ldg(o + i);
    }
    __syncthreads();
    if (sl == 0 && y < g.Y) {
        Sa st;
#pragma unroll
        for (int k = 0; k < Sa::K; ++k) st.v[k] = starts[((long long)y * g.ngroup + blockIdx.x) * Sa::K + k];
        for (int i = 0; i < kSegS && blockIdx.x * kSegS + i < g.nseg; ++i) {
            const int j = yl + i * kSegY;
            St l;
#pragma unroll
            for (int k = 0; k < Sa::K; ++k) s_st[k][j] = st.v[k];
#pragma unroll
            for (int k = 0; k < St::K; ++k) l.v[k] = s_v[k][j];
            st.advance(l);
        }
    }
    __syncthreads();
    if (!live) return;
    Sa st;
#pragma unroll
    for (int k = 0; k < Sa::K; ++k) st.v[k] = s_st[k][threadIdx.x];
    double w[3], P[6];
    const long long per = (long long)g.X * g.T, r0 = (long long)seg * g.L;
    if (!st.weights(w, P)) {   // a segment inside the chain where R is still near singular
        if (todo[y / g.sec] == 0) todo[y / g.sec] = kTodoErrors;
        return;
    }
    const double iv[3] = {norm[3], norm[4], norm[5]}, nlo[3] = {-(norm[0] * iv[0]), -(norm[1] * iv[1]), -(norm[2] * iv[2])};
    const int cnt = (int)(per - r0 < g.L ? per - r0 : g.L);
    int xi = (int)(r0 / g.T), t = (int)(r0 - (long long)xi * g.T);
    float* out = err2 + (long long)y * per + r0;
    double x[3], d;
    seg_load(S3, D, g, NV, nlo, iv, y, t, xi, x, d);
    for (int i = 0; i < cnt; ++i) {
        if (++t == g.T) { t = 0; ++xi; }
        double xn[3] = {0.0, 0.0, 0.0}, dn = 0.0;
        if (i + 1 < cnt) seg_load(S3, D, g, NV, nlo, iv, y, t, xi, xn, dn);
        const double e = d - (w[0] * x[0] + w[1] * x[1] + w[2] * x[2]);
        out[i] = (float)(e * e);
        if (RLS) {
            const double p0 = P[0] * x[0] + P[1] * x[1] + P[2] * x[2];
            const double p1 = P[1] * x[0] + P[3] * x[1] + P[4] * x[2];
            const double p2 = P[2] * x[0] + P[4] * x[1] + P[5] * x[2];
            const double inv = reciprocal(1.0 + x[0] * p0 + x[1] * p1 + x[2] * p2);
            const double k0 = p0 * inv, k1 = p1 * inv, k2 = p2 * inv;
            w[0] += k0 * e;
            w[1] += k1 * e;
            w[2] += k2 * e;
            P[0] -= k0 * p0; P[1] -= k0 * p1; P[2] -= k0 * p2;
            P[3] -= k1 * p1; P[4] -= k1 * p2; P[5] -= k2 * p2;
        } else {
            const double ge = g.method == ADAPT_NLMS
                                  ? g.mu * e * reciprocal(g.eps + (x[0] * x[0] + x[1] * x[1] + x[2] * x[2]))
                                  : g.mu * e;
#pragma unroll
            for (int m = 0; m < 3; ++m) w[m] += ge * x[m];
        }
        x[0] = xn[0]; x[1] = xn[1]; x[2] = xn[2];
        d = dn;
    }
}

// Scratch of the regrouped form: segment states, group states, group starts (12, 12 and 9 doubles at most), marks.
struct SegPlan {
    SegGeo g;
    int blocks;   // chains
    size_t segs, groups, starts, todo, bytes;
};

SegPlan seg_plan(int T, int X, int Y, int sec) {
    SegPlan p{};
    const long long per = (long long)T * X, total = per * Y;
    // segments enough to fill the GPU with a thread each (4 blocks per SM), and no shorter than kMinSeg steps
    const long long want = 4LL * kSegThreads * device_sms();
    const long long L = std::min<long long>(per, std::max<long long>(kMinSeg, (total + want - 1) / want));
    p.g = SegGeo{T, X, Y, sec, (int)L, (int)((per + L - 1) / L), 0, 0, 0.0, 0.0, 0.0};
    p.g.ngroup = (p.g.nseg + kSegS - 1) / kSegS;
    p.blocks = (Y + sec - 1) / sec;
    const size_t ngr = (size_t)Y * p.g.ngroup;
    p.segs = 0;
    p.groups = p.segs + (size_t)Y * p.g.nseg * 12 * sizeof(double);
    p.starts = p.groups + ngr * 12 * sizeof(double);
    p.todo = p.starts + ngr * 9 * sizeof(double);
    p.bytes = p.todo + (size_t)p.blocks * sizeof(int);
    return p;
}

template <bool RLS>
void regrouped_launch(const float* S3, const float* D, const SegPlan& p, const float* norm, float* W_out, float* err2,
                      unsigned char* scratch, cudaStream_t s) {
    double* segs = reinterpret_cast<double*>(scratch + p.segs);
    double* groups = reinterpret_cast<double*>(scratch + p.groups);
    double* starts = err2 ? reinterpret_cast<double*>(scratch + p.starts) : nullptr;
    int* todo = reinterpret_cast<int*>(scratch + p.todo);
    const dim3 grid(p.g.ngroup, (p.g.Y + kSegY - 1) / kSegY);
    k3_adapt_segments<RLS><<<grid, kSegThreads, 0, s>>>(S3, D, p.g, norm, segs, groups, todo);
    k3_adapt_chain<RLS><<<p.blocks, kChainThreads, 0, s>>>(p.g, groups, starts, W_out, todo);
    if (err2) k3_adapt_errors<RLS><<<grid, kSegThreads, 0, s>>>(S3, D, p.g, norm, segs, starts, err2, todo);
    note_launches(err2 ? 3 : 2);
}

}  // namespace

// The regrouped form wherever its scratch fits (about 6 bytes a voxel against the 12 of the handle's feature planes;
// sections of less than about 40 samples do not) and the chains are long enough: its launches take 78 to 109 us (LMS), 84 to
// 121 (NLMS) and 48 to 94 (RLS) without and with the errors on 12 x 16 x 20 voxels, in which the step-by-step filter, all
// chains side by side, takes 192 steps of 0.36 (LMS), 0.80 and 1.77 us.  RLS only with lambda = 1, where its information
// form is a plain sum.
constexpr long long min_chain(int method) { return method == ADAPT_LMS ? 272 : method == ADAPT_NLMS ? 136 : 64; }

cudaError_t adapt_launch(const float* S3, const float* D, int T, int X, int Y, int method, double mu, double eps,
                         double lambda, double delta, int sections, const Reduce& r, float* W_out, float* err2,
                         void* scratch, size_t scratch_bytes, cudaStream_t s) {
    const float* norm = r.norm;
    const int sec = sections > 0 ? std::min(sections, Y) : Y;
    const int blocks = (Y + sec - 1) / sec;
    SegPlan p = seg_plan(T, X, Y, sec);
    const bool regroup = scratch && p.bytes <= scratch_bytes && (long long)T * X * sec >= min_chain(method) &&
                         (Y + kSegY - 1) / kSegY <= 65535 && (method != ADAPT_RLS || lambda == 1.0);
    const int* todo = nullptr;
    if (regroup) {
        p.g.method = method;
        p.g.mu = mu;
        p.g.eps = eps;
        p.g.delta = delta;
        unsigned char* b = static_cast<unsigned char*>(scratch);
        const cudaError_t e = cudaMemsetAsync(b + p.todo, 0, (size_t)p.blocks * sizeof(int), s);
        if (e != cudaSuccess) return e;
        if (method == ADAPT_RLS) regrouped_launch<true>(S3, D, p, norm, W_out, err2, b, s);
        else regrouped_launch<false>(S3, D, p, norm, W_out, err2, b, s);
        todo = reinterpret_cast<const int*>(b + p.todo);
    }
    k3_adapt<<<blocks, 32, 0, s>>>(S3, D, T, X, Y, method, mu, eps, lambda, delta, sec, norm, W_out, err2, todo,
                                  r.counter);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace sal

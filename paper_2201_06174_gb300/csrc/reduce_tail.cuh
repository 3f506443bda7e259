// The tails of the volume-wide reductions: the last block of a grid to finish reduces every block's partials itself, so
// that a reduction is one launch instead of two: on small volumes a launch and its gap cost more than what it reduces.  A
// whole FP32 call with the template fit on 10 x 9 x 37 voxels, window 8^3: 65.6 -> 55.3 us; a BF16 call on 1 x 462 x 951,
// window 16^3: 583 -> 571 us; on 128^3: 2435 -> 2414 us.  Blocks of kTailThreads threads.
#pragma once

#include <cfloat>

#include "sal_internal.cuh"

namespace sal {
namespace tail {

constexpr int kTailThreads = 256;
// The counters of a handle, one per kernel of a call.  Each is zero again when its launch ends, unless calls overlapped on the
// handle (which it does not allow).  What these leave is cleared before it is counted on again: a launch clears the others'
// counters, every call begins with C_MAPS, and each call that uses it has a launch behind it that clears C_MAPS (the adaptive
// filter's own, where no second counter is in use).
enum : int { C_MAPS = 0, C_GRAM = 1, C_COMBINE = 2, C_WEIGHTS = 3 };
enum : int { N_LO = 0, N_INV = 3, N_W = 6, N_LOC = 9, N_INVC = 10 };   // layout of Reduce::norm

__device__ __forceinline__ float flat_inv(float lo, float hi) {
    const float span = hi - lo;
    return (span > 1e-30f * fmaxf(1.f, fabsf(hi))) ? 1.f / span : 0.f;
}

__device__ __forceinline__ void clear_others(unsigned* counters, int mine) {
    if (blockIdx.x == 0 && threadIdx.x < 4 && (int)threadIdx.x != mine) counters[threadIdx.x] = 0u;
}

// True in every thread of the last of the grid's blocks to get here, its view of the other blocks' writes complete; the
// counter is zero again for the next launch.
__device__ __forceinline__ bool last_block(unsigned* counters, int mine) {
    __shared__ int s_last;
    unsigned* counter = counters + mine;
    clear_others(counters, mine);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        s_last = atomicAdd(counter, 1u) == gridDim.x - 1 ? 1 : 0;
        if (s_last) *counter = 0u;
    }
    __syncthreads();
    if (s_last) __threadfence();
    return s_last != 0;
}

// Per-block min/max partials (layout [part][8]: min at c, max at 3 + c) of NM maps -> lo and 1 / (hi - lo) (0 for a flat
// map), by one block.
template <int NM>
__device__ __forceinline__ void minmax(const float* mm_part, int nparts, float* lo, float* inv) {
    __shared__ float s_min[NM][kTailThreads / 32], s_max[NM][kTailThreads / 32];
    float a[NM], b[NM];
#pragma unroll
    for (int m = 0; m < NM; ++m) {
        a[m] = FLT_MAX;
        b[m] = -FLT_MAX;
    }
    for (int i = threadIdx.x; i < nparts; i += kTailThreads)
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            a[m] = fminf(a[m], __ldcg(mm_part + i * 8 + m));
            b[m] = fmaxf(b[m], __ldcg(mm_part + i * 8 + 3 + m));
        }
#pragma unroll
    for (int m = 0; m < NM; ++m) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a[m] = fminf(a[m], __shfl_xor_sync(0xffffffffu, a[m], o));
            b[m] = fmaxf(b[m], __shfl_xor_sync(0xffffffffu, b[m], o));
        }
        if ((threadIdx.x & 31) == 0) {
            s_min[m][threadIdx.x / 32] = a[m];
            s_max[m][threadIdx.x / 32] = b[m];
        }
    }
    __syncthreads();
    if (threadIdx.x < NM) {
        const int m = threadIdx.x;
        float l = s_min[m][0], h = s_max[m][0];
        for (int w = 1; w < kTailThreads / 32; ++w) {
            l = fminf(l, s_min[m][w]);
            h = fmaxf(h, s_max[m][w]);
        }
        lo[m] = l;
        inv[m] = flat_inv(l, h);
    }
}

// The bounds of the three maps from the partials of the block's launch, and equal (W_in null) or given weights, into norm
// (mode 2, the template fit, takes its weights from the Gram sums later).
__device__ __forceinline__ void bounds_and_weights(const float* mm_part, const MapTail& t) {
    minmax<3>(mm_part, gridDim.x, t.norm + N_LO, t.norm + N_INV);
    if (threadIdx.x < 3 && t.mode != 2) {
        const float w = t.mode == 0 ? (float)(1.0 / 3.0) : t.W_in[threadIdx.x];
        t.norm[N_W + threadIdx.x] = w;
        if (t.W_out) t.W_out[threadIdx.x] = w;
    }
}

}  // namespace tail
}  // namespace sal

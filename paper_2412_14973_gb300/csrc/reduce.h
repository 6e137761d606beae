// Reduction helpers shared by the vector kernels and the fused residual step:
// warp / block sums in FP64 and the compensated FP32 per-thread accumulator.
#pragma once

#include "internal.h"

namespace tlr {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Block-wide sums of K values per thread (256 threads); thread k < K returns sum k,
// the others 0.  FP64 adds run at 2 lanes per cycle and SM on this part, so the
// tree is folded through shared memory first (8 values per thread, 32 lanes per
// sum): 12 warp-wide adds per value in all, where a shuffle tree in every warp
// takes 45 (the six line-search products: 4300 -> 1150 cycles per block).
// Every call sums in the same order.
template <int K>
__device__ __forceinline__ double block_sums(const double (&v)[K], double (*sh)[256]) {
    static_assert(K <= 8, "one warp per sum");
    const int t = threadIdx.x, w = t >> 5, l = t & 31;
#pragma unroll
    for (int k = 0; k < K; ++k) sh[k][t] = v[k];
    __syncthreads();
    double r = 0.0;
    if (w < K) {
#pragma unroll
        for (int j = 0; j < 8; ++j) r += sh[w][j * 32 + l];
        r = warp_sum(r);
        if (l == 0) sh[w][0] = r;
    }
    __syncthreads();
    r = t < K ? sh[t][0] : 0.0;
    return r;
}

// True in every thread of the last block of a grid of `blocks` to arrive at *ctr
// (zero before the launch, zero again after it); what the other blocks wrote
// before the call is then visible to it.
__device__ __forceinline__ bool last_block(unsigned* ctr, unsigned blocks) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(ctr, 1u) == blocks - 1;
        if (last) *ctr = 0;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// Per-thread partial sum: FP32 terms accumulated with Knuth's two-sum
// compensation (error-free transformation), so a thread's partial is as good
// as an FP64 sum of its FP32 terms while costing FP32 adds only; partials are
// then combined in FP64.  Elementwise FP64 multiply-adds would cost far more on
// this part than the memory traffic they sit on.
struct Acc {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float t = s + x;
        const float z = t - s;
        c += (s - (t - z)) + (x - z);
        s = t;
    }
    __device__ __forceinline__ double val() const { return (double)s + (double)c; }
};

// The same with the compensation compensated in turn: the sum's error is of the order
// of 2^-70 of the terms' magnitudes (FP64 adds: 2^-53), for 13 FP32 adds a term.
struct Acc2 {
    float s = 0.f, c = 0.f, e = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float t = s + x;
        const float z = t - s;
        const float d = (s - (t - z)) + (x - z);
        s = t;
        const float t2 = c + d;
        const float z2 = t2 - c;
        e += (c - (t2 - z2)) + (d - z2);
        c = t2;
    }
    __device__ __forceinline__ double val() const { return (double)s + ((double)c + (double)e); }
};

}  // namespace tlr

// Dot products: accumulators of a thread, and the two-stage sum over a grid of
// 256-thread blocks.
//
// FP64 instructions are slow on this part: a warp's FP64 add or conversion takes
// about 64 clocks of its quarter of the SM however many lanes take part, so a
// chain of them at the end of a short kernel is a large part of it.  Therefore
//   - FP32 dots stay float-float pairs up to the block's sum; one warp converts
//     the pairs of all warps and both sums at once;
//   - two sums share the lanes of one shuffle tree (lower and upper half warp)
//     and, in the sums over warps, two lanes of one chain;
//   - warps that hold no block partial take no part.
// The additions and their order are unchanged by this: a warp's xor tree
// (16, 8, 4, 2, 1), the eight warps one after another, thread t the blocks t,
// t + 256, ... one after another, the tree again, the warps one after another.
#pragma once
#include "internal.cuh"

namespace stk {

// Float-float sum over a warp, before its conversion (see warp_sum_ff).
__device__ __forceinline__ float2 warp_ff(float hi, float lo) {
    for (int o = 16; o > 0; o >>= 1) {
        const float oh = __shfl_xor_sync(0xffffffffu, hi, o), ol = __shfl_xor_sync(0xffffffffu, lo, o);
        float s, e;
        two_sum(hi, oh, s, e);
        e += lo + ol;
        hi = s + e;
        lo = e - (hi - s);
    }
    return make_float2(hi, lo);
}

template <class T> struct Acc;
template <> struct Acc<double> {
    double s = 0.0;
    __device__ void add(double a, double b) { s = fma(a, b, s); }
    __device__ double warp() { return warp_sum(s); }
};
// FP32 vectors: products and sums kept as float-float pairs (TwoProd via FMA,
// TwoSum) so the partial is accurate to ~2^-44 relative without FP64 math.
template <> struct Acc<float> {
    float hi = 0.f, lo = 0.f;
    __device__ void add(float a, float b) {
        float p = a * b;
        float e = fmaf(a, b, -p);
        float s, t;
        two_sum(hi, p, s, t);
        lo += t + e;
        hi = s;
    }
    __device__ double warp() { return warp_sum_ff(hi, lo); }
};

// Warp sums of one value (lane 0) or of two (lane 0: a, lane 16: b).
__device__ __forceinline__ double warp_sums(const double (&v)[1]) { return warp_sum(v[0]); }
__device__ __forceinline__ double warp_sums(const double (&v)[2]) {
    const bool up = (threadIdx.x & 16) != 0;
    const double give = up ? v[0] : v[1], keep = up ? v[1] : v[0];
    double s = keep + __shfl_xor_sync(0xffffffffu, give, 16);
    for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// Shared scratch of a 256-thread block's sums of Q quantities.
template <int Q> struct BlockSumSmem {
    double red[8 * Q];           // by warp, then quantity
    float2 ff[8 * Q];
    bool last;
};

// The block's sums of its first 256 threads' accumulators into partial[Q blockIdx.x + q];
// the last block to finish adds up all blocks and calls fin(totals) in one
// thread.  Every thread of the block calls it, once per kernel.
template <class T, int Q, class Fin>
__device__ __forceinline__ void block_sums(const Acc<T> (&acc)[Q], double* partial, unsigned* counter, int nblocks, Fin fin) {
    __shared__ BlockSumSmem<Q> sm;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    if (w >= 8) {
    } else if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const float2 v = warp_ff(acc[q].hi, acc[q].lo);
            if (lane == 0) sm.ff[w * Q + q] = v;
        }
    } else {
        double v[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) v[q] = acc[q].s;
        const double s = warp_sums(v);
        if (lane == 0) sm.red[w * Q] = s;
        if (Q == 2 && lane == 16) sm.red[w * Q + 1] = s;
    }
    __syncthreads();
    if (w == 0) {
        if constexpr (sizeof(T) == 4) {
            if (lane < 8 * Q) sm.red[lane] = (double)sm.ff[lane].x + (double)sm.ff[lane].y;
            __syncwarp();
        }
        if (lane < Q) {
            double s = sm.red[lane];
            for (int k = 1; k < 8; ++k) s += sm.red[k * Q + lane];
            partial[Q * blockIdx.x + lane] = s;
            __threadfence();
        }
        __syncwarp();
        if (lane == 0) sm.last = atomicAdd(counter, 1u) == (unsigned)nblocks - 1u;
    }
    __syncthreads();
    if (!sm.last) return;
    __threadfence();
    if (w < 8 && 32 * w < nblocks) {
        double v[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) v[q] = t < nblocks ? ((volatile double*)partial)[Q * t + q] : 0.0;
        for (int b = t + 256; b < nblocks; b += 256)
#pragma unroll
            for (int q = 0; q < Q; ++q) v[q] += ((volatile double*)partial)[Q * b + q];
        __syncwarp();
        const double s = warp_sums(v);
        if (lane == 0) sm.red[w * Q] = s;
        if (Q == 2 && lane == 16) sm.red[w * Q + 1] = s;
    }
    __syncthreads();
    if (w == 0) {
        double s = 0.0;
        if (lane < Q) {
            s = sm.red[lane];
            for (int k = 1; 32 * k < nblocks && k < 8; ++k) s += sm.red[k * Q + lane];
        }
        double tot[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) tot[q] = __shfl_sync(0xffffffffu, s, q);
        if (lane == 0) {
            fin(tot);
            *counter = 0u;
        }
    }
}

}  // namespace stk

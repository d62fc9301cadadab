// Pieces of the cooperative CG kernels (cgloop.cu, schwarz_loop.cu).
#pragma once
#include <algorithm>
#include <atomic>
#include "internal.cuh"
#include "ctx.cuh"
#include "grid_gather.cuh"
#include "reduce.cuh"

namespace stk {

// a b + c d with the first product fused: written out so that the kernel rounds
// as the separate applies do.
template <class T> __device__ __forceinline__ T fma_first(T a, T b, T c, T d) { return fma(a, b, c * d); }

// Warp sums of a CTA on their way to an exchange: FP32 kernels leave float-float
// pairs, which one warp converts.
template <class T, int NW> struct WarpSums {
    double rows[2 * NW];
    float2 ff[sizeof(T) == 4 ? 2 * NW : 1];
    __device__ void put(int i, const Acc<T>& acc, bool any = true) {
        const int lane = threadIdx.x & 31;
        if constexpr (sizeof(T) == 4) {
            const float2 v = any ? warp_ff(acc.hi, acc.lo) : make_float2(0.f, 0.f);
            if (lane == 0) ff[i] = v;
        } else {
            const double v = any ? warp_sum(acc.s) : 0.0;
            if (lane == 0) rows[i] = v;
        }
    }
    // two sums at once
    __device__ void put2(int i, const Acc<T>& a, int j, const Acc<T>& b, bool any = true) {
        if constexpr (sizeof(T) == 4) {
            put(i, a, any);
            put(j, b, any);
        } else {
            const int lane = threadIdx.x & 31;
            const double two[2] = {a.s, b.s};
            const double v = any ? warp_sums(two) : 0.0;
            if (lane == 0) rows[i] = v;
            if (lane == 16) rows[j] = v;
        }
    }
    // rows[0 .. n) as doubles (n <= 32); the CTA has passed a barrier since put; warp 0
    __device__ void convert(int n) {
        if constexpr (sizeof(T) == 4) {
            const int lane = threadIdx.x & 31;
            if (lane < n) rows[lane] = (double)ff[lane].x + (double)ff[lane].y;
            __syncwarp();
        }
    }
    // the block sums of k_cg_init / k_cg_update: r.z of warps 0, 1, ... one after
    // another in rows[0], r.r likewise in rows[1] (both arrays were put at 0 and NW)
    __device__ void block2() {
        __syncthreads();
        if (threadIdx.x < 32) {
            convert(2 * NW);
            double s = 0.0;
            if (threadIdx.x < 2)
                for (int q = 0; q < NW; ++q) s += rows[threadIdx.x * NW + q];
            __syncwarp();
            if (threadIdx.x < 2) rows[threadIdx.x] = s;
        }
    }
};

// The place in the (ascending) tile list of a tile id, -1 if it is not there.
__device__ __forceinline__ int tile_place(const int* __restrict__ tiles, int n, int id) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (tiles[mid] < id) lo = mid + 1;
        else hi = mid;
    }
    return lo < n && tiles[lo] == id ? lo : -1;
}

// z of a slot at the edge of a CTA, for its neighbours: words tagged with the
// iteration (FP64: low and high half).  No fence or barrier orders them: a
// reader polls the words themselves, and their writer overwrites them only
// after an exchange that the reader enters after reading.
template <class T> struct ZWords;
template <> struct ZWords<float> {
    static constexpr int N = 1;
    static __device__ __forceinline__ void put(unsigned long long* p, unsigned tag, float z) { post_word(p, tag, __float_as_uint(z)); }
    static __device__ __forceinline__ float get(const unsigned long long (&v)[1]) { return __uint_as_float((unsigned)v[0]); }
};
template <> struct ZWords<double> {
    static constexpr int N = 2;
    static __device__ __forceinline__ void put(unsigned long long* p, unsigned tag, double z) {
        const unsigned long long u = __double_as_longlong(z);
        post_word(p, tag, (unsigned)u);
        post_word(p + 1, tag, (unsigned)(u >> 32));
    }
    static __device__ __forceinline__ double get(const unsigned long long (&v)[2]) { return from_words(v[0], v[1]); }
};

// A loop's words, allocated on first use; false (and no error left) if there is no
// room for them.
static bool loop_words(Ctx* c, unsigned long long*& words, size_t bytes) {
    if (words) return true;
    if (cudaMalloc((void**)&words, bytes) != cudaSuccess) {
        words = nullptr;
        cudaGetLastError();
        return false;
    }
    c->allocs.push_back(words);
    return true;
}
// Whether a cooperative launch went through.  The device may refuse it although
// the kernel fits on all of it: a process limited to a part of the SMs, a share of
// the device held by others.  The separate kernels then take the solve (and report
// an error that has another cause).
static bool loop_launched(cudaError_t e) {
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess;
}

// CTAs of a kernel that fit on the device at once (cached per device).
template <class K>
static int fit(K k, int threads, size_t smem, std::atomic<int>* cache) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 16) return 0;
    int n = cache[dev].load(std::memory_order_relaxed);
    if (n == 0) {
        int sms = 0, per = 0, coop = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
        // (the most there is: a kernel may be launched with several sizes)
        if (smem > 48 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, threads, smem);
        n = coop ? sms * per : -1;
        cache[dev].store(n ? n : -1, std::memory_order_relaxed);
    }
    return std::max(n, 0);
}

}  // namespace stk

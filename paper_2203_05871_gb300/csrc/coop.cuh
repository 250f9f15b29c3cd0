// Device helpers shared by the cooperative per-op kernels (QR, Jacobi SVD):
// a bounded barrier among the CTAs that work on one op, and warp reductions.
#pragma once

#include <cuda_runtime.h>

#include "internal.h"

namespace mpdo {

// per-op sync words: [0] barrier arrivals, [1] abort flag, [2, 8) Jacobi pair counters,
// [8 + s] rotations and [8 + kMaxSweepsCap + s] largest off-orthogonality in Jacobi
// sweep s, then one version per Jacobi row block (at most 4 kMaxChi blocks)
constexpr int kSyncWords = 8 + 2 * kMaxSweepsCap + 4 * kMaxChi;

__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Barrier of the G CTAs working on one op; returns false if it gave up.
__device__ __forceinline__ bool op_barrier(unsigned* sw, int G, unsigned& gen, unsigned long long timeout_ns) {
    __shared__ int s_ok;
    __threadfence();
    __syncthreads();
    if (G == 1) return true;
    ++gen;
    if (threadIdx.x == 0) {
        atomicAdd(&sw[0], 1u);
        const unsigned target = gen * (unsigned)G;
        const unsigned long long t0 = globaltimer_ns();
        int ok = 1;
        while (ld_acquire(&sw[0]) < target) {
            if (ld_acquire(&sw[1]) != 0u) {
                ok = 0;
                break;
            }
            if (globaltimer_ns() - t0 > timeout_ns) {
                atomicExch(&sw[1], 1u);
                ok = 0;
                break;
            }
            __nanosleep(64);
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The kk-th largest of v[0..c), c <= NMAX (non-negative), by bisection on the
// bit pattern (non-negative doubles order like their bits).  Called by every
// thread of a CTA of NT threads; every thread returns the same value.
template <int NT, int NMAX>
__device__ double kth_largest(const double* v, int c, int kk) {
    constexpr int kPer = (NMAX + NT - 1) / NT;
    __shared__ int s_cnt[NT / 32];
    unsigned long long key[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int j = threadIdx.x + i * NT;
        key[i] = j < c ? (unsigned long long)__double_as_longlong(fmax(__ldcg(v + j), 0.0)) : 0ull;
    }
    unsigned long long x = 0ull;
    for (int bit = 62; bit >= 0; --bit) {
        const unsigned long long cand = x | (1ull << bit);
        int n = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) n += key[i] >= cand;
        n = __reduce_add_sync(0xffffffffu, n);
        if ((threadIdx.x & 31) == 0) s_cnt[threadIdx.x >> 5] = n;
        __syncthreads();
        int tot = 0;
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) tot += s_cnt[w];
        __syncthreads();
        if (tot >= kk) x = cand;
    }
    return __longlong_as_double((long long)x);
}

}  // namespace mpdo


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
constexpr int kSwQueue = 2;   // words 2, 3: the Jacobi block-pair counters of alternate sweeps
constexpr int kSwVer = 8 + 2 * kMaxSweepsCap;   // the versions

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

__device__ __forceinline__ void st_release(unsigned* p, unsigned v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Wait (thread 0) until row blocks P and Q (those < nb) have left round R - 1,
// i.e. their versions reached R; bounded by timeout_ns, after which the op's
// abort flag is raised.  Returns 0 if it gave up.
__device__ inline int wait_blocks(const unsigned* ver, int P, int Q, int nb, unsigned R, unsigned* abort_flag,
                           unsigned long long timeout_ns) {
    const unsigned long long t0 = globaltimer_ns();
    for (;;) {
        const bool okP = P >= nb || ld_acquire(ver + P) >= R;
        const bool okQ = Q >= nb || ld_acquire(ver + Q) >= R;
        if (okP && okQ) return 1;
        if (ld_acquire(abort_flag) != 0u) return 0;
        if (globaltimer_ns() - t0 > timeout_ns) {
            atomicExch(abort_flag, 1u);
            return 0;
        }
        __nanosleep(32);
    }
}

// player in place x of a circle tournament of cp players at a step
__device__ __forceinline__ int tour_player(int x, int step, int cp) {
    return x == 0 ? 0 : 1 + ((x - 1 + step) % (cp - 1));
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

// The same for c float values val(j) (non-negative): 31 counting rounds.
template <int NT, int NMAX, class F>
__device__ float kth_largest_f(F val, int c, int kk) {
    constexpr int kPer = (NMAX + NT - 1) / NT;
    __shared__ int s_cnt[2][NT / 32];
    unsigned key[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int j = threadIdx.x + i * NT;
        key[i] = j < c ? __float_as_uint(fmaxf(val(j), 0.0f)) : 0u;
    }
    unsigned x = 0u;
    for (int bit = 30; bit >= 0; --bit) {
        const unsigned cand = x | (1u << bit);
        int n = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) n += key[i] >= cand;
        n = __reduce_add_sync(0xffffffffu, n);
        if ((threadIdx.x & 31) == 0) s_cnt[bit & 1][threadIdx.x >> 5] = n;
        __syncthreads();
        int tot = 0;
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) tot += s_cnt[bit & 1][w];
        if (tot >= kk) x = cand;
    }
    __syncthreads();
    return __uint_as_float(x);
}

// Squared norm under which two rows need not be made orthogonal to one another, whatever
// the margin below chi_max: the rows under it hold less than a thousandth of the weight
// that the cutoff discards, and rotations among them leave that sum as it is, so the
// rank and the kept rows do not depend on them (0: every row may be needed).  total is
// the sum of all squared norms.  Bonds with a handful of kept rows out of tens are where
// it counts: their tails, down to rounding level, kept the FP32 pass at 8 to 15 sweeps
// and left one op in five of a grid's evolution to the FP64 pass.
__device__ __forceinline__ double cutoff_floor(const OpDesc& d, double total) {
    return d.full_svd || d.forced_k > 0 ? 0.0 : 1e-3 * fmin(fmax(d.cutoff, 0.0), 1.0) * total / d.c;
}

}  // namespace mpdo

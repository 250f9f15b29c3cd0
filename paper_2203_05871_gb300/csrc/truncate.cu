// Truncation of one bond after the Jacobi SVD (App. B).
//
// s_j = |w_j| (row norms after Jacobi), sorted descending with ties kept in
// row order.  k_cut = smallest k >= 1 whose discarded weight
// sum_{i>=k} s_i^2 is <= cutoff * sum_i s_i^2 (the tail is summed from the
// smallest value up); k = min(chi_max, k_cut).  Writes lambda_p = s[:k],
// Yk[j] = v_j^T (rows of W normalised, or rows of Z), the new site p+1
// B'[j][s2][r] = Yk[j][s2*cr + r] and the new bond dimension.  A forced rank
// (replay of a recorded run) replaces k_cut, still capped by chi_max and c.
// When the adjoint records a tape, all c sorted singular values and
// normalised rows are written as well.
#include <cooperative_groups.h>
#include <mpdo.h>

#include "internal.h"

namespace mpdo {

namespace {

constexpr int TT = 512;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// A cluster of 8 CTAs per op: the rows' norms, the normalised rows and the new site
// are an eighth each (one CTA read and wrote 16 MB through one SM at chi = 256,
// 1.3 ms); every CTA ranks all norms and sums the tails itself.
constexpr int TC = 8;
__global__ void __cluster_dims__(TC, 1, 1) __launch_bounds__(TT, 1) truncate_kernel(const OpDesc* descs, int chi_cap) {
    namespace cg = cooperative_groups;
    const cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const OpDesc& d = descs[blockIdx.x / TC];
    const int c = d.c, L = d.L, ld = 4 * chi_cap;
    extern __shared__ double smem[];
    double* s = smem;                        // [c] norms
    double* tail = smem + ld;                // [c + 1] sum_{i >= k} s_perm(i)^2; first the sorted norms
    int* perm = reinterpret_cast<int*>(smem + 2 * ld + 1);
    __shared__ int s_k, s_bad;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        s_bad = 0;
        s_k = c;
    }
    cluster.sync();   // every CTA runs before its shared memory is written
    for (int j = rank + TC * warp; j < c; j += TC * (TT / 32)) {
        const double* w = d.W + (size_t)j * ld;
        double a = 0.0;
        for (int i = lane; i < L; i += 32) {
            const double x = w[i];
            a = fma(x, x, a);
        }
        a = warp_sum(a);
        const double v = sqrt(a);
        if (lane < TC) cluster.map_shared_rank(s, lane)[j] = v;
    }
    cluster.sync();
    for (int j = threadIdx.x; j < c; j += TT)
        if (!isfinite(s[j])) s_bad = 1;
    __syncthreads();
    const int bad = s_bad;
    for (int j = threadIdx.x; j < c; j += TT) {
        if (bad) {
            perm[j] = j;
            continue;
        }
        // by their bit patterns (norms are >= 0): c^2 FP64 comparisons would take the FP64
        // pipe 0.5 ms at chi = 256
        const long long sj = __double_as_longlong(s[j]);
        int r = 0;
#pragma unroll 8
        for (int i = 0; i < c; ++i) {
            const long long si = __double_as_longlong(s[i]);
            r += si > sj || (si == sj && i < j);
        }
        perm[r] = j;
        tail[r] = s[j];
    }
    __syncthreads();
    if (threadIdx.x == 0 && !bad) {
        // the tails, accumulated from the smallest value up
        double t = 0.0;
        tail[c] = 0.0;
        for (int i = c - 1; i >= 0; --i) {
            const double v = tail[i];
            t = fma(v, v, t);
            tail[i] = t;
        }
    }
    __syncthreads();
    // the smallest k >= 1 whose tail is within the cutoff (the tails do not increase with k)
    if (!bad)
        for (int k = 1 + threadIdx.x; k < c; k += TT)
            if (tail[k] <= d.cutoff * tail[0]) atomicMin(&s_k, k);
    __syncthreads();
    int k = s_k;
    if (k > d.chi_max) k = d.chi_max;
    if (d.forced_k > 0) k = d.forced_k < d.chi_max ? d.forced_k : d.chi_max;
    if (k > c) k = c;
    if (k < 1 || bad) k = 1;
    if (rank == 0 && threadIdx.x == 0) {
        if (bad) atomicOr(d.status, (int)MPDO_ST_NONFINITE);
        *d.k_out = k;
        if (d.rank_log) *d.rank_log = k;
        const double disc = !bad && tail[0] > 0.0 ? tail[k] / tail[0] : 0.0;
        atomicMax((unsigned long long*)d.max_disc, (unsigned long long)__double_as_longlong(disc));
    }
    const int t0 = rank * TT + threadIdx.x, w0 = rank + TC * warp;
    for (int j = t0; j < k; j += TC * TT) d.lam_out[j] = bad ? 0.0 : s[perm[j]];
    const double* rows = d.transposed ? d.Z : d.W;   // s_j v_j^T, or of unit norm
    if (d.tape_V) {
        // every sorted right singular vector (zero rows stay zero) for the adjoint
        for (int j = t0; j < c; j += TC * TT) d.tape_s[j] = bad ? 0.0 : s[perm[j]];
        for (int j = w0; j < c; j += TC * (TT / 32)) {
            const int src = perm[j];
            const double sv = s[src];
            const double inv = (sv > 0.0 && !bad) ? (d.transposed ? 1.0 : 1.0 / sv) : 0.0;
            const double* wr = rows + (size_t)src * ld;
            double* v = d.tape_V + (size_t)j * d.n;
            for (int i = lane; i < d.n; i += 32) v[i] = wr[i] * inv;
        }
    }
    const int cr = d.cr;
    for (int j = w0; j < k; j += TC * (TT / 32)) {
        const int src = perm[j];
        double* y = d.Yk + (size_t)j * ld;
        const size_t bnew = (size_t)j * 4 * chi_cap;   // row j of the new site p+1
        const double* wr = rows + (size_t)src * ld;
        const double sv = s[src];
        const double inv = (sv > 0.0 && !bad) ? (d.transposed ? 1.0 : 1.0 / sv) : 0.0;
        for (int s2 = 0; s2 < 4; ++s2)
            for (int r = lane; r < cr; r += 32) {
                const int i = s2 * cr + r;
                const double v = wr[i] * inv;
                y[i] = v;
                site_st(d.B, bnew + (size_t)s2 * chi_cap + r, v, d.site_f32);
            }
    }
}

static_assert((2 * 4 * kMaxChi + 1) * 8 + 4 * kMaxChi * 4 <= 48 * 1024, "within the default shared memory");

}  // namespace

cudaError_t launch_truncate(const OpDesc* d_desc, int nops, int chi_cap, cudaStream_t st) {
    if (nops <= 0) return cudaSuccess;
    const size_t ld = 4 * (size_t)chi_cap;
    truncate_kernel<<<TC * nops, TT, (2 * ld + 1) * sizeof(double) + ld * sizeof(int), st>>>(d_desc, chi_cap);
    return cudaGetLastError();
}

}  // namespace mpdo

// Bond gauges that the slice products do not resolve.
//
// Tensors are defined up to an invertible matrix on every bond: A D and D^-1 B are the
// same state.  A product formed from slices (oz_gemm.cu) has an error of 2^-54 of
// max|A row| max|B column|, where FP64 dot products have 2^-53 of sum_k |A_ik B_kj|: a
// diagonal D of 10^+-4 on one bond costs a step eight digits that dot products keep
// (2e-8 against 5e-15 in <X>, <Y>, <Z> of six qubits), and the SVD's stages in FP32 see
// rows and columns that far apart.  So before tensors of mpdo_set_state, which can be in any
// gauge, are first worked on, every bond is looked at:
//   loss = max_k log2|A_k| + max_k log2|B_k| - max_k (log2|A_k| + log2|B_k|)
// with |A_k|, |B_k| the largest entries of column k of the left and row k of the right
// site.  Bonds that lose more than kGaugeBits are flagged until their next op, whose SVD
// gives them a gauge of its own; ops on or next to a flagged bond and the entropies of
// such a state take the FP64 dot products, QR and Jacobi pass of contract.cu, gemm.cu,
// qr.cu and jacobi.cu.  With four bits the operands' rounding (2^-56 each) comes to
// 2^-51, what a dot product of 16 terms has.  States of the solver itself, saved and
// loaded again, lose nothing: after an op the right site's rows have unit norm, and the
// leading column of the left site is among its largest (0 bits at every bond of all the
// evolutions, steps and gradients it was measured on).  Mixed contexts, whose products are
// six slices throughout, are not looked at.
//
// One block per bond reads both sites once, exponents only (integer work: GB300 issues
// two FP64 instructions per SM and clock).
#include <mpdo.h>

#include <algorithm>

#include "ctx.h"
#include "internal.h"

namespace mpdo {

namespace {

constexpr int kGaugeBits = 4;
constexpr int NT = 1024;

// biased exponent of element i (0: zero or subnormal)
__device__ __forceinline__ int exponent_at(const void* p, int f32, size_t i) {
    return f32 ? (int)((__float_as_uint(static_cast<const float*>(p)[i]) >> 23) & 0xff)
               : (int)(((unsigned)__double2hiint(static_cast<const double*>(p)[i]) >> 20) & 0x7ff);
}

__global__ void __launch_bounds__(NT) gauge_kernel(const void* sites, int f32, const int* dims, int n, int cap,
                                                   int* loss) {
    const int m = blockIdx.x + 1, b = blockIdx.y;
    const int* dm = dims + (size_t)b * (n + 1);
    const int chi = dm[m], arows = 4 * dm[m - 1], cr = dm[m + 1];
    const size_t elems = (size_t)cap * 4 * cap, es = f32 ? sizeof(float) : sizeof(double);
    const void* A = static_cast<const char*>(sites) + ((size_t)b * n + m - 1) * elems * es;
    const void* B = static_cast<const char*>(sites) + ((size_t)b * n + m) * elems * es;
    __shared__ int ea[kMaxChi], eb[kMaxChi], top[3];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int k = threadIdx.x; k < chi; k += NT) ea[k] = 0;
    if (threadIdx.x < 3) top[threadIdx.x] = 0;
    __syncthreads();
    for (int k = lane; k < chi; k += 32) {
        int e = 0;
#pragma unroll 8
        for (int r = warp; r < arows; r += NT / 32) e = max(e, exponent_at(A, f32, (size_t)r * cap + k));
        atomicMax(&ea[k], e);
    }
    for (int k = warp; k < chi; k += NT / 32) {
        int e = 0;
        for (int s = 0; s < 4; ++s)
#pragma unroll 4
            for (int r = lane; r < cr; r += 32) e = max(e, exponent_at(B, f32, ((size_t)k * 4 + s) * cap + r));
        e = __reduce_max_sync(0xffffffffu, e);
        if (lane == 0) eb[k] = e;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < chi; k += NT) {
        atomicMax(&top[0], ea[k]);
        atomicMax(&top[1], eb[k]);
        if (ea[k] > 0 && eb[k] > 0) atomicMax(&top[2], ea[k] + eb[k]);
    }
    __syncthreads();
    if (threadIdx.x == 0) loss[(size_t)b * (n + 1) + m] = top[2] > 0 ? top[0] + top[1] - top[2] : 0;
}

}  // namespace

cudaError_t launch_gauge(const void* sites, int sites_f32, const int* dims, int n, int B, int chi_cap, int* loss,
                         cudaStream_t st) {
    gauge_kernel<<<dim3(n - 1, B), NT, 0, st>>>(sites, sites_f32, dims, n, chi_cap, loss);
    return cudaGetLastError();
}

int refresh_gauge(mpdo_ctx* c) {
    if (!c->precond || c->mixed || std::count(c->loaded.begin(), c->loaded.end(), 0) == c->B) return MPDO_OK;
    const int N = c->N;
    int* d_loss = reinterpret_cast<int*>(c->d_out);   // [B][N * N] doubles, free between calls
    CU(launch_gauge(c->d_sites, sites_f32(c), c->d_dims, N, c->B, c->cap, d_loss, c->st));
    std::vector<int> loss((size_t)c->B * (N + 1), 0);
    CU(cudaMemcpyAsync(loss.data(), d_loss, sizeof(int) * loss.size(), cudaMemcpyDeviceToHost, c->st));
    CU(cudaStreamSynchronize(c->st));
    for (int b = 0; b < c->B; ++b) {
        if (!c->loaded[b]) continue;
        for (int m = 1; m < N; ++m) {
            const size_t i = (size_t)b * (N + 1) + m;
            c->wide[i] = loss[i] > kGaugeBits;
        }
        c->loaded[b] = 0;
    }
    return MPDO_OK;
}

bool wide_instance(const mpdo_ctx* c, int b) {
    const auto w = c->wide.begin() + (size_t)b * (c->N + 1);
    return std::any_of(w, w + c->N + 1, [](unsigned char x) { return x != 0; });
}

bool wide_any(const mpdo_ctx* c) {
    return std::any_of(c->wide.begin(), c->wide.end(), [](unsigned char x) { return x != 0; });
}

}  // namespace mpdo

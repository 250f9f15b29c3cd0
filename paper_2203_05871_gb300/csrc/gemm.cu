// Batched small dense FP64 GEMMs: the adjoint's products that slices would not resolve
// (grad.cu), the Gram sweeps of contexts and states without the slice products (global.cu).
//
//   C = alpha * op(A) op(B) + beta * D  (- I if sub_identity)
// with A (M x K, or K x M when a_trans) and B (K x N, or N x K when b_trans)
// row-major, stored as
// float or double (converted on load), accumulated and
// written as double.  One launch serves a list of problems of different
// sizes (grid.z = problem); CTAs outside a problem's tiles return at once.
// 64 x 64 tiles (32 or 16 where few), k-step 16, 256 threads.
// A symmetric product (sym: X' = B^T (X B)) computes the tiles on and above the
// diagonal only and writes each strictly upper tile to both triangles.
#include "internal.h"

namespace mpdo {

namespace {

constexpr int GK = 16;

__device__ __forceinline__ double load(const void* p, int is_f32, size_t i) {
    return is_f32 ? (double)static_cast<const float*>(p)[i] : static_cast<const double*>(p)[i];
}

// GT x GT tiles, R x R outputs per thread; the next k tile is on its way into
// registers while this one is used.  Every output is the same sum in the same order
// whatever GT is.
template <int GT>
__global__ void __launch_bounds__(256) gemm_kernel(const GemmDesc* descs) {
    constexpr int R = GT / 16;
    static_assert(GT * GK == 256 * R, "R elements of each operand per thread");
    const GemmDesc& g = descs[blockIdx.z];
    const int i0 = blockIdx.y * GT, j0 = blockIdx.x * GT;
    if (i0 >= g.M || j0 >= g.N) return;
    if (g.sym && i0 > j0) return;   // the mirror of a tile above the diagonal
    __shared__ double As[GK][GT + 1];
    __shared__ double Bs[GK][GT + 1];
    const int t = threadIdx.x, ty = t >> 4, tx = t & 15;
    double acc[R][R], pa[R], pb[R];
#pragma unroll
    for (int u = 0; u < R; ++u)
#pragma unroll
        for (int v = 0; v < R; ++v) acc[u][v] = 0.0;
    // element e of a tile's operand: along the stored rows
    auto at_a = [&](int e, int& kk, int& ii) {   // A stored M x K, or K x M when a_trans
        kk = g.a_trans ? e / GT : e % GK;
        ii = g.a_trans ? e % GT : e / GK;
    };
    auto at_b = [&](int e, int& kk, int& jj) {   // B stored K x N, or N x K when b_trans
        kk = g.b_trans ? e % GK : e / GT;
        jj = g.b_trans ? e / GK : e % GT;
    };
    auto fetch = [&](int k0) {
#pragma unroll
        for (int u = 0; u < R; ++u) {
            int kk, x;
            at_a(t + 256 * u, kk, x);
            const int gi = i0 + x, ka = k0 + kk;
            pa[u] = gi < g.M && ka < g.K
                        ? load(g.A, g.a_f32, g.a_trans ? (size_t)ka * g.lda + gi : (size_t)gi * g.lda + ka)
                        : 0.0;
            at_b(t + 256 * u, kk, x);
            const int gj = j0 + x, kb = k0 + kk;
            pb[u] = gj < g.N && kb < g.K
                        ? load(g.B, g.b_f32, g.b_trans ? (size_t)gj * g.ldb + kb : (size_t)kb * g.ldb + gj)
                        : 0.0;
        }
    };
    fetch(0);
    for (int k0 = 0; k0 < g.K; k0 += GK) {
#pragma unroll
        for (int u = 0; u < R; ++u) {
            int kk, x;
            at_a(t + 256 * u, kk, x);
            As[kk][x] = pa[u];
            at_b(t + 256 * u, kk, x);
            Bs[kk][x] = pb[u];
        }
        __syncthreads();
        if (k0 + GK < g.K) fetch(k0 + GK);
#pragma unroll 4
        for (int kk = 0; kk < GK; ++kk) {
            double a[R], b[R];
#pragma unroll
            for (int u = 0; u < R; ++u) {
                a[u] = As[kk][ty * R + u];
                b[u] = Bs[kk][tx * R + u];
            }
#pragma unroll
            for (int u = 0; u < R; ++u)
#pragma unroll
                for (int v = 0; v < R; ++v) acc[u][v] = fma(a[u], b[v], acc[u][v]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int gi = i0 + ty * R + u;
        if (gi >= g.M) continue;
#pragma unroll
        for (int v = 0; v < R; ++v) {
            const int gj = j0 + tx * R + v;
            if (gj >= g.N) continue;
            double r = g.alpha * acc[u][v];
            if (g.D) r += g.beta * load(g.D, g.d_f32, (size_t)gi * g.ldd + gj);
            if (g.sub_identity && gi == gj) r -= 1.0;
            g.C[(size_t)gi * g.ldc + gj] = r;
            if (g.sym && i0 < j0) g.C[(size_t)gj * g.ldc + gi] = r;
        }
    }
}

template <int GT>
cudaError_t launch_tiles(const GemmDesc* d_desc, int count, int max_m, int max_n, cudaStream_t st) {
    const dim3 grid((max_n + GT - 1) / GT, (max_m + GT - 1) / GT, count);
    gemm_kernel<GT><<<grid, 256, 0, st>>>(d_desc);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_gemm(const GemmDesc* d_desc, int count, int max_m, int max_n, cudaStream_t st) {
    if (count <= 0 || max_m <= 0 || max_n <= 0) return cudaSuccess;
    // The FP64 pipe, two FMAs per SM and clock, bounds every tile: 64 x 64 outputs take
    // it 2048 K clocks, so tiles shrink until the launch fills the chip (the adjoint's
    // products of 128 x 64 x 64 ran on two SMs, 120 us each).
    const long long tiles = (long long)((max_n + 63) / 64) * ((max_m + 63) / 64) * count;
    if (tiles * 4 <= 152) return launch_tiles<16>(d_desc, count, max_m, max_n, st);
    if (tiles <= 152) return launch_tiles<32>(d_desc, count, max_m, max_n, st);
    return launch_tiles<64>(d_desc, count, max_m, max_n, st);
}

}  // namespace mpdo

// FP32 Householder QR of the weighted bond matrices: the orthogonal start of the
// SVD.
//
// The SVD needs the rows of theta~ (m x n, m <= n; theta~^T otherwise) turned by an
// orthogonal matrix that grades them (qr.cu says why: Jacobi then converges in a
// third of the sweeps).  Any such matrix will do as long as it is orthogonal to
// FP64 accuracy when it is applied, so it is found in FP32: A_1, the m columns of
// largest norm in that order with the other n - m folded onto them (from the last
// on; alone, the rows of theta~ of largest weight can leave out whole directions:
// a third more Jacobi sweeps on some), is factored A_1 = Q R by blocked Householder
// reflections, Q^T is
// accumulated explicitly in U32, and the tensor-core products (api.cu) then
// orthogonalise it (E = U U^T - I, one step) and form W0 = Q^T theta~ in FP64
// accuracy.  (theta~^T is turned as it is, Z following along: R alone would need
// the factorisation itself to be accurate to FP64.)  W0's rows are graded like those of R down to FP32 rounding of the
// largest; below that they are resolved by the FP32 Jacobi pass that follows,
// which sees them as they are.
// Sorting the columns once by norm replaces pivoting at every column: on the
// bond matrices of evolved and of random states the Jacobi pass needs 6 to 7
// sweeps either way (a numpy model of both; 20 and more without the QR).  No
// column then waits for the one before it, and the FP64 column QR of a
// 1024 x 1024 matrix (26 us per column: its FP64 work alone is 10 ms per chunk
// of nine, at two FMAs per SM and clock) becomes 64 panels.
//
// One panel is 16 columns.  Every CTA of the op factors it redundantly in
// registers (a thread holds up to four rows of 16), so a panel costs one barrier:
//   step j: d_k = sum_i x_i P_ik over the rows i >= j for all 16 columns at once
//     (x = column j; k < j: the reflector k), one block reduction; then
//     |x|^2 = d_j, v = x - alpha e_j, v.P_k = d_k - alpha P_jk, and the columns
//     k > j are reflected;
//   T from the v.v_k collected on the way, Q^T_panel = I - V T^T V^T;
//   the columns of A_1 still to come and all columns of Q^T are shared among the
//     op's CTAs in tiles of 32: W = V^T A, W <- T^T W, A <- A - V W on the tensor
//     cores (mma.sync tf32, operands split in two as in jacobi32.cu).
// The op's CTAs meet in a bounded barrier (cooperative launch).
#include <mpdo.h>

#include "coop.cuh"
#include "internal.h"

namespace mpdo {

namespace {

constexpr int NT = 512;
constexpr int NWARP = NT / 32;
constexpr int PB = 16;                // columns per panel
constexpr int CT = 32;                // columns per tile of the update
constexpr int kMaxM = 4 * kMaxChi;
constexpr int VS = PB + 4;            // row stride of V in shared memory

struct Smem {
    float V[kMaxM * VS];              // reflectors of the panel, row i - j0
    float red[NWARP * PB * CT];       // partial V^T A of the warps; column norms and order before the panels
    float W[PB * CT], W2[PB * CT];
    float part[2][NWARP][PB], row[2][PB];
    float VV[PB][PB], T[PB][PB], beta[PB];
    double sum[NWARP], scale;
};
static_assert(sizeof(Smem) <= 227 * 1024, "shared memory");
static_assert(2 * kMaxM <= NWARP * PB * CT, "norms and order fit");

// x = hi + lo, both read as tf32 (hi: the leading 11 bits)
__device__ __forceinline__ void split(float x, uint32_t& hi, uint32_t& lo) {
    hi = __float_as_uint(x) & 0xffffe000u;
    lo = __float_as_uint(x - __uint_as_float(hi));
}

__device__ __forceinline__ void mma_tf32(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// Factors the panel of columns j0 .. j0 + 15 (rows j0 .. m - 1 of A): V, the
// inner products of the reflectors and their betas into shared memory.  Thread
// t holds rows t, t + NT, ...: R of them.
template <int R>
__device__ void factor_panel(Smem& S, const float* A, int ld, int m, int j0, int warp, int lane) {
    float p[R][PB];
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int r = threadIdx.x + u * NT;
#pragma unroll
        for (int q = 0; q < PB / 4; ++q) {
            float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (r >= j0 && r < m && j0 + 4 * q < m) v = __ldcg(reinterpret_cast<const float4*>(A + (size_t)r * ld + j0 + 4 * q));
            p[u][4 * q] = v.x;
            p[u][4 * q + 1] = v.y;
            p[u][4 * q + 2] = v.z;
            p[u][4 * q + 3] = v.w;
        }
    }
#pragma unroll
    for (int j = 0; j < PB; ++j) {
        const int jr = j0 + j, buf = j & 1;
        if (jr >= m) {   // past the last row (m is a multiple of 4): no reflector
            if (threadIdx.x == 0) S.beta[j] = 0.0f;
            if (threadIdx.x < PB) S.VV[threadIdx.x][j] = 0.0f;
#pragma unroll
            for (int u = 0; u < R; ++u) p[u][j] = 0.0f;
            continue;
        }
        float x[R], d[PB];
#pragma unroll
        for (int u = 0; u < R; ++u) {
            const int r = threadIdx.x + u * NT;
            x[u] = r >= jr ? p[u][j] : 0.0f;
            if (r == jr) {
#pragma unroll
                for (int k = 0; k < PB; ++k) S.row[buf][k] = p[u][k];
            }
        }
#pragma unroll
        for (int k = 0; k < PB; ++k) {
            d[k] = x[0] * p[0][k];
#pragma unroll
            for (int u = 1; u < R; ++u) d[k] = fmaf(x[u], p[u][k], d[k]);
        }
        // warp sums of the 16 values, each step halving the values a lane keeps:
        // lane l ends with the sum of value l & 15
#pragma unroll
        for (int w = PB / 2; w > 0; w >>= 1) {
            const bool up = (lane & w) != 0;
#pragma unroll
            for (int k = 0; k < PB / 2; ++k) {
                if (k >= w) break;
                const float send = up ? d[k] : d[k + w], keep = up ? d[k + w] : d[k];
                d[k] = keep + __shfl_xor_sync(0xffffffffu, send, w);
            }
        }
        d[0] += __shfl_xor_sync(0xffffffffu, d[0], 16);
        if (lane < PB) S.part[buf][warp][lane] = d[0];
        __syncthreads();
        float D = 0.0f;
#pragma unroll
        for (int w = 0; w < NWARP / 2; ++w) D += S.part[buf][w + (lane >> 4) * (NWARP / 2)][lane & 15];
        D += __shfl_xor_sync(0xffffffffu, D, 16);
        const float n2 = __shfl_sync(0xffffffffu, D, j);
        const float x0 = S.row[buf][j], nrm = sqrtf(n2);
        const float alpha = x0 > 0.0f ? -nrm : nrm;
        // 2 / v.v; a column 16 decades under the rows' mean norm is left alone (1 / v.v
        // stays in FP32's range, and the transform orthogonal)
        const float beta = n2 > 1e-32f ? 1.0f / (nrm * (nrm + fabsf(x0))) : 0.0f;
        const float vp = fmaf(-alpha, S.row[buf][lane & 15], D);                    // v . column (lane & 15)
        if (warp == 0) {
            if (lane < j) S.VV[lane][j] = vp;
            if (lane == 0) S.beta[j] = beta;
        }
        const float s = beta * vp;
#pragma unroll
        for (int u = 0; u < R; ++u) {
            const int r = threadIdx.x + u * NT;
            if (r == jr) x[u] = x0 - alpha;
            p[u][j] = x[u];   // v (0 above the pivot row)
        }
#pragma unroll
        for (int k = j + 1; k < PB; ++k) {
            const float sk = __shfl_sync(0xffffffffu, s, k);
#pragma unroll
            for (int u = 0; u < R; ++u) p[u][k] = fmaf(-sk, x[u], p[u][k]);
        }
    }
    // rows of the panel, zero to the next multiple of 16
    const int rows = (m - j0 + 15) & ~15;
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int i = (int)threadIdx.x + u * NT - j0;
        if (i < 0 || i >= rows) continue;
#pragma unroll
        for (int k = 0; k < PB; ++k) S.V[i * VS + k] = p[u][k];
    }
    for (int i = R * NT - j0 + threadIdx.x; i < rows; i += NT)
        for (int k = 0; k < PB; ++k) S.V[i * VS + k] = 0.0f;
    __syncthreads();
    // T = (diag(1 / beta) + strictly upper V^T V)^-1, lane = column
    if (warp == 0 && lane < PB) {
        float t[PB];
#pragma unroll
        for (int i = PB - 1; i >= 0; --i) {
            float a = 0.0f;
#pragma unroll
            for (int l = i + 1; l < PB; ++l) a = fmaf(l <= lane ? S.VV[i][l] : 0.0f, t[l], a);
            t[i] = i == lane ? S.beta[i] : (i < lane ? -S.beta[i] * a : 0.0f);
        }
#pragma unroll
        for (int i = 0; i < PB; ++i) S.T[i][lane] = t[i];
    }
    __syncthreads();
}

// A[j0 .. m)[c0 .. c0 + 31] <- (I - V T^T V^T) A, columns below ncol
__device__ void update_tile(Smem& S, float* A, int ld, int m, int j0, int c0, int ncol, int warp, int lane) {
    const int g = lane >> 2, tg = lane & 3;
    const int rows = m - j0, steps = (rows + 7) / 8;
    float acc[CT / 8][4];
#pragma unroll
    for (int n = 0; n < CT / 8; ++n)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[n][v] = 0.0f;
#pragma unroll 2
    for (int ks = warp; ks < steps; ks += NWARP) {
        const int i0 = 8 * ks + tg;
        float b[CT / 8][2];
#pragma unroll
        for (int n = 0; n < CT / 8; ++n)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = i0 + 4 * h, col = c0 + 8 * n + g;
                b[n][h] = i < rows && col < ncol ? __ldcg(A + (size_t)(j0 + i) * ld + col) : 0.0f;
            }
        uint32_t ah[4], al[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) split(S.V[(i0 + 4 * (v >> 1)) * VS + g + 8 * (v & 1)], ah[v], al[v]);
#pragma unroll
        for (int n = 0; n < CT / 8; ++n) {
            uint32_t bh[2], bl[2];
            split(b[n][0], bh[0], bl[0]);
            split(b[n][1], bh[1], bl[1]);
            mma_tf32(acc[n], al, bh);
            mma_tf32(acc[n], ah, bl);
            mma_tf32(acc[n], ah, bh);
        }
    }
#pragma unroll
    for (int n = 0; n < CT / 8; ++n)
#pragma unroll
        for (int h = 0; h < 2; ++h)
            *reinterpret_cast<float2*>(S.red + warp * PB * CT + (g + 8 * h) * CT + 8 * n + 2 * tg) =
                make_float2(acc[n][2 * h], acc[n][2 * h + 1]);
    __syncthreads();
    {
        static_assert(NT == PB * CT, "one element of W per thread");
        float s = 0.0f;
#pragma unroll
        for (int w = 0; w < NWARP; ++w) s += S.red[w * PB * CT + threadIdx.x];
        S.W[threadIdx.x] = s;
    }
    __syncthreads();
    {
        const int r = threadIdx.x / CT, c = threadIdx.x % CT;
        float s = 0.0f;
#pragma unroll
        for (int l = 0; l < PB; ++l) s = fmaf(S.T[l][r], S.W[l * CT + c], s);   // T is upper triangular
        S.W2[threadIdx.x] = -s;
    }
    __syncthreads();
    uint32_t bh[2][CT / 8][2], bl[2][CT / 8][2];
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int n = 0; n < CT / 8; ++n)
#pragma unroll
            for (int h = 0; h < 2; ++h) split(S.W2[(8 * k + tg + 4 * h) * CT + 8 * n + g], bh[k][n][h], bl[k][n][h]);
    for (int mt = warp; 16 * mt < rows; mt += NWARP) {
        const int i = 16 * mt + g;
        float2 a[CT / 8][2];
#pragma unroll
        for (int n = 0; n < CT / 8; ++n)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int col = c0 + 8 * n + 2 * tg;
                a[n][h] = i + 8 * h < rows && col < ncol
                              ? __ldcg(reinterpret_cast<const float2*>(A + (size_t)(j0 + i + 8 * h) * ld + col))
                              : make_float2(0.0f, 0.0f);
            }
        uint32_t ah[2][4], al[2][4];
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int v = 0; v < 4; ++v)
                split(S.V[(i + 8 * (v & 1)) * VS + 8 * k + tg + 4 * (v >> 1)], ah[k][v], al[k][v]);
#pragma unroll
        for (int n = 0; n < CT / 8; ++n) {
            float c[4] = {a[n][0].x, a[n][0].y, a[n][1].x, a[n][1].y};
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                mma_tf32(c, al[k], bh[k][n]);
                mma_tf32(c, ah[k], bl[k][n]);
                mma_tf32(c, ah[k], bh[k][n]);
            }
            const int col = c0 + 8 * n + 2 * tg;
            if (col >= ncol) continue;   // ncol is a multiple of 4
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (i + 8 * h < rows)
                    __stcg(reinterpret_cast<float2*>(A + (size_t)(j0 + i + 8 * h) * ld + col),
                           make_float2(c[2 * h], c[2 * h + 1]));
        }
    }
    __syncthreads();   // W2 and red are reused by the next tile
}

__global__ void __launch_bounds__(NT, 1) qr32_kernel(const OpDesc* descs, const int* cta_op, const int* cta_rank,
                                                     const int* group, unsigned* sync, unsigned long long timeout_ns,
                                                     int ld) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem& S = *reinterpret_cast<Smem*>(smem_raw);
    const int op = cta_op[blockIdx.x];
    if (op < 0) return;   // a CTA the plan left unused (graph step)
    const int rank = cta_rank[blockIdx.x];
    const int G = group[op];
    const OpDesc& d = descs[op];
    unsigned* sw = sync + (size_t)op * kSyncWords;
    const int m = d.c, n = d.L;   // of theta~, or of theta~^T
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned gen = 0;
    float* A = d.W32;
    float* U = d.U32;
    // squared column norms of theta~ (column-major in Acm)
    for (int k = rank * NWARP + warp; k < n; k += G * NWARP) {
        const double* y = d.Acm + (size_t)k * ld;
        double s = 0.0;
        for (int i = lane; i < m; i += 32) s = fma(y[i], y[i], s);
        s = warp_sum(s);
        if (lane == 0) __stcg(d.snorm + k, s);
    }
    if (!op_barrier(sw, G, gen, timeout_ns)) goto timeout;
    {
        double f = 0.0;
        for (int k = threadIdx.x; k < n; k += NT) f += __ldcg(d.snorm + k);
        f = warp_sum(f);
        if (lane == 0) S.sum[warp] = f;
        __syncthreads();
        if (threadIdx.x == 0) {
            f = 0.0;
            for (int w = 0; w < NWARP; ++w) f += S.sum[w];
            S.scale = f > 0.0 ? sqrt((double)m / f) : 1.0;   // rows of unit mean square norm
        }
        __syncthreads();
        // columns by decreasing norm (ties: by index), the same order in every CTA
        float* nrm = S.red;
        int* perm = reinterpret_cast<int*>(S.red + kMaxM);
        const double sc2 = S.scale * S.scale;
        for (int k = threadIdx.x; k < n; k += NT) {
            nrm[k] = (float)(__ldcg(d.snorm + k) * sc2);
            perm[k] = k;
        }
        __syncthreads();
        for (int k = threadIdx.x; k < n; k += NT) {
            const float v = nrm[k];
            int r = 0;
            for (int l = 0; l < n; ++l) r += nrm[l] > v || (nrm[l] == v && l < k);
            perm[r] = k;
        }
        __syncthreads();
        // A_1 and Q^T = I, row by row
        const double sc = S.scale;
        for (int i = rank * NWARP + warp; i < m; i += G * NWARP) {
            for (int j = lane; j < m; j += 32) {
                double a = 0.0;
                for (int f = 0; f * m < n; ++f) {   // fold f, every other one backwards
                    const int k = f * m + (f & 1 ? m - 1 - j : j);
                    if (k >= n) continue;
                    const int row = d.transposed ? perm[k] : i, col = d.transposed ? i : perm[k];
                    const double lam = d.lam_left ? d.lam_left[row >> 2] : 1.0;
                    a += lam * d.thetap[(size_t)row * ld + col];
                }
                __stcg(A + (size_t)i * ld + j, (float)(sc * a));
                __stcg(U + (size_t)i * ld + j, i == j ? 1.0f : 0.0f);
            }
        }
    }
    if (!op_barrier(sw, G, gen, timeout_ns)) goto timeout;
    for (int j0 = 0; j0 < m; j0 += PB) {
        if (m <= NT)
            factor_panel<1>(S, A, ld, m, j0, warp, lane);
        else if (m <= 2 * NT)
            factor_panel<2>(S, A, ld, m, j0, warp, lane);
        else
            factor_panel<4>(S, A, ld, m, j0, warp, lane);
        const int first = j0 + PB;
        const int ta = first < m ? (m - first + CT - 1) / CT : 0, tq = (m + CT - 1) / CT;
        for (int t = rank; t < ta + tq; t += G) {
            if (t < ta)
                update_tile(S, A, ld, m, j0, first + t * CT, m, warp, lane);
            else
                update_tile(S, U, ld, m, j0, (t - ta) * CT, m, warp, lane);
        }
        if (!op_barrier(sw, G, gen, timeout_ns)) goto timeout;
    }
    return;
timeout:
    if (threadIdx.x == 0) atomicOr(d.status, (int)MPDO_ST_TIMEOUT);
}

}  // namespace

cudaError_t qr32_max_resident(int* blocks) {
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(qr32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, qr32_kernel, NT, sizeof(Smem));
    *blocks = sms * per;
    return e;
}

cudaError_t launch_qr32(const OpDesc* d_desc, const int* d_cta_op, const int* d_cta_rank, const int* d_group,
                        unsigned* d_sync, int grid, unsigned long long timeout_ns, int ld, cudaStream_t st) {
    if (grid <= 0) return cudaSuccess;
    void* args[] = {(void*)&d_desc, (void*)&d_cta_op,   (void*)&d_cta_rank, (void*)&d_group,
                    (void*)&d_sync, (void*)&timeout_ns, (void*)&ld};
    return cudaLaunchCooperativeKernel((const void*)qr32_kernel, dim3(grid), dim3(NT), args, sizeof(Smem), st);
}

}  // namespace mpdo

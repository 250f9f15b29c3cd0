// Trace forcing and Pauli observables from the MPO (Sec. 2.3-2.4, App. A).
//
// With r_{a1..aN} = B_0[a1] ... B_{N-1}[aN] the coefficients of rho in the
// normalised Pauli basis, Tr(P_a/sqrt2) = sqrt2 delta_{a,I} per site gives
//   tr rho = 2^{N/2} E(I...I),   Tr(sigma^a_i rho) = 2^{N/2} E(..a at i..),
// E(string) = product over sites of the selected a-slices of the B's.  So
//   <sigma^a_i> = E(a at i)/E(I..I),  <sigma^a_i sigma^b_j> = E(a at i, b at j)/E(I..I).
// Left environments L_p = E-prefix over sites < p (row vectors), right
// environments R_p = suffix over sites >= p (column vectors), all with I.
#include <cooperative_groups.h>
#include <mpdo.h>

#include "internal.h"

namespace mpdo {

namespace {

// one site tensor, read as double whatever the storage (f64 or f32)
struct SiteRef {
    const void* p;
    int f32;
    __device__ double operator[](size_t i) const { return site_ld(p, i, f32); }
};

__device__ __forceinline__ SiteRef site_ptr(const void* sites, int f32, int b, int p, int n, int cap) {
    const size_t off = ((size_t)b * n + p) * (size_t)cap * 4 * cap;
    return SiteRef{f32 ? (const void*)(static_cast<const float*>(sites) + off)
                       : (const void*)(static_cast<const double*>(sites) + off),
                   f32};
}

// ---------------------------------------------------------------------------
// Products of a vector with one Pauli slice, a CTA's share of the output.  A slice
// is read once and its rows are contiguous, so the lanes run along r in both.  What
// bounds them is the FP64 pipe, two FMAs per SM and clock: an instruction of a warp
// takes it 16 clocks whether one lane or all are active, so lanes without a column
// take other rows and the sums over lanes fold four rows at once.
constexpr int CW = 8;                 // warps per CTA
constexpr int kColTile = 64;          // columns per CTA of a row product at most

// out(c) = sum_l v[l] S[l][comp][r0 + c], c < w <= kColTile; red: CW * kColTile doubles
template <class F>
__device__ __forceinline__ void row_product(SiteRef S, int comp, int cl, int cap, const double* v, int r0, int w,
                                            double* red, F out) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int U = 8;   // rows in flight
    if (w > 32) {
        double a0 = 0.0, a1 = 0.0;
        const bool two = lane + 32 < w;
        for (int l = warp; l < cl; l += U * CW) {
            double x[U], y[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const size_t at = ((size_t)(l + u * CW) * 4 + comp) * cap + r0 + lane;
                x[u] = l + u * CW < cl ? S[at] : 0.0;
                y[u] = l + u * CW < cl && two ? S[at + 32] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (l + u * CW < cl) {
                    a0 = fma(v[l + u * CW], x[u], a0);
                    a1 = fma(v[l + u * CW], y[u], a1);
                }
        }
        red[warp * kColTile + lane] = a0;
        red[warp * kColTile + 32 + lane] = a1;
    } else if (w > 0) {
        int cb = 1;
        while (cb < w) cb <<= 1;   // lanes per row
        const int rows = 32 / cb, g = lane / cb, c = lane % cb, step = CW * rows;
        double a0 = 0.0;
        for (int l0 = warp * rows; l0 < cl; l0 += U * step) {
            double x[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int l = l0 + u * step + g;
                x[u] = l < cl && c < w ? S[((size_t)l * 4 + comp) * cap + r0 + c] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (l0 + u * step < cl) {
                    const int l = l0 + u * step + g;
                    a0 = fma(l < cl ? v[l] : 0.0, x[u], a0);
                }
        }
        for (int o = cb; o < 32; o <<= 1) a0 += __shfl_xor_sync(0xffffffffu, a0, o);
        if (g == 0) red[warp * kColTile + c] = a0;
    }
    __syncthreads();
    for (int c = threadIdx.x; c < w; c += CW * 32) {
        double sum = 0.0;
#pragma unroll
        for (int u = 0; u < CW; ++u) sum += red[u * kColTile + c];
        out(c, sum);
    }
    __syncthreads();
}

// out(l) = sum_r S[l][comp][r] v[r] for l0 <= l < l1 (called by one lane of a warp),
// four rows per warp at a time
template <class F>
__device__ __forceinline__ void column_product(SiteRef S, int comp, int cr, int cap, const double* v, int l0, int l1,
                                               F out) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int U = 4;   // loads in flight per row
    for (int lb = l0 + 4 * warp; lb < l1; lb += 4 * CW) {
        double a[4] = {};
        for (int rb = 0; rb < cr; rb += 32 * U) {
            double x[4][U];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int r = rb + 32 * u + lane;
                    x[i][u] = lb + i < l1 && r < cr ? S[((size_t)(lb + i) * 4 + comp) * cap + r] : 0.0;
                }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (rb + 32 * u < cr) {
                    const int r = rb + 32 * u + lane;
                    const double vr = r < cr ? v[r] : 0.0;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (lb + i < l1) a[i] = fma(x[i][u], vr, a[i]);
                }
        }
        // lanes 0, 8, 16, 24 end with rows 0 .. 3
        const bool h = lane & 16, q = lane & 8;
        const double k0 = (h ? a[2] : a[0]) + __shfl_xor_sync(0xffffffffu, h ? a[0] : a[2], 16);
        const double k1 = (h ? a[3] : a[1]) + __shfl_xor_sync(0xffffffffu, h ? a[1] : a[3], 16);
        double k = (q ? k1 : k0) + __shfl_xor_sync(0xffffffffu, q ? k0 : k1, 8);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
        const int l = lb + (h ? 2 : 0) + (q ? 1 : 0);
        if ((lane & 7) == 0 && l < l1) out(l, k);
    }
}

// A cluster of 1 to 16 CTAs carries a vector through the chain, from the left
// (v <- v B_p[I], p = 0 ..) or from the right (v <- B_p[I] v, p = n - 1 ..).  The
// sites are serial, so what counts is a site's latency: every CTA takes its share
// of the output, writes it into all copies of the vector through distributed
// shared memory, and the cluster's barrier ends the site.  With a launch per site and
// the pairs below carried through the whole chain, <X>, <Y>, <Z> and all <ZZ> of 40
// sites at chi 512 took 3.97 ms, of four chains of 8 at chi 32 383 us; now 2.07 ms
// and 263 us.  E, if not null, receives the vector at every bond.  Returns the first entry of the last vector.
__device__ double chain(bool left, const void* sites, int f32, const int* dm, int b, int n, int cap, double* E) {
    namespace cg = cooperative_groups;
    const cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), EC = (int)cluster.num_blocks();
    __shared__ double v[2][kMaxChi];
    __shared__ double red[CW * kColTile];
    if (threadIdx.x == 0) {
        v[0][0] = 1.0;
        if (E && rank == 0) E[left ? 0 : (size_t)n * cap] = 1.0;
    }
    cluster.sync();   // every CTA runs before its shared memory is written
    int cur = 0;
    for (int t = 0; t < n; ++t) {
        const int p = left ? t : n - 1 - t, cl = dm[p], cr = dm[p + 1];
        const SiteRef S = site_ptr(sites, f32, b, p, n, cap);
        const int len = left ? cr : cl, w = (len + EC - 1) / EC;
        const int o0 = min(rank * w, len), o1 = min(o0 + w, len);
        double* row = E ? E + (size_t)(left ? p + 1 : p) * cap : nullptr;
        double* next = v[cur ^ 1];
        auto put = [&](int o, double x) {
            if (row) row[o] = x;
            for (int k = 0; k < EC; ++k) cluster.map_shared_rank(next, k)[o] = x;
        };
        if (left)
            row_product(S, 0, cl, cap, v[cur], o0, o1 - o0, red, [&](int c, double x) { put(o0 + c, x); });
        else
            column_product(S, 0, cr, cap, v[cur], o0, o1, put);
        cur ^= 1;
        cluster.sync();
    }
    return v[cur][0];
}

// CTAs per cluster: chi^2 / 2 clocks of the FP64 pipe per site are shared among them,
// a cluster barrier is about 700.
constexpr int kBigCluster = 16;   // beyond the portable 8
int chain_ctas(int chi_cap) { return chi_cap <= 32 ? 1 : chi_cap <= 64 ? 4 : chi_cap <= 128 ? 8 : kBigCluster; }
static_assert(kMaxChi <= 8 * kColTile && 32 <= kColTile && 64 <= 4 * kColTile, "a CTA's share of a row product");

template <class... P, class... A>
cudaError_t launch_cluster(void (*kernel)(P...), dim3 grid, int ctas, cudaStream_t st, A... args) {
    cudaError_t e = cudaSuccess;
    if (ctas > 8) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(CW * 32);
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = ctas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Tr rho of every instance; force: site 0 over it
__global__ void __launch_bounds__(CW * 32)
    trace_kernel(void* sites, int f32, const int* dims, int n, int cap, int force, double* trace_out, int* status) {
    const int EC = (int)cooperative_groups::this_cluster().num_blocks(), b = blockIdx.x / EC;
    const int* dm = dims + (size_t)b * (n + 1);
    const double tr = exp2(0.5 * n) * chain(true, sites, f32, dm, b, n, cap, nullptr);
    if (blockIdx.x % EC) return;
    if (threadIdx.x == 0) {
        trace_out[b] = tr;
        if (!isfinite(tr) || tr == 0.0) atomicOr(status + b, (int)MPDO_ST_NONFINITE);
    }
    if (force && isfinite(tr) && tr != 0.0) {
        void* S = const_cast<void*>(site_ptr(sites, f32, b, 0, n, cap).p);
        const double inv = 1.0 / tr;
        const int cr = dm[1];
        for (int e = threadIdx.x; e < 4 * cr; e += blockDim.x) {
            const size_t i = (size_t)(e / cr) * cap + (e % cr);
            site_st(S, i, site_ld(S, i, f32) * inv, f32);
        }
    }
}

// Both environments in one launch, blockIdx.y 0 from the left (L_{p+1} = L_p B_p[I]),
// 1 from the right (R_p = B_p[I] R_{p+1}).
__global__ void __launch_bounds__(CW * 32)
    env_chain_kernel(const void* sites, int f32, const int* dims, int n, int cap, double* envL, double* envR) {
    const int b = blockIdx.z;
    const bool left = blockIdx.y == 0;
    chain(left, sites, f32, dims + (size_t)b * (n + 1), b, n, cap,
          (left ? envL : envR) + (size_t)b * (n + 1) * cap);
}

// out[b*nq + k] = E(comp at q_k) / E0 (qs null: q_k = k), the rows of the site shared
// by a cluster of CTAs
__global__ void __launch_bounds__(CW * 32)
    one_kernel(const void* sites, int f32, const int* dims, int n, int cap, const double* envL, const double* envR,
               const int* qs, int nq, int comp, double* out) {
    namespace cg = cooperative_groups;
    const cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), EC = (int)cluster.num_blocks();
    const int k = blockIdx.x / EC, b = blockIdx.y;
    const int q = qs ? qs[k] : k;
    const int* dm = dims + (size_t)b * (n + 1);
    const double* Lq = envL + ((size_t)b * (n + 1) + q) * cap;
    const double* Rq = envR + ((size_t)b * (n + 1) + q + 1) * cap;
    const SiteRef S = site_ptr(sites, f32, b, q, n, cap);
    const int cl = dm[q], cr = dm[q + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __shared__ double sums[kBigCluster], red[CW];
    const int w = (cl + EC - 1) / EC, l0 = min(rank * w, cl), l1 = min(l0 + w, cl);
    double part = 0.0;
    cluster.sync();   // every CTA runs before its shared memory is written
    column_product(S, comp, cr, cap, Rq, l0, l1, [&](int l, double x) { part = fma(Lq[l], x, part); });
#pragma unroll
    for (int o = 16; o >= 8; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);   // lanes 0, 8, 16, 24
    if (lane == 0) red[warp] = part;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int u = 0; u < CW; ++u) s += red[u];
        cluster.map_shared_rank(sums, 0)[rank] = s;
    }
    cluster.sync();
    if (rank == 0 && threadIdx.x == 0) {
        double s = 0.0;
        for (int u = 0; u < EC; ++u) s += sums[u];
        out[(size_t)b * nq + k] = s / envL[((size_t)b * (n + 1) + n) * cap];
    }
}

// ---------------------------------------------------------------------------
// All-pairs two-point values.  With s_i = L_i B_i[ca] (at bond i + 1) and
// u_j = B_j[cb] R_{j+1} (at bond j), E(ca at i, cb at j) is s_i carried through the
// sites between them, dotted with u_j.  The chain is cut in the middle, at bond
// m = n / 2: the s_i of the left half are carried right to it, the u_j of the right
// half left to it, each step taking one site of either half:
//   left, site t:  E(i, t) = w_i . u_t, then w_i <- w_i B_t[I], for i < t;
//   right, site p: E(p, j) = s_p . u_j, then u_j <- B_p[I] u_j, for j > p;
// and the pairs across the middle are dot products at bond m.  Against carrying
// every s_i through all later sites with both slices, that is half the steps, an
// eighth of the FP64 work and one slice per site instead of three (the propagation
// is bound by the FP64 pipe at chi 512, by the serial steps below).
//
// Scratch (doubles): seeds s [b][n][cap], u [b][n][cap], then two buffers
// [b][n][cap] of carried rows (i < m: w_i, j >= m: u_j).
struct Pairs {
    const void* sites;
    int f32;
    const int* dims;
    int n, cap, B;
    const double *envL, *envR;
    const int* need;      // [n] rows i, then [n] columns j, that some pair asks for
    double *s, *u, *buf;  // scratch
    double* full;         // [b][i][j]
    __device__ double* row(int which, int b, int i) const {
        return buf + (((size_t)which * B + b) * n + i) * cap;
    }
    __device__ void put(int b, int i, int j, double e) const {
        full[((size_t)b * n + i) * n + j] = e / envL[((size_t)b * (n + 1) + n) * cap];
    }
};

__device__ __forceinline__ double warp_dot(const double* x, const double* y, int len, int lane) {
    double a = 0.0;
    for (int k = lane; k < len; k += 32) a = fma(x[k], y[k], a);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    return a;
}

// the seeds: grid (tiles of kColTile x 2, site, instance)
__global__ void __launch_bounds__(CW * 32) pair_seed_kernel(Pairs P, int ca, int cb) {
    const int p = blockIdx.y, b = blockIdx.z;
    const bool left = (blockIdx.x & 1) == 0;
    if (!P.need[left ? p : P.n + p]) return;
    const int* dm = P.dims + (size_t)b * (P.n + 1);
    const int cl = dm[p], cr = dm[p + 1], o0 = (blockIdx.x >> 1) * kColTile, len = left ? cr : cl;
    if (o0 >= len) return;
    const SiteRef S = site_ptr(P.sites, P.f32, b, p, P.n, P.cap);
    __shared__ double red[CW * kColTile];
    const size_t at = ((size_t)b * P.n + p) * P.cap, env = ((size_t)b * (P.n + 1) + p) * P.cap;
    if (left)
        row_product(S, ca, cl, P.cap, P.envL + env, o0, min(kColTile, len - o0), red,
                    [&](int c, double x) { P.s[at + o0 + c] = x; });
    else
        column_product(S, cb, cr, P.cap, P.envR + env + P.cap, o0, min(o0 + kColTile, len),
                       [&](int l, double x) { P.u[at + l] = x; });
}

// Step s: site s of the left half (blockIdx.y 0), site n - 1 - s of the right half
// (1).  A CTA takes TW outputs of every carried row, the slice's part for them in
// shared memory, a warp one row at a time; the rows' dot products are spread over
// the CTAs.
constexpr int TW = 4;
__global__ void __launch_bounds__(CW * 32) pair_step_kernel(Pairs P, int s, int m) {
    const bool left = blockIdx.y == 0;
    const int p = left ? s : P.n - 1 - s, b = blockIdx.z, n = P.n, cap = P.cap;
    if (left ? p >= m : p < m) return;
    const int* dm = P.dims + (size_t)b * (n + 1);
    const int cl = dm[p], cr = dm[p + 1];
    const int len = left ? cr : cl, in = left ? cl : cr;   // outputs, inputs
    const int ntiles = (len + TW - 1) / TW, o0 = blockIdx.x * TW;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r0 = left ? 0 : p + 1, r1 = left ? p : n;     // carried rows
    const int* need = left ? P.need : P.need + n;
    auto source = [&](int r) -> const double* {   // a row enters from its seed
        if (left ? r == p - 1 : r == p + 1) return (left ? P.s : P.u) + ((size_t)b * n + r) * cap;
        return P.row((s - 1) & 1, b, r);
    };
    // dot products with the site's own seed, one row per warp of the launch
    if (P.need[left ? n + p : p]) {
        const double* own = (left ? P.u : P.s) + ((size_t)b * n + p) * cap;
        for (int r = r0 + blockIdx.x * CW + warp; r < r1; r += gridDim.x * CW) {
            if (!need[r]) continue;
            const double e = warp_dot(source(r), own, in, lane);
            if (lane == 0) P.put(b, left ? r : p, left ? p : r, e);
        }
    }
    if ((int)blockIdx.x >= ntiles) return;
    extern __shared__ double sI[];   // [in][TW]: slice I, the tile's outputs
    const SiteRef S = site_ptr(P.sites, P.f32, b, p, n, cap);
    for (int e = threadIdx.x; e < in * TW; e += CW * 32) {
        const int x = left ? e / TW : e % in, o = left ? e % TW : e / in;   // along r in both
        const int l = left ? x : o0 + o, r = left ? o0 + o : x;
        sI[x * TW + o] = o0 + o < len ? S[(size_t)l * 4 * cap + r] : 0.0;
    }
    __syncthreads();
    for (int r = r0 + warp; r < r1; r += CW) {
        if (!need[r]) continue;
        const double* w = source(r);
        double a[TW] = {};
        for (int x = lane; x < in; x += 32) {
            const double wx = w[x];
            const double2 q0 = *reinterpret_cast<const double2*>(sI + x * TW);
            const double2 q1 = *reinterpret_cast<const double2*>(sI + x * TW + 2);
            a[0] = fma(wx, q0.x, a[0]);
            a[1] = fma(wx, q0.y, a[1]);
            a[2] = fma(wx, q1.x, a[2]);
            a[3] = fma(wx, q1.y, a[3]);
        }
#pragma unroll
        for (int c = 0; c < TW; ++c)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a[c] += __shfl_xor_sync(0xffffffffu, a[c], o);
        if (lane < TW && o0 + lane < len)
            P.row(s & 1, b, r)[o0 + lane] = lane == 0 ? a[0] : lane == 1 ? a[1] : lane == 2 ? a[2] : a[3];
    }
}

// pairs i < m <= j at bond m, one per warp
__global__ void __launch_bounds__(CW * 32) pair_cross_kernel(Pairs P, int m) {
    const int b = blockIdx.y, n = P.n, lane = threadIdx.x & 31;
    const int e = blockIdx.x * CW + (threadIdx.x >> 5);
    if (e >= m * (n - m)) return;
    const int i = e / (n - m), j = m + e % (n - m);
    if (!P.need[i] || !P.need[n + j]) return;
    const double* w = i == m - 1 ? P.s + ((size_t)b * n + i) * P.cap : P.row((m - 1) & 1, b, i);
    const double* u = j == m ? P.u + ((size_t)b * n + j) * P.cap : P.row((n - 1 - m) & 1, b, j);
    const double v = warp_dot(w, u, P.dims[(size_t)b * (n + 1) + m], lane);
    if (lane == 0) P.put(b, i, j, v);
}

// trip[t] = (i, j, k): out[b][k] = full[b][i][j] (minus one_a[b][i] one_b[b][j] if connected)
__global__ void gather_kernel(const double* full, const double* one_a, const double* one_b, const int* trip, int m,
                              int np, int n, int B, int connected, double* out) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m * B) return;
    const int b = t / m, u = t % m;
    const int i = trip[3 * u], j = trip[3 * u + 1], k = trip[3 * u + 2];
    double v = full[((size_t)b * n + i) * n + j];
    if (connected) v -= one_a[(size_t)b * n + i] * one_b[(size_t)b * n + j];
    out[(size_t)b * np + k] = v;
}

}  // namespace

cudaError_t launch_trace_normalize(void* sites, int sites_f32, const int* dims, int n, int B, int chi_cap, int force,
                                   double* trace_out, int* status, cudaStream_t st) {
    const int ctas = chain_ctas(chi_cap);
    return launch_cluster(trace_kernel, dim3(ctas * B), ctas, st, sites, sites_f32, dims, n, chi_cap, force, trace_out,
                          status);
}

cudaError_t launch_environments(const void* sites, int sites_f32, const int* dims, int n, int B, int chi_cap,
                                double* envL, double* envR, cudaStream_t st) {
    const int ctas = chain_ctas(chi_cap);
    return launch_cluster(env_chain_kernel, dim3(ctas, 2, B), ctas, st, sites, sites_f32, dims, n, chi_cap, envL, envR);
}

cudaError_t launch_measure_1q(const void* sites, int sites_f32, const int* dims, int n, int B, int chi_cap,
                              const double* envL, const double* envR, const int* d_q, int nq, int comp, double* out,
                              cudaStream_t st) {
    if (nq <= 0) return cudaSuccess;
    const int ctas = chi_cap <= 64 ? 1 : chi_cap <= 128 ? 4 : 8;
    return launch_cluster(one_kernel, dim3(ctas * nq, B), ctas, st, sites, sites_f32, dims, n, chi_cap, envL, envR, d_q,
                          nq, comp, out);
}

size_t two_stack_doubles(int n, int B, int chi_cap) { return (size_t)4 * B * n * chi_cap; }

cudaError_t launch_measure_2q(const void* sites, int sites_f32, const int* dims, int n, int B, int chi_cap,
                              const double* envL, const double* envR, int ca, int cb, const int* d_need,
                              double* wstack, double* full, cudaStream_t st) {
    const size_t rows = (size_t)B * n * chi_cap;
    const Pairs P{sites, sites_f32, dims, n, chi_cap, B, envL, envR, d_need, wstack, wstack + rows, wstack + 2 * rows, full};
    const int m = n / 2, steps = n - 1 - m > m - 1 ? n - 1 - m : m - 1;
    pair_seed_kernel<<<dim3(2 * ((chi_cap + kColTile - 1) / kColTile), n, B), CW * 32, 0, st>>>(P, ca, cb);
    cudaError_t e = cudaGetLastError();
    const size_t smem = (size_t)chi_cap * TW * sizeof(double);
    static_assert((size_t)kMaxChi * TW * sizeof(double) <= 48 * 1024, "within the default shared memory");
    for (int s = 1; s <= steps && e == cudaSuccess; ++s) {
        pair_step_kernel<<<dim3((chi_cap + TW - 1) / TW, 2, B), CW * 32, smem, st>>>(P, s, m);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
    pair_cross_kernel<<<dim3((m * (n - m) + CW - 1) / CW, B), CW * 32, 0, st>>>(P, m);
    return cudaGetLastError();
}

cudaError_t launch_gather_2q(const double* full, const double* one_a, const double* one_b, const int* d_trip,
                             int m, int np, int n, int B, int connected, double* out, cudaStream_t st) {
    if (m <= 0) return cudaSuccess;
    const int tot = m * B;
    gather_kernel<<<(tot + 255) / 256, 256, 0, st>>>(full, one_a, one_b, d_trip, m, np, n, B, connected, out);
    return cudaGetLastError();
}

}  // namespace mpdo

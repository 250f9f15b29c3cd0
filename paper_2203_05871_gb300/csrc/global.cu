// Global characteristics of the state (Sec. 2.3): the second Renyi entropy
// S2 = -ln tr(rho^2) (Eq. (S_2)) and the operator space entanglement entropy
// of the vectorised state |rho>> for a cut of the MPO path (Eq. (OSEE)).
//
// The basis P_a/sqrt2 is orthonormal for the trace inner product, so
// tr(rho^2) = sum_a r_a^2 = <<rho|rho>>, the squared norm of the coefficient
// MPS, and for the normalised rho tr(rho^2) = <<rho|rho>> / (tr rho)^2.
//
// Gram matrices of the two halves of the chain at bond p (between positions
// p and p+1), both chi x chi with chi = dims[p+1]:
//   X_0 = [1],      X_{q+1} = sum_s B_q[s]^T X_q B_q[s]      (q = 0 .. p)
//   Y_N = [1],      Y_q     = sum_s B_q[s] Y_{q+1} B_q[s]^T  (q = N-1 .. p+1)
// With r = M_L M_R through the bond index, X = M_L^T M_L and Y = M_R M_R^T, and
// the squared Schmidt values of |rho>> at the cut are the eigenvalues of X Y.
// Each Gram matrix is factored by the one-sided Jacobi SVD of its rows
// (X = V diag(x) V^T, rows w_j = x_j v_j^T after convergence), F_X = rows
// w_j / sqrt(x_j) with F_X^T F_X = X, and likewise F_Y; then eig(X Y) =
// sv(F_X F_Y^T)^2, so a third Jacobi SVD, of C = F_X F_Y^T, gives the Schmidt
// values s_k and OSEE = -sum_k p_k ln p_k with p_k = s_k^2 / sum s^2.
// FP64 throughout.  The Gram sweeps are batched products: on FP64 contexts exact
// slice products on the tensor cores (oz_gemm.cu, seven slices), else, and for states
// in a bond gauge that those do not resolve (gauge.cu), FP64 GEMMs
// (gemm.cu: 0.68 ms for X' at chi 256, where 16 CTAs share it, against 0.07 ms).
// The SVDs end at the strict tolerance sqrt(L) eps, through a step's stages where
// staged_svd says so, else in the FP64 pass of jacobi.cu alone.  Squaring
// the bond matrix into X and Y costs accuracy only on the smallest p_k, at the
// 1e-16 level of the largest, which moves the entropy by ~1e-14.
#include <mpdo.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "ctx.h"
#include "internal.h"

using namespace mpdo;

namespace mpdo {

namespace {

// X and Y of instance i of a chunk: slots 2i and 2i+1; [0][0] = 1
__global__ void gram_unit_kernel(double* W, size_t mat, int m) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 2 * m) return;
    W[(size_t)i * mat] = 1.0;
}

// norms[s * 2 ld + j] = |row j| of the matrix in slot s (rows j < chi[s]), staged or not
__global__ void row_norms_kernel(const double* W, const double* Ws, size_t mat, int ld, const int* chi,
                                 const int* staged, double* norms) {
    const int s = blockIdx.y;
    const int n = chi[s];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const double* M = (staged[s] ? Ws : W) + (size_t)s * mat;
    for (int j = blockIdx.x * 8 + warp; j < n; j += gridDim.x * 8) {
        double a = 0.0;
        for (int k = lane; k < n; k += 32) a = fma(M[(size_t)j * ld + k], M[(size_t)j * ld + k], a);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane == 0) norms[(size_t)s * 2 * ld + j] = sqrt(a);
    }
}

// slot s of C: [j][k] /= sqrt(|x_j| |y_k|) (0 where either norm is 0), x the rows of slot
// s and y those of its partner: F_X F_Y^T (even slots) or its transpose (odd ones, staged)
__global__ void scale_kernel(double* C, size_t mat, int ld, const int* chi, const int* staged, const double* norms) {
    const int s = blockIdx.y;
    if ((s & 1) && !staged[s]) return;
    const int n = chi[s];
    const double* nx = norms + (size_t)s * 2 * ld;
    const double* ny = norms + (size_t)(s ^ 1) * 2 * ld;
    double* M = C + (size_t)s * mat;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += gridDim.x * blockDim.x) {
        const int j = e / n, k = e % n;
        const double d = nx[j] * ny[k];
        M[(size_t)j * ld + k] = d > 0.0 ? M[(size_t)j * ld + k] / sqrt(d) : 0.0;
    }
}

// out[b0 + i] = OSEE from the row norms s_k of C_i after its Jacobi SVD
__global__ void osee_kernel(const double* C, const double* Cs, size_t mat, int ld, const int* chi, const int* staged,
                            int b0, double* out) {
    const int i = blockIdx.x;
    const int n = chi[2 * i];
    const double* M = (staged[2 * i] ? Cs : C) + (size_t)(2 * i) * mat;
    __shared__ double s2[4 * kMaxChi];
    __shared__ double red[32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int j = warp; j < n; j += nw) {
        double a = 0.0;
        for (int k = lane; k < n; k += 32) a = fma(M[(size_t)j * ld + k], M[(size_t)j * ld + k], a);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane == 0) s2[j] = a;
    }
    __syncthreads();
    double t = 0.0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) t += s2[j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) red[warp] = t;
    __syncthreads();
    double tot = 0.0;
    for (int w = 0; w < nw; ++w) tot += red[w];
    __syncthreads();
    double h = 0.0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const double p = tot > 0.0 ? s2[j] / tot : 0.0;
        if (p > 0.0) h -= p * log(p);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
    if (lane == 0) red[warp] = h;
    __syncthreads();
    if (threadIdx.x == 0) {
        double e = 0.0;
        for (int w = 0; w < nw; ++w) e += red[w];
        out[b0 + i] = e;
    }
}

// out[b0 + i] = -ln(X_i[0][0] / (2^{N/2} E0_b)^2), X_i = <<rho|rho>> after the full left sweep
__global__ void renyi2_kernel(const double* W, size_t mat, const double* envL, int n, int cap, int b0, int m,
                              double* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const int b = b0 + i;
    const double nrm2 = W[(size_t)(2 * i) * mat];
    const double tr = exp2(0.5 * n) * envL[((size_t)b * (n + 1) + n) * cap];
    out[b] = -log(nrm2 / (tr * tr));
}

struct GqPlan {
    std::vector<GemmDesc> g;
    struct Launch {
        size_t first;
        int count, max_m, max_n;
    };
    std::vector<Launch> launches;
    void begin() { launches.push_back(Launch{g.size(), 0, 1, 1}); }
    void add(GemmDesc d, int* status) {
        d.status = status;
        g.push_back(d);
        Launch& L = launches.back();
        ++L.count;
        L.max_m = std::max(L.max_m, d.M);
        L.max_n = std::max(L.max_n, d.N);
    }
};

// Left Gram sweep over sites 0..last of the chunk's instances, those with a bond gauge that
// slice products do not resolve (gauge.cu) or the others: X (slot 2i) is
// chi x chi with chi = dims[last + 1] at the end.  T (thetap slot 2i) holds X B.
void plan_left(mpdo_ctx* c, int b0, int m, int last, bool wide, GqPlan& P) {
    const int N = c->N, cap = c->cap, ld = c->ld;
    const size_t mat = (size_t)ld * ld;
    const int f32 = sites_f32(c);
    for (int q = 0; q <= last; ++q) {
        P.begin();
        for (int i = 0; i < m; ++i) {
            const int b = b0 + i;
            if (wide_instance(c, b) != wide) continue;
            const int l = c->h_dims[(size_t)b * (N + 1) + q], r = c->h_dims[(size_t)b * (N + 1) + q + 1];
            double* X = c->d_Z + (size_t)(2 * i) * mat;
            double* T = c->d_thetap + (size_t)(2 * i) * mat;
            // T[l][(s, r)] = sum_l' X[l][l'] B[l'][s][r]
            P.add(GemmDesc{l, 3 * cap + r, l, X, ld, 0, site_v(c, b, q), 4 * cap, f32, 0, T, 4 * cap, 1.0, 0.0,
                           nullptr, 0, 0, 0, 0, 0}, c->d_status + b);
        }
        P.begin();
        for (int i = 0; i < m; ++i) {
            const int b = b0 + i;
            if (wide_instance(c, b) != wide) continue;
            const int l = c->h_dims[(size_t)b * (N + 1) + q], r = c->h_dims[(size_t)b * (N + 1) + q + 1];
            double* X = c->d_Z + (size_t)(2 * i) * mat;
            double* T = c->d_thetap + (size_t)(2 * i) * mat;
            // X'[r][r'] = sum_{(l, s)} B[(l, s)][r] T[(l, s)][r']  (both (4 l) x r with row stride cap)
            P.add(GemmDesc{r, r, 4 * l, site_v(c, b, q), cap, f32, T, cap, 0, 0, X, ld, 1.0, 0.0, nullptr, 0, 0, 0, 1,
                           1}, c->d_status + b);
        }
    }
}

// Right Gram sweep over sites N-1..first: Y (slot 2i + 1), U (thetap slot 2i + 1) holds B Y.
void plan_right(mpdo_ctx* c, int b0, int m, int first, bool wide, GqPlan& P) {
    const int N = c->N, cap = c->cap, ld = c->ld;
    const size_t mat = (size_t)ld * ld;
    const int f32 = sites_f32(c);
    for (int q = N - 1; q >= first; --q) {
        P.begin();
        for (int i = 0; i < m; ++i) {
            const int b = b0 + i;
            if (wide_instance(c, b) != wide) continue;
            const int l = c->h_dims[(size_t)b * (N + 1) + q], r = c->h_dims[(size_t)b * (N + 1) + q + 1];
            double* Y = c->d_Z + (size_t)(2 * i + 1) * mat;
            double* U = c->d_thetap + (size_t)(2 * i + 1) * mat;
            // U[(l, s)][r'] = sum_r B[(l, s)][r] Y[r][r']
            P.add(GemmDesc{4 * l, r, r, site_v(c, b, q), cap, f32, Y, ld, 0, 0, U, cap, 1.0, 0.0, nullptr, 0, 0, 0, 0,
                           0}, c->d_status + b);
        }
        for (int s = 0; s < 4; ++s) {
            P.begin();
            for (int i = 0; i < m; ++i) {
                const int b = b0 + i;
                if (wide_instance(c, b) != wide) continue;
                const int l = c->h_dims[(size_t)b * (N + 1) + q], r = c->h_dims[(size_t)b * (N + 1) + q + 1];
                double* Y = c->d_Z + (size_t)(2 * i + 1) * mat;
                double* U = c->d_thetap + (size_t)(2 * i + 1) * mat;
                const void* Bs = static_cast<const char*>(site_v(c, b, q)) + (size_t)s * cap * site_esize(c);
                // Y'[l][l'] (+)= sum_r U[(l, s)][r] B[(l', s)][r]
                P.add(GemmDesc{l, l, r, U + (size_t)s * cap, 4 * cap, 0, Bs, 4 * cap, f32, 1, Y, ld, 1.0,
                               s > 0 ? 1.0 : 0.0, s > 0 ? Y : nullptr, ld, 0, 0, 0, 0}, c->d_status + b);
            }
        }
    }
}

int run_plan(mpdo_ctx* c, bool wide, GqPlan& P) {
    if (P.g.empty()) return MPDO_OK;
    if (c->gq_cap < P.g.size()) {
        if (c->d_gq) cudaFree(c->d_gq);
        c->d_gq = nullptr;
        c->gq_cap = 0;
        CU(dalloc(&c->d_gq, P.g.size()));
        c->gq_cap = P.g.size();
    }
    CU(cudaMemcpyAsync(c->d_gq, P.g.data(), sizeof(GemmDesc) * P.g.size(), cudaMemcpyHostToDevice, c->st));
    const bool tc = c->precond && c->oz_s == 7 && !wide;
    const OzScratch scr{static_cast<unsigned char*>(c->d_oz_as), static_cast<unsigned char*>(c->d_oz_bs), c->d_oz_ea,
                        c->d_oz_eb, c->d_oz, c->oz_slot_bytes, oz_exp_ints(c->ld)};
    const unsigned long long timeout_ns = (unsigned long long)c->cfg.barrier_timeout_ms * 1000000ull;
    for (const auto& L : P.launches) {
        if (L.count == 0) continue;
        if (tc)
            CU(launch_gemm_tc(c->d_gq + L.first, L.count, L.max_m, L.max_n, c->ld, scr, 7, timeout_ns, c->st));
        else
            CU(launch_gemm(c->d_gq + L.first, L.count, L.max_m, L.max_n, c->st));
    }
    CU(cudaStreamSynchronize(c->st));   // the host descriptors are rebuilt by the next plan
    return MPDO_OK;
}

// Whether the SVDs of an instance's chi x chi matrices take the stages of a step's SVDs
// (FP32 QR and Jacobi, tensor-core refinement, FP64 Jacobi) in place of the FP64
// Jacobi alone.  FP64 contexts only: a mixed one's products resolve 2^-48.  Below
// 32 rows a matrix is a single block pair of one CTA and the stages' launches cost
// more than its sweeps.
bool staged_svd(const mpdo_ctx* c, int chi) { return refine_on(c) && c->oz_s == 7 && chi >= 32; }

// zero rows and columns from chi up to the next multiple of 4 (the stages' row groups)
__global__ void pad_kernel(double* M, size_t mat, int ld, const int* chi) {
    const int s = blockIdx.x, n = chi[s], n4 = (n + 3) & ~3;
    double* X = M + (size_t)s * mat;
    for (int e = threadIdx.x; e < n4; e += blockDim.x)
        for (int k = n; k < n4; ++k) X[(size_t)e * ld + k] = X[(size_t)k * ld + e] = 0.0;
}

// SVD (strict tolerance, every pair) of the chi x chi matrices in M + slot * mat for
// the listed slots (rows j < chi of length chi), in place; staged: into W + slot * mat,
// the transposed matrices being in MT + slot * mat.
int run_svds(mpdo_ctx* c, double* M, double* MT, bool staged, const std::vector<int>& slots, const std::vector<int>& chis,
             const std::vector<int>& inst) {
    const int ld = c->ld;
    const size_t mat = (size_t)ld * ld;
    const int nops = (int)slots.size();
    if (nops == 0) return MPDO_OK;
    for (int k = 0; k < nops; ++k) {
        OpDesc d{};
        const int s = slots[k], n = staged ? (chis[k] + 3) & ~3 : chis[k];
        d.b = inst[k];
        d.c = n;
        d.L = n;
        d.m = n;
        d.n = n;
        d.chi_max = n;
        if (staged) {
            d.thetap = M + (size_t)s * mat;   // row-major
            d.Acm = MT + (size_t)s * mat;     // column-major
            svd_buffers(c, s, d);
        } else {
            d.W = M + (size_t)s * mat;
            d.W0 = d.W;
        }
        d.snorm = c->d_snorm + (size_t)s * 2 * ld;
        d.status = c->d_status + inst[k];
        d.sweeps_out = c->d_sweeps + s;
        d.full_svd = 1;
        d.jb = jacobi_block_rows(n, n, 8);
        c->h_desc[k] = d;
    }
    CU(cudaMemcpyAsync(c->d_desc, c->h_desc, sizeof(OpDesc) * nops, cudaMemcpyHostToDevice, c->st));
    if (staged) {
        const bool prof = c->prof;   // the stage counters are those of the steps
        c->prof = false;
        SvdWork w;
        const int rc = run_svd(c, nops, 0.0, w);
        c->prof = prof;
        if (rc) return rc;
        CU(cudaStreamSynchronize(c->st));   // h_desc / h_cta are reused by the next call
        return MPDO_OK;
    }
    int total = 0;
    int rc = plan_jacobi(c, c->h_desc, nops, false, c->h_cta, total);
    if (rc) return rc;
    CU(cudaMemcpyAsync(c->d_cta, c->h_cta, sizeof(int) * (2 * total + nops), cudaMemcpyHostToDevice, c->st));
    CU(cudaMemsetAsync(c->d_sync, 0, sizeof(unsigned) * jacobi_sync_words(nops), c->st));
    const unsigned long long timeout_ns = (unsigned long long)c->cfg.barrier_timeout_ms * 1000000ull;
    CU(launch_jacobi(c->d_desc, nops, c->d_cta, c->d_cta + total, c->d_cta + 2 * total, c->d_sync, total,
                     c->cfg.jacobi_max_sweeps, 0.0, timeout_ns, ld, false, c->st));
    CU(cudaStreamSynchronize(c->st));   // h_desc / h_cta are reused by the next call
    return MPDO_OK;
}

int global_prepare(mpdo_ctx* c, double* out) {
    if (!c || !out) return fail(MPDO_EINVAL, "NULL argument");
    CU(cudaSetDevice(c->dev));
    if (!c->built) return fail(MPDO_ESTATE, "mpdo_build_gates must come first");
    if (c->slots < 2) return fail(MPDO_ECAPACITY, "needs at least two workspace slots");
    CU(cudaMemcpyAsync(c->h_dims.data(), c->d_dims, sizeof(int) * c->h_dims.size(), cudaMemcpyDeviceToHost, c->st));
    CU(cudaStreamSynchronize(c->st));
    return refresh_gauge(c);
}

int finish(mpdo_ctx* c, double* out, int out_on_device) {
    if (!out_on_device) {
        CU(cudaMemcpyAsync(out, c->d_out, sizeof(double) * c->B, cudaMemcpyDeviceToHost, c->st));
        CU(cudaStreamSynchronize(c->st));
    }
    return MPDO_OK;
}

}  // namespace

}  // namespace mpdo

extern "C" int mpdo_renyi2(mpdo_ctx* c, double* out, int out_on_device) {
    int rc = global_prepare(c, out);
    if (rc) return rc;
    const int N = c->N, B = c->B;
    const size_t mat = (size_t)c->ld * c->ld;
    double* dst = out_on_device ? out : c->d_out;
    CU(launch_environments(c->d_sites, sites_f32(c), c->d_dims, N, B, c->cap, c->d_envL, c->d_envR, c->st));
    const int per = std::max(1, c->slots / 2);
    for (int b0 = 0; b0 < B; b0 += per) {
        const int m = std::min(per, B - b0);
        gram_unit_kernel<<<(2 * m + 127) / 128, 128, 0, c->st>>>(c->d_Z, mat, m);
        CU(cudaGetLastError());
        for (bool wide : {false, true}) {
            GqPlan P;
            plan_left(c, b0, m, N - 1, wide, P);
            rc = run_plan(c, wide, P);
            if (rc) return rc;
        }
        renyi2_kernel<<<(m + 127) / 128, 128, 0, c->st>>>(c->d_Z, mat, c->d_envL, N, c->cap, b0, m, dst);
        CU(cudaGetLastError());
    }
    return finish(c, out, out_on_device);
}

extern "C" int mpdo_osee(mpdo_ctx* c, int bond, double* out, int out_on_device) {
    int rc = global_prepare(c, out);
    if (rc) return rc;
    const int N = c->N, B = c->B, ld = c->ld;
    if (bond < 0 || bond > N - 2) return fail(MPDO_EINVAL, "bond must be in [0, N-2]");
    const size_t mat = (size_t)ld * ld;
    double* dst = out_on_device ? out : c->d_out;
    const int per = std::max(1, c->slots / 2);
    int* d_chi = c->d_q;   // [2 m] chi of each slot (ints; N >= 2 m is not guaranteed, so chunk by it too)
    int* d_staged = c->d_q + N;   // [2 m] whether its SVD takes the stages
    const int per_chi = std::max(1, N / 2);
    for (int b0 = 0; b0 < B; b0 += std::min(per, per_chi)) {
        const int m = std::min(std::min(per, per_chi), B - b0);
        gram_unit_kernel<<<(2 * m + 127) / 128, 128, 0, c->st>>>(c->d_Z, mat, m);
        CU(cudaGetLastError());
        for (bool wide : {false, true}) {
            GqPlan P;
            plan_left(c, b0, m, bond, wide, P);
            plan_right(c, b0, m, bond + 1, wide, P);
            rc = run_plan(c, wide, P);
            if (rc) return rc;
        }
        // the instances of each route: [0] the FP64 Jacobi alone, [1] the stages
        std::vector<int> slots[2], chis[2], inst[2], chi2(2 * m), route(2 * m);
        int maxchi = 1;
        for (int i = 0; i < m; ++i) {
            const int b = b0 + i;
            const int chi = c->h_dims[(size_t)b * (N + 1) + bond + 1];
            const int st = staged_svd(c, chi) && !wide_instance(c, b) ? 1 : 0;
            maxchi = std::max(maxchi, chi);
            for (int h = 0; h < 2; ++h) {
                slots[st].push_back(2 * i + h);
                chis[st].push_back(chi);
                inst[st].push_back(b);
                chi2[2 * i + h] = chi;
                route[2 * i + h] = st;
            }
        }
        CU(cudaMemcpyAsync(d_chi, chi2.data(), sizeof(int) * 2 * m, cudaMemcpyHostToDevice, c->st));
        CU(cudaMemcpyAsync(d_staged, route.data(), sizeof(int) * 2 * m, cudaMemcpyHostToDevice, c->st));
        const bool any = !slots[1].empty();
        if (any) {
            pad_kernel<<<2 * m, 256, 0, c->st>>>(c->d_Z, mat, ld, d_chi);
            CU(cudaGetLastError());
        }
        for (int st = 0; st < 2; ++st) {   // X and Y factored: their rows in d_Z, staged in d_W
            rc = run_svds(c, c->d_Z, c->d_Z, st == 1, slots[st], chis[st], inst[st]);
            if (rc) return rc;
        }
        row_norms_kernel<<<dim3((maxchi + 7) / 8, 2 * m), 256, 0, c->st>>>(c->d_Z, c->d_W, mat, ld, d_chi, d_staged,
                                                                           c->d_snorm);
        CU(cudaGetLastError());
        // C_i = (rows of X) (rows of Y)^T into thetap slot 2i, then scaled to F_X F_Y^T
        // (staged: its transpose into slot 2i + 1)
        GqPlan Pc[2];   // [1]: flagged instances
        Pc[0].begin();
        Pc[1].begin();
        for (int s = 0; s < 2 * m; ++s) {
            if ((s & 1) && !route[s]) continue;
            double* F = route[s] ? c->d_W : c->d_Z;
            Pc[wide_instance(c, b0 + s / 2)].add(GemmDesc{chi2[s], chi2[s], chi2[s], F + (size_t)s * mat, ld, 0, F + (size_t)(s ^ 1) * mat, ld, 0,
                            1, c->d_thetap + (size_t)s * mat, ld, 1.0, 0.0, nullptr, 0, 0, 0, 0, 0},
                   c->d_status + b0 + s / 2);
        }
        for (bool wide : {false, true}) {
            rc = run_plan(c, wide, Pc[wide]);
            if (rc) return rc;
        }
        scale_kernel<<<dim3(64, 2 * m), 256, 0, c->st>>>(c->d_thetap, mat, ld, d_chi, d_staged, c->d_snorm);
        CU(cudaGetLastError());
        if (any) {
            pad_kernel<<<2 * m, 256, 0, c->st>>>(c->d_thetap, mat, ld, d_chi);
            CU(cudaGetLastError());
        }
        for (int st = 0; st < 2; ++st) {
            std::vector<int> s1, c1, i1;
            for (size_t k = 0; k < slots[st].size(); k += 2) {
                s1.push_back(slots[st][k]);
                c1.push_back(chis[st][k]);
                i1.push_back(inst[st][k]);
            }
            rc = run_svds(c, c->d_thetap, c->d_thetap + mat, st == 1, s1, c1, i1);
            if (rc) return rc;
        }
        osee_kernel<<<m, 512, 0, c->st>>>(c->d_thetap, c->d_W, mat, ld, d_chi, d_staged, b0, dst);
        CU(cudaGetLastError());
    }
    return finish(c, out, out_on_device);
}

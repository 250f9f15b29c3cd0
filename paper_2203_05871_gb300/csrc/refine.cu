// Finish of the preconditioned SVD: all pairs of rows at once, through their
// Gram matrix.
//
// After the FP32 preconditioning pass and its FP64-accurate application the c
// rows of W are orthogonal to ~1e-6 of their norms.  The FP64 Jacobi sweeps that
// used to finish them read every pair of rows with FP64 FMAs, of which GB300
// issues two per SM and clock.  One iteration here instead
//   1. forms G = W W^T as a tensor-core product (oz_gemm.cu; every row and
//      column scaled by its own exponent, so G_ij is accurate relative to
//      |w_i| |w_j| however graded the rows are),
//   2. takes the Jacobi angle theta_ij of every pair that is not orthogonal to
//      tol, X_ij = -theta_ij (antisymmetric), and
//   3. turns all rows by the rotation W <- P(X) W, P(X) = I + X + X^2/2 + X^3/8.
// P(X) P(X)^T = I - X^6/64 + ..., and with the terms through X^2 or X only it is
// I + X^4/4 or I - X^2: each iteration takes the fewest terms whose defect is
// below its tolerance.  The residual after an iteration is of second order
// (angle times off-orthogonality), so two iterations finish a typical op.
// In P(X) W the product X W scales column k of X by |w_k| and row k of W by its
// inverse (exponents only), so a row is accurate relative to its own norm.
//
// An op ends in state kRefineDone when a Gram matrix shows every needed pair at
// tol, or when the predicted residual is under a tenth of it; the FP64 Jacobi
// pass then returns at once.  Everything the expansion does not cover (a pair
// whose angle is too large: nearly equal singular values that are not yet
// separated; a non-finite entry) leaves the op to the Jacobi pass, which starts
// from the rows as they are.  Needed pairs, zero rows and tol are the Jacobi
// pass's (jacobi.cu): two rows that the truncation discards need not be
// orthogonal to one another, a row of norm <= eps |W|_F is set to zero.
#include <float.h>
#include <mpdo.h>

#include "coop.cuh"
#include "internal.h"

namespace mpdo {

namespace {

constexpr int NT = 256;

// squared row norms and their inverse roots from G's diagonal, the zero floor
// (rows at or under it are set to zero) and the discard threshold, fixed once open
__global__ void __launch_bounds__(NT) refine_diag_kernel(const OpDesc* descs, int ld) {
    grid_begin();
    const OpDesc& d = descs[blockIdx.x];
    RefineOp& r = *d.rf;
    if (d.plain) return;
    if (r.state != kRefineActive) {
        if (threadIdx.x == 0) r.order = r.turn = 0;   // no rotation in this iteration
        return;
    }
    const int c = d.c;
    double* a = d.snorm;
    double* inv = d.snorm + ld;
    __shared__ double red[NT / 32], s_floor2;
    double f = 0.0;
    for (int i = threadIdx.x; i < c; i += NT) {
        const double v = d.E[(size_t)i * ld + i];
        a[i] = v;
        f += v;
    }
    f = warp_sum(f);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = f;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < NT / 32; ++w) t += red[w];
        s_floor2 = DBL_EPSILON * DBL_EPSILON * t;
    }
    __syncthreads();
    const double floor2 = s_floor2;
    for (int i = threadIdx.x; i < c; i += NT) inv[i] = a[i] > floor2 ? 1.0 / sqrt(a[i]) : 0.0;
    for (int i = threadIdx.x; i < c; i += NT)
        if (a[i] <= floor2 && a[i] != 0.0)   // rare: numerically zero rows
            for (int k = 0; k < d.L; ++k) d.W[(size_t)i * ld + k] = 0.0;
    const int kk = d.chi_max + max(16, d.chi_max / 8);
    const bool settled = r.order > 0 ? __uint_as_float(r.rho2) <= 1e-8f : (d.pre_ok && *d.pre_ok == 1);
    double thr = r.thr;
    __syncthreads();
    if (thr == 0.0 && settled && !d.full_svd && kk < c) thr = kth_largest<NT, 4 * kMaxChi>(a, c, kk);
    if (threadIdx.x == 0) {
        r.thr = thr;
        r.need = fmax(thr, cutoff_floor(d, floor2 / (DBL_EPSILON * DBL_EPSILON)));
        r.floor2 = floor2;
        r.rho2 = 0u;
        r.row1 = 0u;
        r.far = 0;
        r.blocks = 0u;
    }
}

// scratch of the pairing, in the FP32 pass's Gram blocks: the row each row chose (-1: none)
// and the tangent of its angle
__device__ __forceinline__ int* partner_of(const OpDesc& d) { return reinterpret_cast<int*>(d.D32); }
__device__ __forceinline__ float* angle_of(const OpDesc& d, int ld) { return d.D32 + ld; }

// The op's state and the order of this iteration's rotation.
__device__ void decide(const OpDesc& d, RefineOp& r, double tol_in, int can_finish, float defect, int last, int turn) {
    r.order = 0;
    if (d.sweeps_out) *d.sweeps_out += 1;
    const float tol = (float)(tol_in > 0.0 ? tol_in : sqrt((double)d.L) * DBL_EPSILON);
    const float rho = sqrtf(__uint_as_float(__ldcg(&r.rho2))), x = __uint_as_float(__ldcg(&r.row1));
    if (rho <= tol) {
        r.state = can_finish ? kRefineDone : kRefineLeft;
        return;
    }
    const float x2 = x * x;
    if (x2 <= defect)
        r.order = 1;
    else if (0.25f * x2 * x2 <= defect)
        r.order = 2;
    else if (x2 * x2 * x2 <= 64.0f * defect)
        r.order = 3;
    else {
        if (!turn) r.state = kRefineLeft;   // beyond the expansion (or not finite)
        if (last) r.state = kRefineLeft;
        return;
    }
    if (!__ldcg(&r.far) && 2.0f * rho * x <= 0.1f * tol)
        r.state = can_finish ? kRefineDone : kRefineLeft;   // after this rotation
    else if (last)
        r.state = kRefineLeft;
}

// X from G, one warp per row; the largest g^2 / (a b) of a needed pair, the
// largest absolute row sum of X (a bound of its norm), and whether an angle
// was too large for the expansion.  The op's last CTA to finish decides.
__global__ void __launch_bounds__(NT) refine_x_kernel(const OpDesc* descs, int ld, double tol_in, float tcap,
                                                      int can_finish, float defect, int last) {
    grid_begin();
    const OpDesc& d = descs[blockIdx.y];
    RefineOp& r = *d.rf;
    const int i = blockIdx.x * (NT / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int blocks = (d.c + NT / 32 - 1) / (NT / 32);
    if ((int)blockIdx.x >= blocks || d.plain || __ldcg(&r.state) != kRefineActive) return;
    if (i < d.c) {
        const float tol = (float)(tol_in > 0.0 ? tol_in : sqrt((double)d.L) * DBL_EPSILON);
        // pairs within a tolerance well above the Gram matrix's own error are turned too,
        // down to 1/100 of it, where that takes an angle of the tolerance's size (1000 of
        // them add 4e-14 to the rotation's defect): it costs nothing and leaves the rows'
        // errors far below the tolerance (a chi 256 step's: 3e-10 without, 1e-11 with it)
        const float turn = tol >= 1e-11f ? 0.01f * tol : tol;
        const double* a = d.snorm;
        const double* inv = d.snorm + ld;
        const double ai = a[i], vi = inv[i], thr = r.need;
        const bool dead = vi == 0.0, low = ai < thr;
        float rho = 0.0f, sum = 0.0f, tfar = 0.0f;
        int far = 0;
        unsigned long long best = 0;   // of the pairs beyond tcap: |t|, then the smallest pair of rows
        for (int j = lane; j < d.c; j += 32) {
            const double aj = a[j], vj = inv[j];
            double x = 0.0;
            if (j != i && !dead && vj != 0.0 && !(low && aj < thr)) {
                const double v = vi * vj;
                const float q = (float)(d.E[(size_t)i * ld + j] * v);   // g / (|w_i| |w_j|)
                rho = !(fabsf(q) <= rho) ? fabsf(q) : rho;              // a NaN stays
                if (fabsf(q) > turn) {
                    const float zeta = (float)((aj - ai) * v) / (2.0f * q);
                    const float t = fabsf(zeta) > 1e18f   // a row far below the other (zeta^2 leaves FP32's range)
                                        ? 0.5f / zeta
                                        : copysignf(1.0f, zeta) / (fabsf(zeta) + sqrtf(fmaf(zeta, zeta, 1.0f)));
                    const bool small = fabsf(q) <= tol;
                    if (fabsf(t) <= (small ? 2.0f * tol : tcap)) {
                        const float th = t * fmaf(-t * t, 1.0f / 3.0f, 1.0f);   // atan t
                        x = -(double)th;
                        if (!small) sum += fabsf(th);
                    } else if (!small) {
                        far = 1;
                        const unsigned pair = ((unsigned)min(i, j) << 16) | (unsigned)max(i, j);
                        const unsigned long long key =
                            ((unsigned long long)__float_as_uint(fabsf(t)) << 32) | (0xffffffffu - pair);
                        if (key > best) {
                            best = key;
                            tfar = t;
                        }
                    }
                }
            }
            d.Q[(size_t)i * ld + j] = x;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float v = __shfl_xor_sync(0xffffffffu, rho, o);
            rho = !(v <= rho) ? v : rho;
        }
        sum = warp_sum(sum);
        far = __any_sync(0xffffffffu, far);
        if (far) {
            unsigned long long top = best;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long v = __shfl_xor_sync(0xffffffffu, top, o);
                top = v > top ? v : top;
            }
            if (best == top) {   // pairs are unique: one lane
                const unsigned pair = 0xffffffffu - (unsigned)top;
                __stcg(partner_of(d) + i, (int)((pair >> 16) == (unsigned)i ? pair & 0xffffu : pair >> 16));
                __stcg(angle_of(d, ld) + i, tfar);
            }
        } else if (lane == 0) {
            __stcg(partner_of(d) + i, -1);
        }
        if (lane == 0) {
            atomicMax(&r.rho2, __float_as_uint(fabsf(rho * rho)));
            atomicMax(&r.row1, __float_as_uint(sum));
            if (far) atomicOr(&r.far, 1);
        }
    }
    __threadfence();
    __syncthreads();
    __shared__ int s_last, s_turn;
    if (threadIdx.x == 0) {
        s_last = atomicAdd(&r.blocks, 1u) == (unsigned)blocks - 1u;
        s_turn = 0;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // Rows that chose one another are turned by their exact rotation (refine_turn_kernel)
    // and take no other part in this iteration.
    __shared__ unsigned mate[4 * kMaxChi / 32];
    const bool any = __ldcg(&r.far) != 0;
    if (any) {
        int* partner = partner_of(d);
        for (int w = threadIdx.x; w < 4 * kMaxChi / 32; w += NT) mate[w] = 0;
        __syncthreads();
        for (int k = threadIdx.x; k < d.c; k += NT) {
            const int j = __ldcg(partner + k);
            if (j >= 0 && __ldcg(partner + j) == k) {
                atomicOr(&mate[k >> 5], 1u << (k & 31));
                s_turn = 1;
            }
        }
        __syncthreads();
        for (int k = threadIdx.x >> 5; k < d.c; k += NT / 32) {
            if ((mate[k >> 5] >> (k & 31)) & 1u) {
                for (int j = lane; j < d.c; j += 32) d.Q[(size_t)k * ld + j] = d.Q[(size_t)j * ld + k] = 0.0;
            } else if (lane == 0) {
                __stcg(partner + k, -1);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        decide(d, r, tol_in, can_finish, defect, last, s_turn);
        r.turn = s_turn && r.state == kRefineActive;
    }
}

// The exact rotations of the rows that refine_x_kernel paired, one pair per warp: rows
// of nearly equal norm that are not yet orthogonal, whose angle is beyond the
// expansion.  Left to the FP64 Jacobi pass, a few of them cost an op whole sweeps over
// all of its pairs (a quarter of the time of a 3 x 3 grid's evolution).
__global__ void __launch_bounds__(NT) refine_turn_kernel(const OpDesc* descs, int ld) {
    grid_begin();
    const OpDesc& d = descs[blockIdx.y];
    if (d.plain || !d.rf->turn) return;
    const int i = blockIdx.x * (NT / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= d.c) return;
    const int j = partner_of(d)[i];
    if (j <= i) return;
    const double t = (double)angle_of(d, ld)[i], cs = 1.0 / sqrt(fma(t, t, 1.0)), sn = cs * t;
    for (int part = 0; part < (d.transposed ? 2 : 1); ++part) {
        double* p = (part ? d.Z : d.W) + (size_t)i * ld;
        double* q = (part ? d.Z : d.W) + (size_t)j * ld;
        const int len = part ? d.c : d.L;
        for (int k = lane; k < len; k += 32) {
            const double x = p[k], y = q[k];
            p[k] = cs * x - sn * y;
            q[k] = sn * x + cs * y;
        }
    }
}

}  // namespace

cudaError_t launch_refine(const OpDesc* d_desc, int nops, int chi_cap, int S, bool with_z, double tol_in,
                          bool can_finish, unsigned long long timeout_ns, cudaStream_t st) {
    if (nops <= 0) return cudaSuccess;
    const int ld = 4 * chi_cap;
    // defect of the rotation's orthogonality: FP64 rounding with 7 slices, the
    // level of 6 slices' products otherwise; the largest single angle follows
    const float defect = S == 7 ? 1e-17f : 1e-13f, tcap = S == 7 ? 2e-3f : 1e-2f;
    for (int it = 0; it < kRefineIters; ++it) {
        cudaError_t e = launch_oz_ops(d_desc, nops, OZ_G, chi_cap, S, false, timeout_ns, st);
        if (e != cudaSuccess) return e;
        if ((e = launch_early(refine_diag_kernel, nops, NT, 0, st, d_desc, ld)) != cudaSuccess) return e;
        e = launch_early(refine_x_kernel, dim3((ld + NT / 32 - 1) / (NT / 32), nops), NT, 0, st, d_desc, ld, tol_in,
                         tcap, can_finish ? 1 : 0, defect, it == kRefineIters - 1);
        if (e != cudaSuccess) return e;
        e = launch_early(refine_turn_kernel, dim3((ld + NT / 32 - 1) / (NT / 32), nops), NT, 0, st, d_desc, ld);
        if (e != cudaSuccess) return e;
        for (int kind : {OZ_R3, OZ_R2, OZ_R1})
            if ((e = launch_oz_ops(d_desc, nops, kind, chi_cap, S, with_z, timeout_ns, st)) != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

}  // namespace mpdo

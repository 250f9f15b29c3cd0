// FP64 one-sided (Hestenes) Jacobi SVD of the bond matrices of one layer.
//
// App. B compresses |rho>> bond by bond from its Schmidt spectrum.  Each op
// hands this kernel c rows of length L (those of theta~ or of R, or of theta~^T when
// m > n, then with the c x c rotations so far, Z, whose rows turn alongside).  Plane rotations from the left make the rows mutually
// orthogonal; row j then equals s_j v_j^T (or Z row j = v_j^T), which the
// truncation step reads.
//
// Block-pair ordering.  The rows are cut into blocks of b rows (b chosen so
// that two blocks, with their Z parts, fit in 128 KB of shared memory).  A
// round-robin ("circle") tournament over the blocks meets every pair of
// blocks once per sweep; in a round each CTA loads one or more block pairs
// into shared memory, rotates every cross pair of rows (and, in the first
// round of a sweep, every pair inside each block), and stores the blocks back
// to their home rows.  The op's CTAs take the block pairs of a sweep from a
// shared counter in round order, and a pair waits only for its two blocks to
// leave the previous round (a version per block); one barrier per sweep.
// Every wait is bounded by a wall-clock limit after which the kernel records
// MPDO_ST_TIMEOUT and returns.  The launch is cooperative (all CTAs resident).
// Within a block pair one warp owns one pair of rows: the inner product is
// reduced with warp shuffles, the rotation is applied in shared memory.
//
// Rotation (Rutishauser): a = |w_p|^2, b = |w_q|^2, g = w_p.w_q,
// zeta = (b - a) / 2g, t = sign(zeta) / (|zeta| + sqrt(1 + zeta^2)),
// cs = 1/sqrt(1+t^2), sn = cs t;  w_p <- cs w_p - sn w_q, w_q <- sn w_p + cs w_q,
// and then |w_p|^2 = a - t g, |w_q|^2 = b + t g (recomputed from the row when
// the update loses more than 90% of the old value, and at every sweep start).
// A pair is skipped when |g| <= tol sqrt(a b) (tol = sqrt(L) eps unless set):
// kept rows are normalised into singular vectors, so they must be orthogonal
// relative to their own norms.
//
// After the FP32 pass (jacobi32.cu) and the refinement through the Gram matrix
// (refine.cu) most ops arrive finished and their CTAs return at once; what is
// left is what those stages do not cover, and every SVD of contexts whose sweep
// limit leaves them out.  A row whose norm is at most eps * ||W||_F (FP64 eps, in
// every stage) is numerically zero: it is set to zero and never rotated (its
// direction is rounding noise).
//
// Further pieces, each described where it is implemented:
//  - scaled (fast) rotations, one FMA per element (scaled_rotate);
//  - pairs of two rows the truncation discards are skipped once the ranking is
//    settled (kth_largest and the sweep-start gate);
//  - convergence: no rotation or a largest rotated rho with rho^2 <= 1e-6 tol
//    (the FP32 pass: <= c/4 rotations or a largest rotated off-orthogonality of
//    1e-3).
#include <float.h>
#include <mpdo.h>

#include "coop.cuh"
#include "internal.h"

namespace mpdo {

namespace {

constexpr int kWarps = 8;   // blocks of 8 rows (L = 1024) feed 8 warps
constexpr int kThreads = kWarps * 32;
constexpr int kRowBytes = kJacobiRowBytes;             // two blocks of rows in shared memory
constexpr int kMaxB = kJacobiMaxB;
constexpr int kSmemBytes = kRowBytes + 6 * kMaxB * 8;  // rows + norms (2b) + scales (2b) + row ids

constexpr double kScaleFloor = 0x1p-32;   // FP64 row scales below this are multiplied into the row

// <x, y> over L elements: lane-strided with four independent accumulators
// (shared-memory latency is hidden by ILP: one CTA of 8 warps per SM)
__device__ __forceinline__ double row_dot(const double* x, const double* y, int L, int lane) {
    double s0 = 0, s1 = 0, s2 = 0, s3 = 0;
    int i = lane;
    for (; i + 96 < L; i += 128) {
        const double x0 = x[i], x1 = x[i + 32], x2 = x[i + 64], x3 = x[i + 96];
        const double y0 = y[i], y1 = y[i + 32], y2 = y[i + 64], y3 = y[i + 96];
        s0 = fma(x0, y0, s0);
        s1 = fma(x1, y1, s1);
        s2 = fma(x2, y2, s2);
        s3 = fma(x3, y3, s3);
    }
    for (; i < L; i += 32) s0 = fma(x[i], y[i], s0);
    return warp_sum((s0 + s1) + (s2 + s3));
}

struct Ctx {
    double* rows;     // [2b][rowlen] in shared memory
    double* nrm;      // [2b]
    double* dsc;      // [2b] the row is dsc times the stored row (scaled rotations)
    int* rid;         // [2b] global row index or -1
    unsigned* rho2;   // largest g^2 / (a b) rotated in this CTA and sweep (float bits)
    int rowlen, L;    // row length in smem (W part + Z part), W part length
    double floor2, tol;
    double thr;       // pairs of rows whose squared norms are both below thr are skipped
};

// Rotation parameters (cs, sn, t) zeroing <w_p, w_q> = g for |w_p|^2 = a,
// |w_q|^2 = b.  FP64: t is found in FP32 (an inexact angle only slows the
// last digits of convergence), cs = 1/sqrt(1+t^2) is then refined by two
// Newton steps in FP64 so that cs^2 + sn^2 = 1 to FP64 rounding: the rotation
// applied to the rows is orthogonal in FP64.  FP32: computed directly.
__device__ __forceinline__ void rot_params(double a, double b, double g, double& cs, double& sn, double& t) {
    const double r = b - a;
    // scale (r, g) by a power of two so that both fit FP32's range
    const double m = fmax(fabs(r), fabs(g));
    int e = (int)((__double_as_longlong(m) >> 52) & 0x7ff) - 1023;
    e = e < -1022 ? -1022 : (e > 1022 ? 1022 : e);
    const double sc = __longlong_as_double((long long)(1023 - e) << 52);
    const float rf = (float)(r * sc), gf = (float)(g * sc);
    const float zeta = rf / (2.0f * gf);
    float tf;
    if (fabsf(zeta) > 1e18f)
        tf = 0.5f / zeta;
    else
        tf = copysignf(1.0f, zeta) / (fabsf(zeta) + sqrtf(1.0f + zeta * zeta));
    t = (double)tf;
    const double q = fma(t, t, 1.0);
    double c = (double)rsqrtf((float)q);
    c = c * fma(-0.5 * q, c * c, 1.5);
    c = c * fma(-0.5 * q, c * c, 1.5);
    cs = c;
    sn = c * t;
}

// FP64 rotation on scaled rows (fast plane rotation with dynamic scaling,
// Anda & Park 1994): the rows are w_p = d_p x_p, w_q = d_q x_q, and
//   w_p' = cs w_p - sn w_q = (cs d_p) (x_p - t (d_q / d_p) x_q),
//   w_q' = sn w_p + cs w_q = (cs d_q) (x_q + t (d_p / d_q) x_p),
// so the stored rows take one FMA per element and the factor cs goes to the
// scales.  |t| <= 1, so a scale shrinks by at most 1/sqrt(2) per rotation; a
// scale below 2^-32 is multiplied into its row.  The kernel multiplies every
// row by its scale after the last sweep.
__device__ int scaled_rotate(const Ctx& C, int p, int q, double* rp, double* rq, double a, double b, double g, double cs,
                             double t, double dp, double dq, int lane) {
    const double al = t * (dq / dp), be = t * (dp / dq);
    int i = lane;
    for (; i + 96 < C.rowlen; i += 128) {
        double x[4], y[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            x[u] = rp[i + 32 * u];
            y[u] = rq[i + 32 * u];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            rp[i + 32 * u] = fma(-al, y[u], x[u]);
            rq[i + 32 * u] = fma(be, x[u], y[u]);
        }
    }
    for (; i < C.rowlen; i += 32) {
        const double x = rp[i], y = rq[i];
        rp[i] = fma(-al, y, x);
        rq[i] = fma(be, x, y);
    }
    __syncwarp();
    dp *= cs;
    dq *= cs;
    double na = fma(-t, g, a), nb = fma(t, g, b);
    if (na < 0.1 * a) na = dp * dp * row_dot(rp, rp, C.L, lane);
    if (nb < 0.1 * b) nb = dq * dq * row_dot(rq, rq, C.L, lane);
    if (dp < kScaleFloor) {
        for (int k = lane; k < C.rowlen; k += 32) rp[k] *= dp;
        dp = 1.0;
    }
    if (dq < kScaleFloor) {
        for (int k = lane; k < C.rowlen; k += 32) rq[k] *= dq;
        dq = 1.0;
    }
    __syncwarp();
    if (lane == 0) {
        C.nrm[p] = na;
        C.nrm[q] = nb;
        C.dsc[p] = dp;
        C.dsc[q] = dq;
    }
    __syncwarp();
    return 1;
}

// One warp: rows p, q (shared-memory slots).  Returns 1 if it rotated.
__device__ int pair_rotate(const Ctx& C, int p, int q, int lane) {
    if (C.rid[p] < 0 || C.rid[q] < 0) return 0;
    if (C.nrm[p] < C.thr && C.nrm[q] < C.thr) return 0;   // two rows the truncation discards
    double* rp = C.rows + (size_t)p * C.rowlen;
    double* rq = C.rows + (size_t)q * C.rowlen;
    const double a = C.nrm[p], b = C.nrm[q];
    if (a <= C.floor2 || b <= C.floor2) {
        if (a <= C.floor2 && a != 0.0) {
            for (int i = lane; i < C.L; i += 32) rp[i] = 0.0;
            __syncwarp();
            if (lane == 0) C.nrm[p] = 0.0;
        }
        if (b <= C.floor2 && b != 0.0) {
            for (int i = lane; i < C.L; i += 32) rq[i] = 0.0;
            __syncwarp();
            if (lane == 0) C.nrm[q] = 0.0;
        }
        __syncwarp();
        return 0;
    }
    double g = row_dot(rp, rq, C.L, lane);
    g *= C.dsc[p] * C.dsc[q];
    if (g == 0.0 || g * g <= C.tol * C.tol * a * b) return 0;
    double cs, sn, t;
    rot_params(a, b, g, cs, sn, t);
    if (t == 0.0) return 0;
    if (lane == 0) atomicMax(C.rho2, __float_as_uint((float)(g / a * (g / b))));
    return scaled_rotate(C, p, q, rp, rq, a, b, g, cs, t, C.dsc[p], C.dsc[q], lane);
}

// All pairs inside each of the two blocks (circle method, first round of a
// sweep only), then all cross pairs between the two blocks.
__device__ int process_block_pair(const Ctx& C, int b, bool intra, int warp, int lane) {
    int rot = 0;
    if (intra && b > 1) {
        const int bp = b + (b & 1);
        for (int t = 0; t < bp - 1; ++t) {
            for (int x = warp; x < bp; x += kWarps) {   // x < bp/2: block 0, else block 1
                const int blk = x < bp / 2 ? 0 : 1;
                const int y = x % (bp / 2);
                const int P = tour_player(y, t, bp), Q = tour_player(bp - 1 - y, t, bp);
                if (P >= b || Q >= b) continue;
                rot += pair_rotate(C, blk * b + min(P, Q), blk * b + max(P, Q), lane);
            }
            __syncthreads();
        }
    }
    for (int t = 0; t < b; ++t) {
        for (int i = warp; i < b; i += kWarps) rot += pair_rotate(C, i, b + (i + t) % b, lane);
        __syncthreads();
    }
    return rot;
}

__global__ void __launch_bounds__(kThreads, 1) jacobi_kernel(const OpDesc* descs, const int* cta_op, const int* cta_rank,
                                                       const int* group, unsigned* sync, int max_sweeps,
                                                       double tol_in, unsigned long long timeout_ns, int ld) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int op = cta_op[blockIdx.x];
    if (op < 0) return;   // a CTA the plan left unused (graph step)
    const int g = cta_rank[blockIdx.x];
    const int G = group[op];
    const OpDesc& d = descs[op];
    if (d.rf && !d.plain && d.rf->state == kRefineDone) return;   // finished by the refinement (refine.cu)
    unsigned* sw = sync + (size_t)op * kSyncWords;
    const int c = d.c, L = d.L;
    const int b = d.jb;
    double* W = d.W;
    double* Z = d.transposed ? d.Z : nullptr;
    const int zl = Z ? c : 0;
    // a block size that does not fit shared memory is a planning error: every
    // CTA of the op sees it and returns at once
    if (b < 1 || b > kMaxB || (size_t)2 * b * (L + zl) * sizeof(double) > (size_t)kRowBytes) {
        if (threadIdx.x == 0) atomicOr(d.status, (int)MPDO_ST_CAPACITY);
        return;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned gen = 0;
    __shared__ double s_floor2, s_red[kWarps];
    __shared__ int s_conv, s_settled;
    __shared__ unsigned s_rho2;
    __shared__ int s_pair;

    Ctx C;
    C.rowlen = L + zl;
    C.L = L;
    C.rows = reinterpret_cast<double*>(smem_raw);
    C.nrm = reinterpret_cast<double*>(smem_raw + kRowBytes);
    C.dsc = reinterpret_cast<double*>(C.nrm + 2 * b);
    C.rid = reinterpret_cast<int*>(C.dsc + 2 * b);
    double* dscale = d.snorm + ld;   // per-row scales (the QR's column norms are dead here)
    C.rho2 = &s_rho2;
    C.thr = 0.0;
    double kth = 0.0, cut = 0.0;   // cut: cutoff_floor, from the same sweep on (before, rows that are not
                                   // yet orthogonal to one another would draw the rest along sweep by sweep)
    float rho2_stop;
    {
        const double tol = tol_in > 0.0 ? tol_in : sqrt((double)(L > 1 ? L : 1)) * DBL_EPSILON;
        C.tol = tol;
        rho2_stop = (float)(1e-6 * tol);
    }

    // squared row norms (for the zero floor)
    for (int row = g * kWarps + warp; row < c; row += G * kWarps) {
        const double* w = W + (size_t)row * ld;
        double a = 0.0;
        for (int i = lane; i < L; i += 32) {
            const double x = __ldcg(w + i);
            a = fma(x, x, a);
        }
        a = warp_sum(a);
        if (lane == 0) {
            __stcg(d.snorm + row, a);
            __stcg(dscale + row, 1.0);
        }
    }
    if (!op_barrier(sw, G, gen, timeout_ns)) goto timeout;
    {
        double f = 0.0;
        for (int j = threadIdx.x; j < c; j += kThreads) f += __ldcg(d.snorm + j);
        f = warp_sum(f);
        if (lane == 0) s_red[warp] = f;
        __syncthreads();
        if (threadIdx.x == 0) {
            f = 0.0;
            for (int w = 0; w < kWarps; ++w) f += s_red[w];
            s_floor2 = DBL_EPSILON * DBL_EPSILON * f;
        }
        __syncthreads();
    }
    C.floor2 = s_floor2;
    if (!op_barrier(sw, G, gen, timeout_ns)) goto timeout;
    {
        const int nb = (c + b - 1) / b;
        const int nbp = nb + (nb & 1);
        const int npair = nbp / 2;
        const int sweeps = max_sweeps < kMaxSweepsCap ? max_sweeps : kMaxSweepsCap;
        int conv = (c <= 1);
        int used = 0;
        for (int sweep = 0; sweep < sweeps && !conv; ++sweep) {
            int rot = 0;
            if (threadIdx.x == 0) s_rho2 = 0u;
            // fresh squared row norms, then the tail threshold (same in every CTA)
            for (int row = g * kWarps + warp; row < c; row += G * kWarps) {
                const double* w = W + (size_t)row * ld;
                double a = 0;
                for (int i = lane; i < L; i += 32) {
                    const double x = __ldcg(w + i);
                    a = fma(x, x, a);
                }
                a = warp_sum(a);
                const double dv = __ldcg(dscale + row);
                if (lane == 0) __stcg(d.snorm + row, a * dv * dv);
            }
            if (!op_barrier(sw, G, gen, timeout_ns)) goto timeout;
            // Rows the truncation discards (below the chi_max + max(16, chi_max / 8)
            // largest) must end orthogonal to the kept rows, not to one another:
            // the kept rows are then exact singular vectors, the discarded weight
            // is the sum of the discarded rows' squared norms (a trace), and
            // rows already orthogonal to ~1e-4 have norms equal to their singular
            // values to ~1e-8, far finer than the margin.  So once the previous
            // sweep rotated by at most 1e-4, pairs of two discarded rows are skipped.
            // The first sweep after the FP32 preconditioner qualifies too when that
            // pass ended by its off-orthogonality rule (every pair at ~1e-6 then).
            if (threadIdx.x == 0) {
                const int kk = d.chi_max + max(16, d.chi_max / 8);
                const bool settled = sweep > 0
                                         ? __uint_as_float(ld_acquire(&sw[8 + kMaxSweepsCap + sweep - 1])) <= 1e-8f
                                         : (d.pre_ok && !d.plain && __ldcg(d.pre_ok) == 1);
                s_conv = settled && !d.full_svd && kk < c;
                s_settled = settled;
            }
            __syncthreads();
            // the threshold is fixed when the gate first opens, so that a row
            // near it keeps its side (a row changing side later would bring its
            // unprocessed pairs back and cost another sweep)
            // (every CTA reads all norms, so a barrier before a pair of this sweep changes them)
            if (s_conv && kth == 0.0) {
                kth = kth_largest<kThreads, 4 * kMaxChi>(d.snorm, c, d.chi_max + max(16, d.chi_max / 8));
                if (!op_barrier(sw, G, gen, timeout_ns)) goto timeout;
            }
            if (s_settled) cut = cutoff_floor(d, s_floor2 / (DBL_EPSILON * DBL_EPSILON));
            C.thr = fmax(kth, cut);
            __syncthreads();
            // The block pairs of a sweep go to the op's CTAs through a shared
            // counter (position q: round q / npair, pair q % npair), and a round
            // has no barrier: a pair waits only until its two blocks have left
            // the previous round (a version per block).  A CTA whose pairs are
            // cheap (both blocks discarded, or already orthogonal) takes more of
            // them, and a round starts where its blocks are ready.  Positions are
            // taken in order, so the pairs a CTA waits for are held by CTAs that
            // can progress.  Two counters alternate by sweep; the next one is
            // cleared during this sweep (every CTA is past its last use).
            if (g == 0 && threadIdx.x == 0) atomicExch(&sw[kSwQueue + ((sweep + 1) & 1)], 0u);
            for (;;) {
                if (threadIdx.x == 0) s_pair = (int)atomicAdd(&sw[kSwQueue + (sweep & 1)], 1u);
                __syncthreads();
                const int qpos = s_pair;
                __syncthreads();   // read by all before thread 0 takes the next one
                if (qpos >= (nbp - 1) * npair) break;
                const int r = qpos / npair, i = qpos % npair;
                const int P = tour_player(i, r, nbp), Q = tour_player(nbp - 1 - i, r, nbp);
                const unsigned R = (unsigned)(sweep * (nbp - 1) + r);   // rounds of this launch before
                if (threadIdx.x == 0) s_conv = wait_blocks(sw + kSwVer, P, Q, nb, R, &sw[1], timeout_ns);
                __syncthreads();
                if (!s_conv) goto timeout;
                const int bl[2] = {P < Q ? P : Q, P < Q ? Q : P};
                do {
                    {   // both blocks discarded: nothing to do
                        int pred = 1;
                        if (threadIdx.x < 2 * b) {
                            const int blk = bl[threadIdx.x / b];
                            const int row = blk * b + (threadIdx.x % b);
                            if (blk < nb && row < c) pred = __ldcg(d.snorm + row) < C.thr;
                        }
                        if (__syncthreads_and(pred)) break;
                    }
                    // load the two blocks (slot s < b: block bl[0]; s >= b: block bl[1])
                    for (int s = warp; s < 2 * b; s += kWarps) {
                        const int blk = bl[s / b];
                        const int row = blk * b + (s % b);
                        const bool ok = blk < nb && row < c;
                        double* dst = C.rows + (size_t)s * C.rowlen;
                        if (ok) {
                            const double* w = W + (size_t)row * ld;
                            for (int k = lane; k < L; k += 32) dst[k] = __ldcg(w + k);
                            if (zl)
                                for (int k = lane; k < c; k += 32) dst[L + k] = __ldcg(Z + (size_t)row * ld + k);
                            __syncwarp();
                            const double nv = (double)__ldcg(d.snorm + row);
                            if (lane == 0) {
                                C.nrm[s] = nv;
                                C.dsc[s] = __ldcg(dscale + row);
                                C.rid[s] = row;
                            }
                        } else if (lane == 0) {
                            C.nrm[s] = 0.0;
                            C.dsc[s] = 1.0;
                            C.rid[s] = -1;
                        }
                    }
                    __syncthreads();
                    rot += process_block_pair(C, b, r == 0, warp, lane);
                    // store back
                    for (int s = warp; s < 2 * b; s += kWarps) {
                        const int row = C.rid[s];
                        if (row < 0) continue;
                        const double* src = C.rows + (size_t)s * C.rowlen;
                        double* w = W + (size_t)row * ld;
                        for (int k = lane; k < L; k += 32) __stcg(w + k, src[k]);
                        if (zl)
                            for (int k = lane; k < c; k += 32) __stcg(Z + (size_t)row * ld + k, src[L + k]);
                        if (lane == 0) {
                            __stcg(d.snorm + row, (double)C.nrm[s]);
                            __stcg(dscale + row, C.dsc[s]);
                        }
                    }
                    __syncthreads();
                } while (false);
                // the pair's rows are stored: its blocks leave round r
                __threadfence();
                __syncthreads();
                if (threadIdx.x == 0) {
                    if (P < nb) st_release(&sw[kSwVer + P], R + 1);
                    if (Q < nb) st_release(&sw[kSwVer + Q], R + 1);
                }
            }
            if (lane == 0 && rot > 0) atomicAdd(&sw[8 + sweep], (unsigned)rot);
            __syncthreads();
            if (threadIdx.x == 0 && s_rho2) atomicMax(&sw[8 + kMaxSweepsCap + sweep], s_rho2);
            if (!op_barrier(sw, G, gen, timeout_ns)) goto timeout;
            // done: no rotation, or the largest rotated rho had rho^2 <= 1e-6 tol: by
            // quadratic convergence the next sweep would meet pairs at ~rho^2, far
            // under tol, and rotate nothing (1e-20 for tol = sqrt(L) eps at L = 1024)
            if (threadIdx.x == 0)
                s_conv = ld_acquire(&sw[8 + sweep]) == 0u ||
                         __uint_as_float(ld_acquire(&sw[8 + kMaxSweepsCap + sweep])) <= rho2_stop;
            __syncthreads();
            conv = s_conv;
            used = sweep + 1;
        }
        // rows out of their scales (the last round ended with a barrier)
        for (int row = g * kWarps + warp; row < c; row += G * kWarps) {
            const double dv = __ldcg(dscale + row);
            if (dv == 1.0) continue;
            double* w = W + (size_t)row * ld;
            for (int i = lane; i < L; i += 32) __stcg(w + i, __ldcg(w + i) * dv);
            if (Z)
                for (int i = lane; i < c; i += 32) __stcg(Z + (size_t)row * ld + i, __ldcg(Z + (size_t)row * ld + i) * dv);
        }
        if (g == 0 && threadIdx.x == 0) {
            if (d.sweeps_out) *d.sweeps_out += used;
            if (!conv) atomicOr(d.status, (int)MPDO_ST_NOCONV);
        }
    }
    return;
timeout:
    if (threadIdx.x == 0) atomicOr(d.status, (int)MPDO_ST_TIMEOUT);
}

}  // namespace

size_t jacobi_sync_words_per_op() { return kSyncWords; }
size_t jacobi_sync_words(int nops) { return (size_t)nops * kSyncWords; }


cudaError_t jacobi_max_resident(int* blocks) {
    int dev = 0, sms = 0, per64 = 0, per32 = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(jacobi_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes)) != cudaSuccess)
        return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per64, jacobi_kernel, kThreads, kSmemBytes)) != cudaSuccess)
        return e;
    if ((e = jacobi32_max_resident(&per32)) != cudaSuccess) return e;
    *blocks = sms * (per64 < per32 ? per64 : per32);
    return cudaSuccess;
}

cudaError_t launch_jacobi(const OpDesc* d_desc, int nops, const int* d_cta_op, const int* d_cta_rank,
                          const int* d_group, unsigned* d_sync, int grid, int max_sweeps, double tol,
                          unsigned long long timeout_ns, int ld, bool fp32, cudaStream_t st, double pre_rho) {
    (void)nops;
    if (fp32)
        return launch_jacobi32(d_desc, d_cta_op, d_cta_rank, d_group, d_sync, grid, max_sweeps, timeout_ns, ld, st,
                               pre_rho);
    if (grid <= 0) return cudaSuccess;
    void* args[] = {(void*)&d_desc, (void*)&d_cta_op, (void*)&d_cta_rank, (void*)&d_group, (void*)&d_sync,
                    (void*)&max_sweeps, (void*)&tol, (void*)&timeout_ns, (void*)&ld};
    return cudaLaunchCooperativeKernel((const void*)jacobi_kernel, dim3(grid), dim3(kThreads), args, kSmemBytes, st);
}

}  // namespace mpdo

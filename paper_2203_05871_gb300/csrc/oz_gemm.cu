// FP64-accurate batched GEMM on the tcgen05 tensor cores (the contractions, the SVD's
// products and, on FP64 contexts, the Gram sweeps of the entropies).
//
//   C = alpha * A B + beta * D  (- I when sub_identity),  A: M x K, B: K x N,
// FP64 (or f32) in and out, computed from exact products of narrow slices of
// the operands (the error-free splitting of Ozaki, Ogita, Oishi & Rump,
// "Error-free transformations of matrix multiplication by using fast routines
// of matrix multiplication and its applications", Numer. Algorithms 59, 2012):
//
// 1. Slicing (oz_slice_kernel).  Each row i of A is scaled by 2^-e_i, e_i the
//    binary exponent of its largest |A_ik| (so |a| < 1), rounded to the
//    integer X = round(2^47 a) and cut into S = 6 balanced base-256 digits,
//    a ~ 2^-7 sum_t sigma_t 2^-8t with integers |sigma_t| <= 128; a slice
//    keeps 8 significant bits, so it is exact in bf16, and it is stored as
//    sigma_t 2^-8t.  B is cut the same way per column j (exponent f_j).  The
//    rounding error is at most 2^-48 of the row's largest entry.  S = 7 (2^55 a)
//    serves the FP64 path, 2^-56.  (tf32 holds the same digits and gives the same
//    products; it takes twice the bytes and half the MMA rate.  Both tensor
//    precisions are formed from bf16 slices.)
// 2. Products (oz_gemm_kernel).  Every slice pair (t, u) with t + u <= 5 is
//    multiplied on the tensor core: a product sigma_t sigma_u has at most 16
//    bits, so it is exact in FP32, and the sums stay exact while they fit 24
//    bits.  One accumulator per level d = t + u in tensor memory (six), each
//    product already at its own scale 2^-8d through the stored slices.  Every
//    256 values of K the accumulators are drained into FP64 registers: 256
//    products of up to 2^14 fit 2^22, so levels 0 to 3 (at most four pairs,
//    2^24) are summed without any rounding, whatever rounding and alignment
//    the tensor core's FP32 accumulation uses; levels 4 and 5 round at 2^-24
//    of themselves, below 2^-50 of the result.  A drain joins the six levels
//    into one int64 (their exact integer parts) and adds it in FP64.  (Folding levels 3-5 into one
//    accumulator was measured at 2e-12 on the GPU: the accumulator then holds
//    level-3 magnitudes and drops the low bits of every level-5 product at
//    every MMA.)  A product whose result is a small correction (the refinement's
//    X W beside W) forms only the levels that reach the sum (levels).
// 3. Epilogue: C_ij = alpha 2^(e_i + f_j - 14) sum_d L_d + beta D_ij.
// Error: about 2^-46 |A_i|_max |B_j|_max per term of the sum (a numpy model of
// the scheme with per-MMA rounding: 3e-14 of |A_i| |B_j| sqrt(K)), against
// FP64's 2^-53 |A_ik B_kj|: FP64-class accuracy at tensor-core speed.
//
// Data layout.  The slices are written in the tcgen05 canonical K-major,
// no-swizzle layout, pre-tiled: a block of R rows x 64 bytes of K (32 bf16
// values; R = 128 for A, 64 for B) is R x 64 bytes, element (row, k) at
// (row/8)*512 + (k/g)*128 + (row%8)*16 + (k%g)*esize, g = 16/esize (core
// matrices of 8 rows x 16 bytes, LBO = 128 B along K, SBO = 512 B along rows),
// so one cp.async.bulk moves a block into shared memory as it is.  Blocks are
// [slice][row tile][k tile].
//
// Kernel.  One CTA per 128 x 64 tile of C, 320 threads: warp 0 issues the
// bulk copies of the 6 + 6 slice blocks of each k tile into a 3-stage ring
// (72 KB per stage; 7 + 7 blocks: two stages of 84 KB), warp 1 issues the 42 MMAs of a k tile (21 pairs x 2
// instructions of K = 16; M = 128, N = 64) and commits, warps
// 2-9 drain the six accumulators (384 TMEM columns; warp w reads lanes
// 32 (w % 4) .. +31, its half of the 64 columns).  Every wait is bounded by timeout_ns; a wait that
// gives up records MPDO_ST_TIMEOUT in the problem's status word, the other roles
// leave their loops at the next poll, outstanding copies and MMAs are waited
// for (bounded) and the tensor memory is released before the CTA returns.
#include <mpdo.h>

#include <cuda_bf16.h>

#include "internal.h"

namespace mpdo {

namespace {

// S slices per operand (6 or 7): S (S + 1) / 2 slice pairs (t, u) with
// t + u < S, one accumulator per level t + u

constexpr int kTileM = 128;            // rows of A (and of C) per tile
constexpr int kTileN = 64;             // columns of B per slice block
constexpr int kBlockA = kTileM * 64;   // bytes of one slice block of A (8 KB)
constexpr int kBlockB = kTileN * 64;   // of B (4 KB)
// bytes of one k tile of a CTA with TN columns, its stages (up to 210 KB), and shared memory
__host__ __device__ constexpr int stage_bytes(int S, int TN) { return S * (kBlockA + TN * 64); }
__host__ __device__ constexpr int stages_of(int S, int TN) { return 216 * 1024 / stage_bytes(S, TN); }
constexpr int kRangeK = 256;           // K values between accumulator drains
constexpr int kThreads = 320;
__host__ __device__ constexpr int smem_of(int S, int TN) { return stages_of(S, TN) * stage_bytes(S, TN) + 1024; }
__host__ __device__ constexpr int tmem_cols(int S, int TN) {   // a power of two
    return S * TN <= 128 ? 128 : S * TN <= 256 ? 256 : 512;
}
static_assert(7 * kTileN <= 512, "accumulators exceed tensor memory");
static_assert(smem_of(6, 64) <= 227 * 1024 && stages_of(7, 64) >= 2, "the ring in shared memory");
static_assert(kTileM == 128 && kTileN == 64, "oz_set_tiles (internal.h) assumes blocks of 128 and 64 rows");
constexpr int LBO = 128, SBO = 512;

constexpr int G = 8;                   // bf16 values per 16-byte store
constexpr int KT = 32;                 // K values of a block

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
    // start >> 4 (bits 0-13), LBO >> 4 (16-29), SBO >> 4 (32-45), version 1 (46-47), no swizzle
    return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)(LBO >> 4) << 16) | ((uint64_t)(SBO >> 4) << 32) |
           (1ull << 46);
}

// D = F32 (bits 4-5 = 1); A, B = BF16 (1) at bits 7-9, 10-12; K-major;
// N >> 3 at bits 17-22; M >> 4 at bits 24-28
__host__ __device__ constexpr uint32_t idesc(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ bool mbar_try(uint32_t mbar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(mbar), "r"(parity)
        : "memory");
    return done != 0;
}

// bounded wait; false when it gave up (timeout) or another role aborted
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity, volatile int* abort_flag,
                                          unsigned long long timeout_ns) {
    const unsigned long long t0 = gtimer();
    for (int it = 0;; ++it) {
        if (mbar_try(mbar, parity)) return true;
        if ((it & 63) == 63) {
            if (*abort_flag) return false;
            if (gtimer() - t0 > timeout_ns) {
                *abort_flag = 1;
                return false;
            }
        }
    }
}

__device__ __forceinline__ void mma(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t id, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(id), "r"(accumulate));
}

__device__ __forceinline__ void commit(uint32_t mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
                 : "memory");
}

// 8 accumulator columns of this warp's 32 lanes
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// (hi 2^24 + lo) 2^e, |hi| < 2^62, |lo| < 2^62, rounded to nearest even: the double is
// put together with integer instructions (GB300 issues about 60 of them in the time
// of one FP64 instruction), unless it leaves the normal range.
__device__ __forceinline__ double scaled(long long hi, long long lo, int e) {
    hi += lo >> 24;
    unsigned long long w = ((unsigned long long)lo & 0xffffffull) << 40;   // the fraction below hi
    const bool neg = hi < 0;
    unsigned long long u = (unsigned long long)hi;
    if (neg) {
        u = ~u + (w == 0);
        w = 0 - w;
    }
    e += 24;
    if (u == 0) {
        u = w;
        w = 0;
        e -= 64;
    }
    if (u == 0) return 0.0;
    const int nz = __clzll((long long)u);
    const unsigned long long v = nz ? (u << nz) | (w >> (64 - nz)) : u;
    const bool sticky = (w << nz) != 0;
    unsigned long long m = v >> 11;
    const unsigned low = (unsigned)v & 0x7ffu;
    m += low > 0x400u || (low == 0x400u && (sticky || (m & 1)));
    const int E = 63 - nz + e + 1023;
    if (E >= 1 && E < 2046) {
        const long long bits = (long long)(((unsigned long long)(E - 1) << 52) + m);
        return __longlong_as_double(neg ? bits | (1ll << 63) : bits);
    }
    const double x = ldexp((double)m, E - 1023 - 52);
    return neg ? -x : x;
}

// index of element (r, k) of an operand view
__device__ __forceinline__ size_t oz_index(const OzOperand& X, int r, int k) {
    if (X.mode == 1) return ((size_t)k * 4 + (size_t)(r / X.cr)) * X.cap + (r % X.cr);
    return (size_t)(X.gather ? X.gather[r] : r) * X.rs + (size_t)k * X.ks;
}

// The slicing works on bit patterns with integer arithmetic only: GB300
// issues FP64 instructions at a small fraction of its integer and FP32 rate,
// and the FP64 form of the same cut (scale, round, subtract, repeat) costs
// about 25 of them per element.
//
// Bit pattern of element (r, k), zero-extended (f32 views: 32 bits).
__device__ __forceinline__ unsigned long long oz_bits(const OzOperand& X, int r, int k) {
    const size_t i = oz_index(X, r, k);
    if (X.f32) return (unsigned long long)__float_as_uint(static_cast<const float*>(X.base)[i]);
    unsigned long long v = (unsigned long long)__double_as_longlong(static_cast<const double*>(X.base)[i]);
    if (X.kn) {   // exponent shift; zeros and non-finite values stay, what would leave the range goes to 0
        const int ek = (int)(((unsigned)__double2hiint(X.kn[k]) >> 20) & 0x7ff);
        const int E = (int)((v >> 52) & 0x7ff);
        if (ek != 0 && E != 0 && E != 0x7ff) {
            const int En = E + X.ksgn * ((ek - 1023) >> 1);
            v = En > 0 && En < 0x7ff ? (v & 0x800fffffffffffffull) | ((unsigned long long)En << 52)
                                     : (En <= 0 ? 0ull : 0x7ff8000000000000ull);
        }
    }
    return v;
}

// |x| as an unsigned key that orders like |x| within one storage type
__device__ __forceinline__ unsigned long long abs_key(unsigned long long bits, bool f32) {
    return f32 ? (bits & 0x7fffffffull) : (bits & 0x7fffffffffffffffull);
}

__device__ __forceinline__ bool key_nonfinite(unsigned long long key, bool f32) {
    return f32 ? key >= 0x7f800000ull : key >= 0x7ff0000000000000ull;
}

// e with 2^(e-1) <= max |x| < 2^e from the largest key (0 for a zero row)
__device__ __forceinline__ int key_exponent(unsigned long long key, bool f32) {
    if (key == 0) return 0;
    int e = 0;
    if (f32) {
        const int E = (int)(key >> 23);
        if (E > 0) return E - 126;
        frexp((double)__uint_as_float((unsigned)key), &e);      // subnormal float
    } else {
        const int E = (int)(key >> 52);
        if (E > 0) return E - 1022;
        frexp(__longlong_as_double((long long)key), &e);        // subnormal double
    }
    return e;
}

// X = round(x 2^(8S - 1 - e)) for a finite x = +-m 2^p of a row with exponent e
// (|x| < 2^e, so |X| <= 2^(8S - 1)), ties away from zero
template <int S>
__device__ __forceinline__ long long fixed_of(unsigned long long bits, bool f32, int e) {
    bool neg;
    unsigned long long m;
    int p;
    if (f32) {
        neg = (bits >> 31) & 1;
        const int E = (int)((bits >> 23) & 0xff);
        m = bits & 0x7fffffull;
        if (E) {
            m |= 1ull << 23;
            p = E - 150;
        } else {
            p = -149;
        }
    } else {
        neg = bits >> 63;
        const int E = (int)((bits >> 52) & 0x7ff);
        m = bits & 0xfffffffffffffull;
        if (E) {
            m |= 1ull << 52;
            p = E - 1075;
        } else {
            p = -1074;
        }
    }
    const int sh = p + (8 * S - 1) - e;
    long long X;
    if (m == 0)
        X = 0;
    else if (sh >= 0)
        X = (long long)(m << (sh < 63 ? sh : 63));   // m 2^sh < 2^(8S - 1): no bits leave
    else if (sh <= -62)
        X = 0;
    else
        X = (long long)((m + (1ull << (-sh - 1))) >> -sh);
    return neg ? -X : X;
}

// The S slices of G consecutive fixed-point values X[0..G) (|X| <= 2^(8S - 1)):
// balanced base-256 digits X = sum_t sigma_t 2^(8(S - 1 - t)), |sigma_t| <= 128,
// from the lowest digit up; stored as sigma_t 2^-8t, 16 bytes per slice.
// nan: the row has a non-finite entry, every slice is NaN.
template <int kS>
__device__ __forceinline__ void slice_group(const long long* X, bool nan, uint4* out /* [kS] */) {
    int sig[kS][G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        long long d = X[g];
#pragma unroll
        for (int t = kS - 1; t > 0; --t) {
            const int lo = (int)(((unsigned)d + 128u) & 255u) - 128;
            sig[t][g] = lo;
            d = (d - lo) >> 8;                                      // exact: d - lo = 0 mod 256
        }
        sig[0][g] = (int)d;
    }
#pragma unroll
    for (int t = 0; t < kS; ++t) {
        const float scale = __int_as_float((127 - 8 * t) << 23);   // 2^-8t
        float sl[G];
#pragma unroll
        for (int g = 0; g < G; ++g) sl[g] = nan ? __int_as_float(0x7fc00000) : (float)sig[t][g] * scale;
        uint32_t w[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const __nv_bfloat162 p = __floats2bfloat162_rn(sl[2 * h], sl[2 * h + 1]);
            w[h] = *reinterpret_cast<const uint32_t*>(&p);
        }
        out[t] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// Where a launch finds its problems: an array, one product kind of the ops of a
// chunk, built from the op's descriptor by each CTA (a kernel of its own for that
// would cost a launch per product), or the launch's own argument.
struct OzSource {
    const OzProblem* probs;
    const OpDesc* descs;
    int kind, cap, nops;   // problems nops .. 2 nops - 1: the same product on Z
    OzProblem one;         // neither: this one problem
};

// The problem of one kind for an op (z: of the same product on Z).
template <int kS>
__device__ OzProblem op_problem(const OpDesc& d, int kind, int cap, bool z) {
    const int ld = 4 * cap;
    OzProblem P{};
    const bool first = (kind & OZ_FIRST) != 0;
    kind &= OZ_FIRST - 1;
    if (z && !d.transposed) kind = -1;
    if (d.dot64 || (d.plain && kind != OZ_MERGE && kind != OZ_RECON)) kind = -1;
    auto rowmajor = [](const void* base, int f32, long long ld_) {   // (r, k) at r * ld + k
        return OzOperand{base, f32, ld_, 1, 0, 1, 1, nullptr, nullptr, 0};
    };
    auto colmajor = [](const void* base, int f32, long long ld_) {   // (r, k) at k * ld + r
        return OzOperand{base, f32, 1, ld_, 0, 1, 1, nullptr, nullptr, 0};
    };
    switch (kind) {
        case OZ_MERGE:   // Theta[(l, s1), (s2, r)] = sum_m A[(l, s1), m] B[m, (s2, r)]
            P.M = 4 * d.cl;
            P.K = d.cm;
            P.N = 4 * d.cr;
            P.A = rowmajor(d.A, d.site_f32, cap);
            P.B = OzOperand{d.B, d.site_f32, 0, 0, 1, d.cr, cap, nullptr, nullptr, 0};
            P.C = d.thetap;
            P.ldc = ld;
            break;
        case OZ_RECON:   // B_p'[(l, s1), j] = sum_c Theta'[(l, s1), c] Yk[j, c], j < k (device)
            P.M = d.m;
            P.K = d.n;
            P.N = min(d.chi_max, d.c);
            P.Ndyn = d.k_out;
            P.A = rowmajor(d.thetap, 0, ld);
            P.B = rowmajor(d.Yk, 0, ld);
            P.C = d.A;
            P.ldc = cap;
            P.c_f32 = d.site_f32;
            break;
        case OZ_E:       // E = U U^T - I
            P.M = P.N = P.K = d.c;
            P.A = rowmajor(d.U32, 1, ld);
            P.B = rowmajor(d.U32, 1, ld);
            P.C = d.E;
            P.ldc = ld;
            P.sub_identity = 1;
            P.sym = 1;
            break;
        case OZ_Q:       // Q = U - E U / 2
        case OZ_T4:      // T = U - 5 E U / 6 (in W, free until OZ_W)
        case OZ_T3:      // T = U - 3 E T / 4
        case OZ_U3:      // T = U - 3 E U / 4
        case OZ_T2:      // Q = U - E T / 2
            P.M = P.N = P.K = d.c;
            P.A = rowmajor(d.E, 0, ld);
            P.B = kind == OZ_T3 || kind == OZ_T2 ? colmajor(d.W, 0, ld) : colmajor(d.U32, 1, ld);
            P.C = kind == OZ_T4 || kind == OZ_T3 || kind == OZ_U3 ? d.W : first && d.transposed ? d.Z : d.Q;
            P.ldc = ld;
            P.alpha = kind == OZ_T4 ? -5.0 / 6.0 : kind == OZ_T3 || kind == OZ_U3 ? -0.75 : -0.5;
            P.beta = 1.0;
            P.unit_d = 1;
            P.D = d.U32;
            P.ldd = ld;
            P.d_f32 = 1;
            break;
        case OZ_G:       // G = W W^T (refinement, while the op takes part in it)
            if (d.rf->state != kRefineActive) break;
            P.M = P.N = d.c;
            P.K = d.L;
            P.A = rowmajor(d.W, 0, ld);
            P.B = rowmajor(d.W, 0, ld);
            P.C = d.E;
            P.ldc = ld;
            P.alpha = 1.0;
            P.sym = 1;
            break;
        case OZ_R3:      // T1 = X W / 8 + W / 2                     (order 3)
        case OZ_R2:      // T1 = X T1 + W, or X W / 2 + W            (order 3, 2)
        case OZ_R1: {    // W  = X T1 + W, or X W + W                (order >= 2, 1)
            const int order = d.rf->order;
            if (order < (kind == OZ_R3 ? 3 : kind == OZ_R2 ? 2 : 1)) break;
            P.M = P.K = d.c;
            P.N = z ? d.c : d.L;
            P.A = rowmajor(d.Q, 0, ld);
            const bool fromT = (kind == OZ_R2 && order == 3) || (kind == OZ_R1 && order >= 2);
            double *X = z ? d.Z : d.W, *T = z ? d.Acm : d.W0;   // Acm is free once W0 is formed
            P.B = colmajor(fromT ? T : X, 0, ld);
            P.C = kind == OZ_R1 ? X : T;
            P.ldc = ld;
            P.D = X;
            P.ldd = ld;
            if (z) {
                P.unit_d = 1;
            } else {
                P.A.kn = P.B.kn = d.snorm;   // squared row norms of W: X_ik |w_k| times w_k / |w_k|
                P.A.ksgn = 1;
                P.B.ksgn = -1;
                // what X W adds to a row of W is below 2^e of it, e from the largest angle
                // and the largest off-orthogonality: that many digits fewer are needed
                P.levels = oz_levels(kS, max((int)(d.rf->row1 >> 23) - 126, ((int)(d.rf->rho2 >> 23) - 126) / 2 + 1));
            }
            P.alpha = kind == OZ_R3 ? 0.125 : (kind == OZ_R2 && order == 2 ? 0.5 : 1.0);
            P.beta = kind == OZ_R3 ? 0.5 : 1.0;
            break;
        }
        case OZ_W:       // W = Q W0 (first: W0 = Q theta~, theta~ column-major)
            P.M = d.c;
            P.N = z ? d.c : d.L;
            P.K = d.c;
            P.A = rowmajor(first && d.transposed ? d.Z : d.Q, 0, ld);
            P.B = first ? rowmajor(d.Acm, 0, ld) : colmajor(z ? d.Z : d.W0, 0, ld);
            P.C = z ? d.Z : first ? d.W0 : d.W;
            P.ldc = ld;
            break;
        default:         // an op that takes no part
            break;
    }
    if (kind == OZ_MERGE || kind == OZ_RECON || kind == OZ_E || kind == OZ_W) P.alpha = 1.0;
    P.as = z ? d.oz_as_z : d.oz_as;
    P.bs = z ? d.oz_bs_z : d.oz_bs;
    P.ea = z ? d.oz_ea_z : d.oz_ea;
    P.eb = z ? d.oz_eb_z : d.oz_eb;
    P.status = d.status;
    oz_set_tiles(P);
    return P;
}

// the CTA's problem, through shared memory (the op's descriptor read by all threads at
// once: one thread's chain of loads from it cost 1 to 2 us)
template <int kS>
__device__ __forceinline__ void fetch_problem(const OzSource& src, OzProblem& P) {
    if (src.descs) {
        __shared__ __align__(16) int sd[sizeof(OpDesc) / 4];
        const bool z = (int)blockIdx.z >= src.nops;
        const int* g = reinterpret_cast<const int*>(src.descs + (z ? blockIdx.z - src.nops : blockIdx.z));
        for (int i = threadIdx.x; i < (int)(sizeof(OpDesc) / 4); i += blockDim.x) sd[i] = g[i];
        __syncthreads();
        if (threadIdx.x == 0) P = op_problem<kS>(*reinterpret_cast<const OpDesc*>(sd), src.kind, src.cap, z);
    } else if (threadIdx.x == 0) {
        P = src.probs ? src.probs[blockIdx.z] : src.one;
    }
    __syncthreads();
}

static_assert(sizeof(OpDesc) % 4 == 0, "copied as words");

// the largest |x| key of elements k0, k0 + step, ... of row r, eight loads in flight
__device__ __forceinline__ unsigned long long row_max(const OzOperand& X, int r, int k0, int step, int K) {
    const bool f32 = X.f32 != 0;
    unsigned long long mx = 0;
    for (int k = k0; k < K; k += 8 * step) {
        unsigned long long b[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) b[u] = k + u * step < K ? oz_bits(X, r, k + u * step) : 0ull;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const unsigned long long key = abs_key(b[u], f32);
            mx = key > mx ? key : mx;
        }
    }
    return mx;
}

// Strided views (a transposed operand, the right site of a merge): four blocks
// take 32 consecutive rows, lane = row and warp = a slice of the K range, so that
// the 32 lanes of a load read 32 neighbouring rows at one k (coalesced).  Each block
// scans all of K for the rows' exponents and cuts a quarter of it (one block per 32
// rows left a product of 1000 x 1500 x 777 with 47 of them and 107 us of slicing).
template <int kS>
__device__ void slice_rows_tiled(const OzOperand& X, int r0, int quarter, int R, int K, int Kt, int lv,
                                 unsigned char* out, int* ex, int tile, int Rt) {
    __shared__ unsigned long long s_mx[8][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool f32 = X.f32 != 0;
    const int r = r0 + lane;
    const bool live = r < R;
    __syncthreads();   // the previous rows' maxima are read
    unsigned long long mx = live ? row_max(X, r, warp, 8, K) : 0;
    s_mx[warp][lane] = mx;
    __syncthreads();
    for (int w = 0; w < 8; ++w) mx = s_mx[w][lane] > mx ? s_mx[w][lane] : mx;
    const bool bad = key_nonfinite(mx, f32);   // the largest key of a row with a NaN or an inf is one
    const int e = bad ? 0 : key_exponent(mx, f32);
    if (!live) return;
    if (warp == 0 && quarter == 0) ex[r] = e;
    const int rt = r / tile, rr = r % tile;
    const size_t block = (size_t)tile * 64;
    const size_t within = (size_t)(rr >> 3) * SBO + (size_t)(rr & 7) * 16;
    for (int g0 = (quarter * 8 + warp) * G; g0 < Kt * KT; g0 += 32 * G) {
        long long x[G];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int k = g0 + g;
            x[g] = (!bad && k < K) ? fixed_of<kS>(oz_bits(X, r, k), f32, e) : 0;
        }
        uint4 sl[kS];
        slice_group<kS>(x, bad, sl);
        const int kt = g0 / KT, kk = g0 % KT;
#pragma unroll
        for (int t = 0; t < kS; ++t) {
            if (t >= lv) break;
            unsigned char* blk = out + (((size_t)t * Rt + rt) * Kt + kt) * block;
            *reinterpret_cast<uint4*>(blk + within + (size_t)(kk / G) * LBO) = sl[t];
        }
    }
}

// grid (row groups of 8, 2 = A | B, problems).  Views whose rows are
// contiguous (ks == 1) take one warp per row, lanes along k; the others 32 rows
// per four blocks (slice_rows_tiled).
template <int kS>
__global__ void __launch_bounds__(256, 3) oz_slice_kernel(OzSource src) {
    __shared__ OzProblem P;
    grid_begin();
    fetch_problem<kS>(src, P);
    const bool isB = blockIdx.y == 1;
    const OzOperand& X = isB ? P.B : P.A;
    const int N = P.Ndyn ? *P.Ndyn : P.N;
    const int R = isB ? N : P.M;
    const int tile = isB ? kTileN : kTileM;         // rows per block
    const int Rt = isB ? P.Nt : P.Mt;
    const int K = P.K, Kt = P.Kt;
    const int lv = P.levels > 0 ? P.levels : kS;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char* out = static_cast<unsigned char*>(isB ? P.bs : P.as);
    int* ex = isB ? P.eb : P.ea;
    // Rows past R need no slices: a row of the result depends on its own rows alone.
    // The groups of 8 rows go round the launch's blocks.
    const bool strided = !(X.mode == 0 && X.ks == 1);
    const int groups = strided ? 4 * ((R + 31) / 32) : (R + 7) / 8;
    for (int rb = blockIdx.x; rb < groups; rb += gridDim.x) {
        if (strided) {
            slice_rows_tiled<kS>(X, (rb >> 2) * 32, rb & 3, R, K, Kt, lv, out, ex, tile, Rt);
            continue;
        }
        const int r = rb * 8 + warp;
        if (r >= R) return;
        const bool f32 = X.f32 != 0;
        unsigned long long mx = row_max(X, r, lane, 32, K);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long y = __shfl_xor_sync(0xffffffffu, mx, o);
            mx = y > mx ? y : mx;
        }
        const bool bad = key_nonfinite(mx, f32);
        const int e = bad ? 0 : key_exponent(mx, f32);
        if (lane == 0) ex[r] = e;
        const int rt = r / tile, rr = r % tile;
        const size_t block = (size_t)tile * 64;
        const size_t within = (size_t)(rr >> 3) * SBO + (size_t)(rr & 7) * 16;
        for (int g0 = lane * G; g0 < Kt * KT; g0 += 32 * G) {
            long long x[G];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const int k = g0 + g;
                x[g] = (!bad && k < K) ? fixed_of<kS>(oz_bits(X, r, k), f32, e) : 0;
            }
            uint4 sl[kS];
            slice_group<kS>(x, bad, sl);
            const int kt = g0 / KT, kk = g0 % KT;
#pragma unroll
            for (int t = 0; t < kS; ++t) {
                if (t >= lv) break;
                unsigned char* blk = out + (((size_t)t * Rt + rt) * Kt + kt) * block;
                *reinterpret_cast<uint4*>(blk + within + (size_t)(kk / G) * LBO) = sl[t];
            }
        }
    }
}

template <int kS, int TN>
__global__ void __launch_bounds__(kThreads, 1) oz_gemm_kernel(OzSource src,
                                                               unsigned long long timeout_ns) {
    constexpr int kRangeTiles = kRangeK / KT;
    constexpr int kLevels = kS, kStages = stages_of(kS, TN), kStageBytes = stage_bytes(kS, TN);
    constexpr int kBytesB = TN * 64;   // of one slice block of B
    // barriers: full[kStages], empty[kStages], accumulators full, accumulators drained, final
    constexpr int kBarFull = 0, kBarEmpty = kStages, kBarAccFull = 2 * kStages, kBarAccEmpty = 2 * kStages + 1,
                  kBarFinal = 2 * kStages + 2;
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ OzProblem P;
    grid_begin();
    fetch_problem<kS>(src, P);
    const int N = P.Ndyn ? *P.Ndyn : P.N;
    const int mt = blockIdx.y, nt = blockIdx.x;
    if (mt * kTileM >= P.M || nt * TN >= N) return;
    if (P.sym && (nt + 1) * TN <= mt * kTileM) return;   // mirrored from above the diagonal
    const int Kt = P.Kt;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int kGroup = 16, kGroups = TN / kGroup;   // columns that share a number of levels
    __shared__ int s_ea, s_eb[kGroups];
    if (threadIdx.x <= kGroups) *(threadIdx.x ? s_eb + threadIdx.x - 1 : &s_ea) = -(1 << 20);

    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes);
    uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + kStages * kStageBytes + 128);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kStages * kStageBytes + 144);
    if (threadIdx.x == 0) {
        *abort_flag = 0;
        for (int s = 0; s < kStages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar + kBarFull + s)));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar + kBarEmpty + s)));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar + kBarAccFull)));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 8;" ::"r"(smem_u32(bar + kBarAccEmpty)));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar + kBarFinal)));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                     "r"(tmem_cols(kS, TN)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tslot;
    int lv = P.levels > 0 ? P.levels : kS;   // slice pairs t + u < lv
    // What A B adds to entries of a unit row of D is below 2^(e_i + f_j).  The levels that
    // count are those of 128 rows and 16 columns whatever TN is (lv is their largest, the
    // epilogue takes each group's own): TN follows from the launch's other problems, the
    // result must not.
    if (P.unit_d) {
        if (threadIdx.x < kTileM) {
            const int i = mt * kTileM + threadIdx.x;
            if (i < P.M) atomicMax(&s_ea, P.ea[i]);
        } else if (threadIdx.x < kTileM + TN) {
            const int j = nt * TN + threadIdx.x - kTileM;
            if (j < N) atomicMax(&s_eb[(threadIdx.x - kTileM) / kGroup], P.eb[j]);
        }
        __syncthreads();
        lv = 0;
        for (int g = 0; g < kGroups; ++g) lv = max(lv, oz_levels(kS, s_ea + s_eb[g]));
    }
    const int nrange = (Kt + kRangeTiles - 1) / kRangeTiles;

    if (warp == 0) {
        // producer: bulk copies of the slice blocks of k tile kt into stage kt % kStages
        if (lane == 0) {
            const unsigned char* as = static_cast<const unsigned char*>(P.as);
            const unsigned char* bs = static_cast<const unsigned char*>(P.bs);
            int issued = 0;
            for (int kt = 0; kt < Kt; ++kt) {
                const int s = kt % kStages;
                if (kt >= kStages &&
                    !mbar_wait(smem_u32(bar + kBarEmpty + s), ((kt / kStages) - 1) & 1, abort_flag, timeout_ns))
                    break;
                const uint32_t full = smem_u32(bar + kBarFull + s);
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full), "r"(lv * (kBlockA + kBytesB))
                             : "memory");
                unsigned char* st = smem + (size_t)s * kStageBytes;
                for (int t = 0; t < lv; ++t) {
                    const unsigned char* srcA = as + (((size_t)t * P.Mt + mt) * Kt + kt) * kBlockA;
                    const unsigned char* srcB = bs + (((size_t)t * P.Nt + nt * TN / kTileN) * Kt + kt) * kBlockB +
                                                (nt * TN % kTileN) * 64;   // 8 rows are 512 consecutive bytes
                    asm volatile(
                        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                            smem_u32(st + t * kBlockA)),
                        "l"(srcA), "r"(kBlockA), "r"(full)
                        : "memory");
                    asm volatile(
                        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                            smem_u32(st + kS * kBlockA + t * kBytesB)),
                        "l"(srcB), "r"(kBytesB), "r"(full)
                        : "memory");
                }
                issued = kt + 1;
            }
            // copies still in flight complete on their full barrier before the CTA leaves
            for (int kt = (issued > kStages ? issued - kStages : 0); kt < issued; ++kt)
                mbar_wait(smem_u32(bar + kBarFull + kt % kStages), (kt / kStages) & 1, abort_flag, timeout_ns);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t id = idesc(kTileM, TN);
            int r = 0;
            bool first[kLevels];
#pragma unroll
            for (int l = 0; l < kLevels; ++l) first[l] = true;
            for (int kt = 0; kt < Kt; ++kt) {
                const int s = kt % kStages;
                if (kt % kRangeTiles == 0 && kt > 0) {
                    // accumulators of the previous range must be drained first
                    if (!mbar_wait(smem_u32(bar + kBarAccEmpty), (r - 1) & 1, abort_flag, timeout_ns)) break;
#pragma unroll
                    for (int l = 0; l < kLevels; ++l) first[l] = true;
                }
                if (!mbar_wait(smem_u32(bar + kBarFull + s), (kt / kStages) & 1, abort_flag, timeout_ns)) break;
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint32_t st = smem_u32(smem + (size_t)s * kStageBytes);
#pragma unroll
                for (int lvl = 0; lvl < kLevels; ++lvl) {
                    if (lvl >= lv) break;
                    const uint32_t d = tmem + (uint32_t)(lvl * TN);
#pragma unroll
                    for (int t = 0; t <= lvl; ++t) {
                        const int u = lvl - t;
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            const uint32_t off = q * 2 * LBO;
                            mma(d, smem_desc(st + t * kBlockA + off),
                                smem_desc(st + kS * kBlockA + u * kBytesB + off), id, first[lvl] ? 0u : 1u);
                            first[lvl] = false;
                        }
                    }
                }
                commit(smem_u32(bar + kBarEmpty + s));   // frees the stage once these MMAs have read it
                if (kt % kRangeTiles == kRangeTiles - 1 || kt == Kt - 1) {
                    commit(smem_u32(bar + kBarAccFull));   // accumulators of range r complete
                    ++r;
                }
            }
            commit(smem_u32(bar + kBarFinal));
            mbar_wait(smem_u32(bar + kBarFinal), 0, abort_flag, timeout_ns);   // every MMA issued has completed
        }
    } else {
        // epilogue warps 2..9: rows 32 (warp % 4) + lane, columns half * CP .. + CP - 1
        constexpr int CP = TN / 2;
        const int ew = warp - 2;
        const int lane_base = 32 * (warp & 3);
        const int half = ew >> 2;
        const uint32_t taddr = tmem + ((uint32_t)lane_base << 16) + (uint32_t)(half * CP);
        // Level d holds n_d 2^-8d with n_d an integer (exact for d <= 3; higher levels are
        // rounded to the nearest 2^-8d).  The sum over the ranges is kept exactly:
        // hi 2^24 + lo in units of 2^-40, hi = n_0 2^16 + n_1 2^8 + n_2 (|.| < 2^39 per
        // range), lo = n_3 2^16 + n_4 2^8 + n_5 + n_6 / 2^8 rounded (|.| < 2^41).  A NaN
        // slice reaches level 0.
        long long hi[CP], lo[CP];
        unsigned nan = 0;
#pragma unroll
        for (int j = 0; j < CP; ++j) hi[j] = lo[j] = 0;
        int lg[(CP + kGroup - 1) / kGroup];   // the levels of this warp's column groups
#pragma unroll
        for (int g = 0; g < (CP + kGroup - 1) / kGroup; ++g)
            lg[g] = P.unit_d ? oz_levels(kS, s_ea + s_eb[half * CP / kGroup + g]) : lv;
        bool ok = true;
        for (int r = 0; r < nrange; ++r) {
            if (!mbar_wait(smem_u32(bar + kBarAccFull), r & 1, abort_flag, timeout_ns)) {
                ok = false;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
            for (int lvl = 0; lvl < kLevels; ++lvl) {
                if (lvl >= lv) break;   // uniform: not formed
                const float scale = __int_as_float((127 + 8 * lvl) << 23);   // 2^8d
#pragma unroll
                for (int c = 0; c < CP; c += 8) {
                    if (lvl >= lg[c / kGroup]) continue;   // uniform
                    float v[8];
                    tmem_ld8(taddr + (uint32_t)(lvl * TN + c), v);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int n = __float2int_rn(v[i] * scale);
                        if (lvl == 0) nan |= (v[i] != v[i]) ? 1u << (c + i) : 0u;
                        if (lvl < 3)
                            hi[c + i] += (long long)n * (1 << (16 - 8 * lvl));
                        else if (lvl < 6)
                            lo[c + i] += (long long)n * (1 << (40 - 8 * lvl));
                        else
                            lo[c + i] += (n + 128) >> 8;
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar + kBarAccEmpty)) : "memory");
        }
        const int i = mt * kTileM + lane_base + lane;
        if (ok && !*abort_flag && i < P.M) {
            // alpha a power of two: into the exponent
            const long long ab = __double_as_longlong(P.alpha);
            const int aE = (int)((ab >> 52) & 0x7ff);
            const bool pow2 = (ab & 0xfffffffffffffll) == 0 && aE > 0 && aE < 0x7ff;
            const int ei = P.ea[i] + (pow2 ? aE - 1023 : 0) - 54;   // the sum is in units of 2^-40
            const size_t row = P.c_gather ? (size_t)P.c_gather[i] : (size_t)i;
            const int j0 = nt * TN + half * CP;
#pragma unroll
            for (int jj = 0; jj < CP; ++jj) {
                const int j = j0 + jj;
                // every entry of a symmetric result has one writer: below the diagonal the mirror
                // of (j, i), whose value differs by rounding where the operands do
                if (j >= N || (P.sym && j < i)) continue;
                double v = scaled(hi[jj], lo[jj], ei + P.eb[j]);
                if (pow2)
                    v = __longlong_as_double(__double_as_longlong(v) ^ (ab & (1ll << 63)));
                else
                    v *= P.alpha;
                if ((nan >> jj) & 1u) v = __longlong_as_double(0x7ff8000000000000ll);
                if (P.D) {
                    const size_t di = row * P.ldd + j;
                    v += P.beta * (P.d_f32 ? (double)static_cast<const float*>(P.D)[di]
                                           : static_cast<const double*>(P.D)[di]);
                }
                if (P.sub_identity && i == j) v -= 1.0;
                const size_t ci = row * P.ldc + j;
                if (P.c_f32)
                    static_cast<float*>(P.C)[ci] = (float)v;
                else
                    static_cast<double*>(P.C)[ci] = v;
                if (P.sym && j > i) static_cast<double*>(P.C)[(size_t)j * P.ldc + i] = v;
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols(kS, TN)));
    if (threadIdx.x == 0 && *abort_flag && P.status) atomicOr(P.status, (int)MPDO_ST_TIMEOUT);
}

// Theta' = G Theta in place (rows (l, s1), columns s2 cr + r) and theta~ =
// lambda_{p-1}[l] Theta' (transposed: theta~^T) column-major in Acm; one thread per (l, r).
__global__ void __launch_bounds__(256) gate_weight_kernel(const OpDesc* descs, int chi_cap) {
    const OpDesc& d = descs[blockIdx.y];
    if (d.dot64) return;
    __shared__ double Gs[256];
    Gs[threadIdx.x] = d.G[threadIdx.x];
    __syncthreads();
    const int ld = 4 * chi_cap;
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= d.cl * d.cr) return;
    const int l = e / d.cr, r = e % d.cr;
    double th[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) th[i] = d.thetap[(size_t)(l * 4 + (i >> 2)) * ld + (i & 3) * d.cr + r];
    const double lam = d.lam_left ? d.lam_left[l] : 1.0;
#pragma unroll 4
    for (int o = 0; o < 16; ++o) {
        double v = 0.0;
#pragma unroll
        for (int i = 0; i < 16; ++i) v = fma(Gs[o * 16 + i], th[i], v);
        const int row = l * 4 + (o >> 2), col = (o & 3) * d.cr + r;
        d.thetap[(size_t)row * ld + col] = v;
        d.Acm[d.transposed ? (size_t)row * ld + col : (size_t)col * ld + row] = lam * v;
    }
}

}  // namespace

cudaError_t launch_gate_weight(const OpDesc* d_desc, int nops, int chi_cap, cudaStream_t st) {
    if (nops <= 0) return cudaSuccess;
    dim3 g((chi_cap * chi_cap + 255) / 256, nops);
    gate_weight_kernel<<<g, 256, 0, st>>>(d_desc, chi_cap);
    return cudaGetLastError();
}

size_t oz_slice_bytes(int rows, int K, int S) {
    // room for either operand: ceil(rows / 128) tiles of 8 KB cover ceil(rows / 64) of 4 KB
    const size_t Rt = (rows + kTileM - 1) / kTileM, Kt = (K + KT - 1) / KT;
    return (size_t)S * Rt * Kt * kBlockA;
}

size_t oz_exp_ints(int rows) { return (size_t)((rows + kTileM - 1) / kTileM) * kTileM; }

namespace {

template <int S, int TN>
cudaError_t prepare_one() {
    return cudaFuncSetAttribute(oz_gemm_kernel<S, TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_of(S, TN));
}

}  // namespace

cudaError_t oz_prepare() {
    for (cudaError_t e : {prepare_one<6, 16>(), prepare_one<6, 32>(), prepare_one<6, 64>(), prepare_one<7, 16>(),
                          prepare_one<7, 32>(), prepare_one<7, 64>()})
        if (e != cudaSuccess) return e;
    return cudaSuccess;
}

namespace {

template <int S, int TN>
cudaError_t launch_tiles(const OzSource& src, int count, int max_m, int max_n, unsigned long long timeout_ns,
                         cudaStream_t st) {
    const dim3 grid((max_n + TN - 1) / TN, (max_m + kTileM - 1) / kTileM, count);
    return launch_early(oz_gemm_kernel<S, TN>, grid, kThreads, smem_of(S, TN), st, src, timeout_ns);
}

// Columns per CTA: 64, the most that the accumulators leave room for, unless the
// launch would not fill the chip; an MMA takes 2/3 of the time with 16 columns
// (A's 4 KB per MMA through shared memory is what bounds it) and the epilogue a
// quarter, so that narrower tiles win as long as each still has an SM.
constexpr int kFill = 152;

template <int S>
cudaError_t launch_oz(const OzSource& src, int count, int max_m, int max_n, int max_rows_sliced,
                      unsigned long long timeout_ns, cudaStream_t st) {
    const int rows = ((max_rows_sliced + kTileM - 1) / kTileM) * kTileM;
    // Many short products (an ensemble of chains at chi 24: 160 of them): about 1200
    // blocks that go round the rows, as each first builds its problem, 1 to 2 us of one
    // thread (a replayed step 17.0 -> 15.5 ms).  Rows of more than 256 are worth a block
    // per eight of them (with the limit, the products of a chi 256 step took a quarter
    // longer).
    const int all = (rows + 7) / 8, share = 1216 / (2 * count) > 0 ? 1216 / (2 * count) : 1;
    const int blocks = rows <= 256 && share < all ? share : all;
    const cudaError_t e = launch_early(oz_slice_kernel<S>, dim3(blocks, 2, count), 256, 0, st, src);
    if (e != cudaSuccess) return e;
    const long long tiles = (long long)((max_m + kTileM - 1) / kTileM) * ((max_n + kTileN - 1) / kTileN) * count;
    if (tiles * 4 <= kFill) return launch_tiles<S, 16>(src, count, max_m, max_n, timeout_ns, st);
    if (tiles * 2 <= kFill) return launch_tiles<S, 32>(src, count, max_m, max_n, timeout_ns, st);
    return launch_tiles<S, 64>(src, count, max_m, max_n, timeout_ns, st);
}

cudaError_t launch_oz_source(const OzSource& src, int count, int max_m, int max_n, int max_rows_sliced, int S,
                             unsigned long long timeout_ns, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    return S == 7 ? launch_oz<7>(src, count, max_m, max_n, max_rows_sliced, timeout_ns, st)
                  : launch_oz<6>(src, count, max_m, max_n, max_rows_sliced, timeout_ns, st);
}

}  // namespace

cudaError_t launch_oz_gemm(const OzProblem* d_probs, int count, int max_m, int max_n, int max_rows_sliced, int S,
                           unsigned long long timeout_ns, cudaStream_t st) {
    return launch_oz_source(OzSource{d_probs, nullptr, 0, 0, 0, {}}, count, max_m, max_n, max_rows_sliced, S,
                            timeout_ns, st);
}

cudaError_t launch_oz_ops(const OpDesc* d_desc, int nops, int kind, int chi_cap, int S, bool with_z,
                          unsigned long long timeout_ns, cudaStream_t st) {
    const int big = 4 * chi_cap;
    return launch_oz_source(OzSource{nullptr, d_desc, kind, chi_cap, nops, {}}, with_z ? 2 * nops : nops, big, big, big,
                            S, timeout_ns, st);
}

namespace {

// problem s of a GemmDesc batch as an OzProblem (one thread per problem)
__global__ void gemm_desc_oz_kernel(const GemmDesc* descs, int count, OzScratch scr) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= count) return;
    const GemmDesc& d = descs[s];
    OzProblem P{};
    P.M = d.M;
    P.N = d.N;
    P.K = d.K;
    // A (M x K): stored M x K, or K x M when a_trans
    P.A = d.a_trans ? OzOperand{d.A, d.a_f32, 1, d.lda, 0, 1, 1, nullptr, nullptr, 0}
                    : OzOperand{d.A, d.a_f32, d.lda, 1, 0, 1, 1, nullptr, nullptr, 0};
    // column j of B (K x N) as a row of K values: stored K x N, or N x K when b_trans
    P.B = d.b_trans ? OzOperand{d.B, d.b_f32, d.ldb, 1, 0, 1, 1, nullptr, nullptr, 0}
                    : OzOperand{d.B, d.b_f32, 1, d.ldb, 0, 1, 1, nullptr, nullptr, 0};
    P.C = d.C;
    P.ldc = d.ldc;
    P.alpha = d.alpha;
    P.beta = d.beta;
    P.D = d.D;
    P.ldd = d.ldd;
    P.d_f32 = d.d_f32;
    P.sub_identity = d.sub_identity;
    P.sym = d.sym;
    P.as = scr.as + (size_t)s * scr.slot_bytes;
    P.bs = scr.bs + (size_t)s * scr.slot_bytes;
    P.ea = scr.ea + (size_t)s * scr.exp_ints;
    P.eb = scr.eb + (size_t)s * scr.exp_ints;
    P.status = d.status;
    oz_set_tiles(P);
    scr.probs[s] = P;
}

}  // namespace

cudaError_t launch_gemm_tc(const GemmDesc* d_desc, int count, int max_m, int max_n, int max_k, const OzScratch& scr,
                           int S, unsigned long long timeout_ns, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    // every operand must fit its slot
    const int big = max_m > max_n ? max_m : max_n;
    if (oz_slice_bytes(big, max_k, S) > scr.slot_bytes || oz_exp_ints(big) > scr.exp_ints)
        return cudaErrorInvalidValue;
    gemm_desc_oz_kernel<<<(count + 127) / 128, 128, 0, st>>>(d_desc, count, scr);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_oz_gemm(scr.probs, count, max_m, max_n, big, S, timeout_ns, st);
}

}  // namespace mpdo

// ---------------------------------------------------------------------------
// mpdo_gemm_tc: the same product on caller matrices (include/mpdo.h)
// ---------------------------------------------------------------------------
#include <cuda.h>

#include <mutex>
#include <string>

namespace mpdo {
namespace {

// The scratch of mpdo_gemm_tc comes from a pool of its own per device, which keeps
// up to 256 MB between calls (the slices of a 4096 x 4096 x 2048 product) and returns
// the rest when a call's stream is synchronised; gemm_pool_trim returns all of it.  Allocation is in stream
// order, so calls on several streams and threads do not share a buffer.  A pool ends with
// its device context: the context's id says whether the one at hand is still that
// (after cudaDeviceReset it is not).
constexpr unsigned long long kGemmPoolKeep = 256ull << 20;
constexpr int kMaxPools = 64;

struct GemmPool {
    cudaMemPool_t pool = nullptr;
    unsigned long long context = 0;
};
std::mutex g_pool_mu;
GemmPool g_pools[kMaxPools];

// id of the calling thread's current context, which is unique in the process
cudaError_t context_id(unsigned long long* id) {
    using GetCurrent = CUresult (*)(CUcontext*);
    using GetId = CUresult (*)(CUcontext, unsigned long long*);
    static GetCurrent current = nullptr;
    static GetId get = nullptr;
    static const cudaError_t found = [] {
        cudaDriverEntryPointQueryResult r;
        void *a = nullptr, *b = nullptr;
        cudaError_t e = cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &a, 12000, cudaEnableDefault, &r);
        if (e == cudaSuccess) e = cudaGetDriverEntryPointByVersion("cuCtxGetId", &b, 12000, cudaEnableDefault, &r);
        current = reinterpret_cast<GetCurrent>(a);
        get = reinterpret_cast<GetId>(b);
        return e != cudaSuccess ? e : a && b ? cudaSuccess : cudaErrorNotSupported;
    }();
    if (found != cudaSuccess) return found;
    CUcontext c = nullptr;
    if (current(&c) != CUDA_SUCCESS || !c || get(c, id) != CUDA_SUCCESS) return cudaErrorDeviceUninitialized;
    return cudaSuccess;
}

// the current device's pool of the context at hand (with make, a new one if there is none)
cudaError_t gemm_pool(cudaMemPool_t* out, bool make) {
    *out = nullptr;
    int dev = 0;
    unsigned long long id = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess && make) e = cudaSetDevice(dev);   // the context exists and is current
    if (e == cudaSuccess) e = context_id(&id);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxPools) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_pool_mu);
    GemmPool& g = g_pools[dev];
    if (g.pool && g.context != id) g.pool = nullptr;   // gone with its context
    if (!g.pool && make) {
        if ((e = oz_prepare()) != cudaSuccess) return e;
        cudaMemPoolProps props{};
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t p = nullptr;
        if ((e = cudaMemPoolCreate(&p, &props)) != cudaSuccess) return e;
        unsigned long long keep = kGemmPoolKeep;
        if ((e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep)) != cudaSuccess) {
            cudaMemPoolDestroy(p);
            return e;
        }
        g.pool = p;
        g.context = id;
    }
    *out = g.pool;
    return cudaSuccess;
}

}  // namespace

void gemm_pool_trim() {
    cudaMemPool_t p = nullptr;
    if (gemm_pool(&p, false) == cudaSuccess && p) cudaMemPoolTrimTo(p, 0);
    cudaGetLastError();
}

}  // namespace mpdo

extern "C" int mpdo_gemm_tc(int M, int N, int K, const double* A, int lda, const double* B, int ldb, double* C,
                            int ldc, int kind, void* cuda_stream) {
    using namespace mpdo;
    if (M < 1 || N < 1 || K < 1 || lda < K || ldb < N || ldc < N || !A || !B || !C) {
        set_last_error("mpdo_gemm_tc: need M, N, K >= 1, lda >= K, ldb >= N, ldc >= N and non-NULL matrices");
        return MPDO_EINVAL;
    }
    if (kind != MPDO_MIXED_TF32 && kind != MPDO_MIXED_BF16X3) {
        set_last_error("mpdo_gemm_tc: kind must be MPDO_MIXED_TF32 or MPDO_MIXED_BF16X3");
        return MPDO_EINVAL;
    }
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    OzProblem P{};
    P.M = M;
    P.N = N;
    P.K = K;
    P.A = OzOperand{A, 0, lda, 1, 0, 1, 1, nullptr, nullptr, 0};
    P.B = OzOperand{B, 0, 1, ldb, 0, 1, 1, nullptr, nullptr, 0};
    P.C = C;
    P.ldc = ldc;
    P.alpha = 1.0;
    oz_set_tiles(P);
    const size_t sa = oz_slice_bytes(M, K, 6), sb = oz_slice_bytes(N, K, 6);
    const size_t ia = oz_exp_ints(M), ib = oz_exp_ints(N);
    const size_t bytes = sa + sb + sizeof(int) * (ia + ib);
    unsigned char* buf = nullptr;
    cudaMemPool_t pool = nullptr;
    cudaError_t e = gemm_pool(&pool, true);
    if (e == cudaSuccess) e = cudaMallocFromPoolAsync((void**)&buf, bytes, pool, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_last_error(std::string("mpdo_gemm_tc: ") + cudaGetErrorString(e));
        return MPDO_ENOMEM;
    }
    P.as = buf;
    P.bs = buf + sa;
    P.ea = reinterpret_cast<int*>(buf + sa + sb);
    P.eb = P.ea + ia;
    OzSource src{};
    src.one = P;
    e = launch_oz_source(src, 1, M, N, M > N ? M : N, 6, 4000000000ull, st);
    const cudaError_t ef = cudaFreeAsync(buf, st);
    if (e == cudaSuccess) e = ef;
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        set_last_error(std::string("mpdo_gemm_tc: ") + cudaGetErrorString(e));
        return MPDO_ECUDA;
    }
    return MPDO_OK;
}

// FP32 preconditioning pass of the SVD: one-sided block Jacobi through the Gram
// matrix of each block pair, the row products on the tensor cores.
//
// Input: the c rows of R (FP64, d.W0).  The pass orthogonalises an FP32 copy
// W32 of them (scaled to unit mean square norm) and turns the rows of U32 (I at
// the start) along: U32 is then orthogonal to FP32 accuracy and U32 R has
// nearly orthogonal rows; the later stages (api.cu, refine.cu) finish in FP64
// accuracy, so this pass only decides how much is left to them.
//
// Rows are cut into blocks of 32.  A round-robin tournament meets every pair of
// blocks once per sweep; the op's CTAs take the pairs from a shared counter in
// round order and wait only for a pair's two blocks to leave the previous round
// (jacobi.cu has the same hand-out).  A pair of blocks is processed in three
// steps:
//   1. the 32 x 32 cross block of the Gram matrix of its 64 rows (the two
//      diagonal blocks were left by the blocks' previous pairs; the first round
//      of a sweep forms all three afresh);
//   2. cyclic Jacobi on that 64 x 64 matrix in shared memory: 32 steps of 32
//      disjoint cross pairs (after 31 steps inside the two blocks in the first
//      round), each rotation applied to both sides of the matrix and to the rows
//      of the accumulated rotation M, while one warp finds the next step's
//      angles from the matrix as it was before the step;
//   3. rows <- M rows for W32 and U32, streamed through shared memory.
// The rotations and their order are those of a row-by-row one-sided Jacobi.  Row
// by row, each of the 1024 pairs of a block pair costs a dot product, a warp
// reduction, an angle and an update in one dependent chain: 127 us per block
// pair at rows of 1024, 87 us at rows of 128, against 75 and 34 us here (two
// thirds of it step 3 at rows of 1024, half of it step 2 at 128).  The chain is one
// angle and one 2 x 2 update per step, about 1000 cycles (most of it the barrier and
// the instruction issue of the 16 warps), and steps 1 and 3 are matrix products:
// mma.sync tf32 on operands split in two (hi hi + hi lo + lo hi, 2^-21 relative
// per term), 3 x 64 x 64 MACs per column of the pair.  mma.sync, not tcgen05:
// a pair's products are 64 rows high, their left operand (M) stays in
// registers over all columns, and the results go straight back to L2.  The same
// product on tcgen05 (128 columns x 64 rows per tile, rows stored transposed,
// operands split in shared memory) measured 75 against 67 ms on the chi 256 step:
// splitting and draining a tile cost more than its MMAs.
// Stopping rule, zero rows and bounded waits as described in jacobi.cu.
#include <float.h>
#include <mpdo.h>

#include "coop.cuh"
#include "internal.h"

namespace mpdo {

namespace {

constexpr int NB = kJacobiB32;       // rows per block
constexpr int NP = 2 * NB;           // rows per block pair
constexpr int NT = 512;
constexpr int NWARP = NT / 32;
constexpr int KT = 128;              // columns per streamed tile
constexpr int TS = KT + 8;           // row stride of a tile: conflict-free B fragments
constexpr int kStages = 3;
constexpr int MS = NP + 8;           // row stride of M^T: conflict-free A fragments
constexpr int kIntra = NB - 1;       // steps of a tournament inside a block
constexpr int kSteps = kIntra + NB;
constexpr int GW = 8;                // warp 0 finds the rotations, 1 .. GW - 1 update the Gram matrix, the others M

struct Smem {
    float tile[kStages][NP * TS];
    float G[2][NP * NP];
    float M[NP * MS];                // M^T: M[i][k] at k * MS + i
    float4 ring[2][NB];              // rotations of this step and the next: cos, sin, t g, 1 if it turns
    uchar2 tab[kSteps][NB];          // the 32 pairs of every step
    uchar2 mate[kSteps][NP];         // of every row: the other row of its pair, the pair (+ 128 for the pair's q)
    float norm[NWARP][NP];           // partial squared row norms
    int rid[NP];                     // global row of each slot, -1: none
    double red[NWARP];
    double floor2, scale;
    int conv, pair, any;
    unsigned rho2;
};
static_assert(NWARP * NB * NB * 4 <= (int)sizeof(float) * kStages * NP * TS, "Gram partials fit the tiles");
static_assert(sizeof(Smem) <= 227 * 1024, "shared memory");

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// columns k0 .. k0 + KT - 1 of the pair's rows of a matrix with rows of len
// elements (a multiple of 4) into a tile, zero outside; one cp.async group
__device__ __forceinline__ void load_tile(float* dst, const float* src, int ld, int len, int k0, const int* rid) {
#pragma unroll
    for (int i = 0; i < NP * (KT / 4) / NT; ++i) {
        const int e = threadIdx.x + i * NT;
        const int row = e / (KT / 4), col = k0 + 4 * (e % (KT / 4));
        const int id = rid[row];
        const bool ok = id >= 0 && col < len;
        const float* g = ok ? src + (size_t)id * ld + col : src;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst + row * TS + (col - k0))),
                     "l"(g), "r"(ok ? 16 : 0)
                     : "memory");
    }
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

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

// G[ra + i][rb + j] = <row ra + i, row rb + j> for i, j < 32 (and its mirror).
// Each warp takes one k step of 8 of every tile for the whole 32 x 32 block;
// the warps' partial sums meet in shared memory.  The cross block (ra != rb) also
// takes the squared norms of all 64 rows: those in the blocks' stored Gram
// matrices have lost their digits where a rotation took most of a row away.
__device__ void gram_block(Smem& S, float* G, const float* W, int ld, int L, int ra, int rb, int warp, int lane) {
    const int g = lane >> 2, tg = lane & 3;
    const int nt = (L + KT - 1) / KT;
    float acc[2][4][4];
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[m][n][v] = 0.0f;
    float na[2][2] = {}, nb[4] = {};
    __syncthreads();   // the tiles are free
#pragma unroll
    for (int s = 0; s < kStages - 1; ++s) {
        if (s < nt) load_tile(S.tile[s], W, ld, L, s * KT, S.rid);
        cp_commit();
    }
    for (int kt = 0; kt < nt; ++kt) {
        cp_wait<kStages - 2>();
        __syncthreads();
        if (kt + kStages - 1 < nt)
            load_tile(S.tile[(kt + kStages - 1) % kStages], W, ld, L, (kt + kStages - 1) * KT, S.rid);
        cp_commit();
        const float* T = S.tile[kt % kStages] + 8 * warp + tg;
        uint32_t bh[4][2], bl[4][2];
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float x = T[(rb + 8 * n + g) * TS + 4 * h];
                nb[n] = fmaf(x, x, nb[n]);
                split(x, bh[n][h], bl[n][h]);
            }
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            uint32_t ah[4], al[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const float x = T[(ra + 16 * m + g + 8 * (v & 1)) * TS + 4 * (v >> 1)];
                na[m][v & 1] = fmaf(x, x, na[m][v & 1]);
                split(x, ah[v], al[v]);
            }
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                mma_tf32(acc[m][n], al, bh[n]);
                mma_tf32(acc[m][n], ah, bl[n]);
                mma_tf32(acc[m][n], ah, bh[n]);
            }
        }
    }
    cp_wait<0>();
    __syncthreads();
    float* red = S.tile[0];
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                *reinterpret_cast<float2*>(red + warp * NB * NB + (16 * m + g + 8 * h) * NB + 8 * n + 2 * tg) =
                    make_float2(acc[m][n][2 * h], acc[m][n][2 * h + 1]);
    if (ra != rb) {
        auto put = [&](int row, float v) {
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            v += __shfl_xor_sync(0xffffffffu, v, 2);
            if (tg == 0) S.norm[warp][row] = v;
        };
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int h = 0; h < 2; ++h) put(ra + 16 * m + g + 8 * h, na[m][h]);
#pragma unroll
        for (int n = 0; n < 4; ++n) put(rb + 8 * n + g, nb[n]);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < NB * NB; e += NT) {
        float s = 0.0f;
#pragma unroll
        for (int w = 0; w < NWARP; ++w) s += red[w * NB * NB + e];
        const int i = e / NB, j = e % NB;
        if (ra != rb || i <= j) {
            G[(ra + i) * NP + rb + j] = s;
            G[(rb + j) * NP + ra + i] = s;
        }
    }
}

// The rotation of a pair with squared norms a, b and inner product g: cos, sin,
// t g and whether it turns.  (2g is never above 2^126: the rows are scaled to unit
// mean square norm.)
struct Limits {
    float floor2, tol;   // zero rows; relative off-orthogonality that is left alone
    float lim;           // pairs of two rows below it do not count for the stopping rule
};
struct Stats {
    float rho2;          // largest squared off-orthogonality turned away in a counted pair
    int count, any;      // counted pairs turned; whether any pair was
};
__device__ __forceinline__ float4 rotation(float a, float b, float g, const Limits& lm, Stats& st) {
    const float q = g * rsqrtf(a) * rsqrtf(b);
    const bool turn = a > lm.floor2 && b > lm.floor2 && fabsf(q) > lm.tol;
    // tan 2 theta = 2 g / (b - a), |theta| <= 45 degrees: with r = hypot(b - a, 2 g),
    // cos^2 = (1 + |b - a| / r) / 2 and sin = sign(b - a) g / (r cos), two reciprocal
    // roots in a row.  Scaled by the larger norm's exponent, so that no square
    // leaves FP32's range (a far smaller 2 g squares to zero beside b - a, as it should).
    const unsigned e = __float_as_uint(fmaxf(a, b)) & 0x7f800000u;
    const float sc = __uint_as_float(0x7f000000u - e);
    const float h = (b - a) * sc, g2 = 2.0f * g * sc;
    const float ri = rsqrtf(fmaf(h, h, g2 * g2));
    const float x = fmaf(0.5f, fabsf(h) * ri, 0.5f), ic = rsqrtf(x);
    const float sn = 0.5f * copysignf(g2, h >= 0.0f ? g2 : -g2) * ri * ic;
    const float t = sn * ic;
    const bool ok = turn && t != 0.0f;
    if (ok) {
        st.any = 1;
        if (fmaxf(a, b) >= lm.lim) {
            st.rho2 = fmaxf(st.rho2, q * q);
            ++st.count;
        }
    }
    return ok ? make_float4(x * ic, sn, t * g, 1.0f) : make_float4(1.0f, 0.0f, 0.0f, 0.0f);
}

// Warp 0, lane = pair.  While step `step` is applied to src by the other warps,
// the rotations of the next step are found from src directly: with p's row turned
// as c x + s x_mate, an element of the next matrix is four of this one.  The chain
// from one barrier to the next runs through here, so the indices are read a step
// ahead.
struct Look {
    uchar2 pq, mp, mq;   // the next step's pair, and the mates of its rows in this step
};
__device__ __forceinline__ Look look(const Smem& S, int step, int end, int lane) {
    Look n{};
    if (step + 1 < end) {
        n.pq = S.tab[step + 1][lane];
        n.mp = S.mate[step][n.pq.x];
        n.mq = S.mate[step][n.pq.y];
    }
    return n;
}
__device__ __forceinline__ void lead_step(Smem& S, const float* src, int step, const Look& n, int lane,
                                          const Limits& lm, Stats& st) {
    const float4* ring = S.ring[step & 1];
    const int p = n.pq.x, q = n.pq.y, p2 = n.mp.x, q2 = n.mq.x;
    const float4 rp = ring[n.mp.y & 127], rq = ring[n.mq.y & 127];
    const float app = src[p * (NP + 1)], aqq = src[q * (NP + 1)];
    const float g00 = src[p * NP + q], g01 = src[p * NP + q2], g10 = src[p2 * NP + q], g11 = src[p2 * NP + q2];
    const float sp = n.mp.y & 128 ? rp.y : -rp.y, sq = n.mq.y & 128 ? rq.y : -rq.y;
    const float a = app + (n.mp.y & 128 ? rp.z : -rp.z);
    const float b = aqq + (n.mq.y & 128 ? rq.z : -rq.z);
    const float g0 = fmaf(sq, g01, rq.x * g00), g1 = fmaf(sq, g11, rq.x * g10);
    S.ring[(step + 1) & 1][lane] = rotation(a, b, fmaf(sp, g1, rp.x * g0), lm, st);
}

// Warps 1 .. GW - 1, lane = pair P: the 2 x 2 blocks (pair P, pair P + e), split
// over the warps by e; G is symmetric, so e <= 16 covers all and each result is
// written with its mirror.  The last of these warps also writes the pairs' own
// blocks.
struct Quad {   // one 2 x 2 block of a lane, and where it goes
    int p2, q2;
    float c2, s2, g00, g01, g10, g11;
};
__device__ __forceinline__ Quad load_quad(const float* src, int p, int q, int pair, float cs, float sn, int e, int lane) {
    const int o = (lane + e) & (NB - 1);
    const int v = __shfl_sync(0xffffffffu, pair, o);
    Quad k;
    k.c2 = __shfl_sync(0xffffffffu, cs, o);
    k.s2 = __shfl_sync(0xffffffffu, sn, o);
    k.p2 = v & 255;
    k.q2 = v >> 8;
    k.g00 = src[p * NP + k.p2];
    k.g01 = src[p * NP + k.q2];
    k.g10 = src[q * NP + k.p2];
    k.g11 = src[q * NP + k.q2];
    return k;
}
__device__ __forceinline__ void turn_quad(const Quad& k, float* dst, int p, int q, float cs, float sn) {
    const float r00 = fmaf(cs, k.g00, -sn * k.g10), r01 = fmaf(cs, k.g01, -sn * k.g11);
    const float r10 = fmaf(sn, k.g00, cs * k.g10), r11 = fmaf(sn, k.g01, cs * k.g11);
    const float x00 = fmaf(k.c2, r00, -k.s2 * r01), x01 = fmaf(k.s2, r00, k.c2 * r01);
    const float x10 = fmaf(k.c2, r10, -k.s2 * r11), x11 = fmaf(k.s2, r10, k.c2 * r11);
    dst[p * NP + k.p2] = x00;
    dst[p * NP + k.q2] = x01;
    dst[q * NP + k.p2] = x10;
    dst[q * NP + k.q2] = x11;
    dst[k.p2 * NP + p] = x00;
    dst[k.q2 * NP + p] = x01;
    dst[k.p2 * NP + q] = x10;
    dst[k.q2 * NP + q] = x11;
}
// pq: the lane's pair of this step, read before the step's barrier
__device__ __forceinline__ void gram_step(const Smem& S, const float* src, float* dst, int step, uchar2 pq, int warp,
                                          int lane) {
    static_assert(GW - 1 == 7, "e = warp, warp + 7, warp + 14 cover 1 .. 16");
    const int p = pq.x, q = pq.y, pair = p | (q << 8);
    const float4 r = S.ring[step & 1][lane];
    // all loads before the first store, so that the blocks' chains overlap
    const Quad k0 = load_quad(src, p, q, pair, r.x, r.y, warp, lane);
    const Quad k1 = load_quad(src, p, q, pair, r.x, r.y, warp + 7, lane);
    if (warp + 14 <= NB / 2) {
        const Quad k2 = load_quad(src, p, q, pair, r.x, r.y, warp + 14, lane);
        if (warp + 14 < NB / 2 || lane < NB / 2) turn_quad(k2, dst, p, q, r.x, r.y);   // e = 16: half the lanes cover it
    }
    if (warp == GW - 1) {
        const float a = src[p * (NP + 1)], b = src[q * (NP + 1)], g = src[p * NP + q];
        dst[p * (NP + 1)] = a - r.z;
        dst[q * (NP + 1)] = b + r.z;
        const float off = r.w != 0.0f ? 0.0f : g;
        dst[p * NP + q] = off;
        dst[q * NP + p] = off;
    }
    turn_quad(k0, dst, p, q, r.x, r.y);
    turn_quad(k1, dst, p, q, r.x, r.y);
}

// The accumulated rotation M in registers: a warp of GW .. NWARP - 1 holds MC
// columns, lane i row i of the first block in x and a row of the second in y.
// Inside the blocks (intra) a row takes its mate's value by a shuffle; in the
// cross steps y moves by one lane per step, so lane i always holds its partner
// (32 steps bring y back).  Shared memory is the step's bottleneck: a column costs
// one or two shuffles here against two loads and two stores there.
constexpr int MC = NP / (NWARP - GW);
struct MCols {
    float x[MC], y[MC];
};

__device__ __forceinline__ void m_step(const Smem& S, MCols& m, int step, int lane) {
    if (step < kIntra) {
        const uchar2 mx = S.mate[step][lane], my = S.mate[step][NB + lane];
        const float4 rx = S.ring[step & 1][mx.y & 127], ry = S.ring[step & 1][my.y & 127];
        const float sx = mx.y & 128 ? rx.y : -rx.y, sy = my.y & 128 ? ry.y : -ry.y;
#pragma unroll
        for (int k = 0; k < MC; ++k) {
            const float vx = __shfl_sync(0xffffffffu, m.x[k], mx.x), vy = __shfl_sync(0xffffffffu, m.y[k], my.x & (NB - 1));
            m.x[k] = fmaf(rx.x, m.x[k], sx * vx);
            m.y[k] = fmaf(ry.x, m.y[k], sy * vy);
        }
    } else {   // lane: pair (lane, NB + (lane + step - kIntra) % NB), whose second row y holds
        const float2 r = *reinterpret_cast<const float2*>(&S.ring[step & 1][lane]);
        const int next = (lane + 1) & (NB - 1);
#pragma unroll
        for (int k = 0; k < MC; ++k) {
            const float x = m.x[k], y = m.y[k];
            m.x[k] = fmaf(r.x, x, -r.y * y);
            m.y[k] = __shfl_sync(0xffffffffu, fmaf(r.y, x, r.x * y), next);
        }
    }
}

// rows <- M rows for the pair's rows of W (L columns) and Z (c columns): warp
// (wm, wc) computes rows 16 wm .. + 15 and columns 32 wc .. + 31 of each tile
// with M's fragments in registers.
__device__ void apply_m(Smem& S, float* W, int L, float* Z, int c, int ld, int warp, int lane) {
    const int g = lane >> 2, tg = lane & 3;
    const int wm = warp >> 2, wc = warp & 3;
    const int nw = (L + KT - 1) / KT, nt = nw + (c + KT - 1) / KT;
    uint32_t ah[NP / 8][4], al[NP / 8][4];
#pragma unroll
    for (int k = 0; k < NP / 8; ++k)
#pragma unroll
        for (int v = 0; v < 4; ++v)
            split(S.M[(8 * k + tg + 4 * (v >> 1)) * MS + 16 * wm + g + 8 * (v & 1)], ah[k][v], al[k][v]);
    const int r0 = S.rid[16 * wm + g], r1 = S.rid[16 * wm + g + 8];
    auto load = [&](int t) {
        if (t < nw)
            load_tile(S.tile[t % kStages], W, ld, L, t * KT, S.rid);
        else if (t < nt)
            load_tile(S.tile[t % kStages], Z, ld, c, (t - nw) * KT, S.rid);
        cp_commit();
    };
    __syncthreads();   // the tiles are free
#pragma unroll
    for (int s = 0; s < kStages - 1; ++s) load(s);
    for (int t = 0; t < nt; ++t) {
        cp_wait<kStages - 2>();
        __syncthreads();
        load(t + kStages - 1);
        const float* T = S.tile[t % kStages] + 32 * wc + g;
        float acc[4][4];
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[n][v] = 0.0f;
#pragma unroll
        for (int k = 0; k < NP / 8; ++k)
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                uint32_t bh[2], bl[2];
                split(T[(8 * k + tg) * TS + 8 * n], bh[0], bl[0]);
                split(T[(8 * k + tg + 4) * TS + 8 * n], bh[1], bl[1]);
                mma_tf32(acc[n], al[k], bh);
                mma_tf32(acc[n], ah[k], bl);
                mma_tf32(acc[n], ah[k], bh);
            }
        float* X = t < nw ? W : Z;
        const int len = t < nw ? L : c, k0 = (t < nw ? t : t - nw) * KT + 32 * wc + 2 * tg;
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            if (k0 + 8 * n >= len) continue;
            if (r0 >= 0)
                __stcg(reinterpret_cast<float2*>(X + (size_t)r0 * ld + k0 + 8 * n), make_float2(acc[n][0], acc[n][1]));
            if (r1 >= 0)
                __stcg(reinterpret_cast<float2*>(X + (size_t)r1 * ld + k0 + 8 * n), make_float2(acc[n][2], acc[n][3]));
        }
    }
    cp_wait<0>();
}

__global__ void __launch_bounds__(NT, 1) jacobi32_kernel(const OpDesc* descs, const int* cta_op, const int* cta_rank,
                                                         const int* group, unsigned* sync, int max_sweeps,
                                                         unsigned long long timeout_ns, int ld, float pre_rho2) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem& S = *reinterpret_cast<Smem*>(smem_raw);
    const int op = cta_op[blockIdx.x];
    if (op < 0) return;   // a CTA the plan left unused (graph step)
    const int rank = cta_rank[blockIdx.x];
    const int G = group[op];
    const OpDesc& d = descs[op];
    if (d.plain) return;
    unsigned* sw = sync + (size_t)op * kSyncWords;
    const int c = d.c, L = d.L;
    float* W = d.W32;
    float* Z = d.U32;
    float* diag = d.D32;   // the blocks' own Gram matrices between their pairs: [block][32][32]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned gen = 0;
    const float tol = sqrtf((float)(L > 1 ? L : 1)) * FLT_EPSILON;

    if (rank == 0 && threadIdx.x == 0) {   // set again only on success
        if (d.pre_ok) *d.pre_ok = 0;
        if (d.rf) {
            d.rf->state = kRefineLeft;
            d.rf->order = 0;
        }
    }
    for (int e = threadIdx.x; e < kSteps * NB; e += NT) {
        const int t = e / NB, i = e % NB;
        int p, q;
        if (t < kIntra) {   // circle method inside both blocks: 16 pairs each
            const int y = i & 15, x0 = tour_player(y, t, NB), x1 = tour_player(NB - 1 - y, t, NB);
            p = (i >> 4) * NB + min(x0, x1);
            q = (i >> 4) * NB + max(x0, x1);
        } else {
            p = i;
            q = NB + (i + t - kIntra) % NB;
        }
        S.tab[t][i] = make_uchar2((unsigned char)p, (unsigned char)q);
        S.mate[t][p] = make_uchar2((unsigned char)q, (unsigned char)i);
        S.mate[t][q] = make_uchar2((unsigned char)p, (unsigned char)(i | 128));
    }
    // squared row norms of the FP64 input, for the zero floor and the FP32 scale
    for (int row = rank * NWARP + warp; row < c; row += G * NWARP) {
        const double* w = d.W0 + (size_t)row * ld;
        double a = 0.0;
        for (int i = lane; i < L; i += 32) {
            const double x = __ldcg(w + i);
            a = fma(x, x, a);
        }
        a = warp_sum(a);
        if (lane == 0) __stcg(d.snorm + row, a);
    }
    if (!op_barrier(sw, G, gen, timeout_ns)) goto timeout;
    {
        double f = 0.0;
        for (int j = threadIdx.x; j < c; j += NT) f += __ldcg(d.snorm + j);
        f = warp_sum(f);
        if (lane == 0) S.red[warp] = f;
        __syncthreads();
        if (threadIdx.x == 0) {
            f = 0.0;
            for (int w = 0; w < NWARP; ++w) f += S.red[w];
            // numerical zero of the FP64 data: the FP32 copy of a row far below
            // eps32 ||W|| is still accurate relative to its own norm (the rows of
            // R are graded), so this pass must rotate it too
            S.floor2 = DBL_EPSILON * DBL_EPSILON * f;
            S.scale = f > 0.0 ? sqrt((double)c / f) : 1.0;
        }
        __syncthreads();
    }
    for (int row = rank * NWARP + warp; row < c; row += G * NWARP) {
        for (int i = lane; i < c; i += 32) __stcg(Z + (size_t)row * ld + i, i == row ? 1.0f : 0.0f);
        const double sc = S.scale;
        for (int i = lane; i < L; i += 32) __stcg(W + (size_t)row * ld + i, (float)(__ldcg(d.W0 + (size_t)row * ld + i) * sc));
    }
    if (!op_barrier(sw, G, gen, timeout_ns)) goto timeout;
    {
        Limits lm{(float)(S.floor2 * S.scale * S.scale), tol, 0.0f};
        const int nb = (c + NB - 1) / NB;
        const int nbp = nb + (nb & 1);
        const int npair = nbp / 2;
        const int sweeps = max_sweeps < kMaxSweepsCap ? max_sweeps : kMaxSweepsCap;
        int conv = (c <= 1);
        int used = 0;
        for (int sweep = 0; sweep < sweeps && !conv; ++sweep) {
            Stats st{0.0f, 0, 0};
            // Rows that the truncation discards need not be orthogonal to one another
            // (jacobi.cu): pairs of two rows a thousand times below the largest
            // discarded ones do not keep the pass going.  (Together they could still
            // not reach into the kept part of the spectrum.)
            lm.lim = 0.0f;
            const int kk = d.chi_max + max(16, d.chi_max / 8);
            if (!d.full_svd && kk < c) {
                const double sc2 = S.scale * S.scale;
                lm.lim = 1e-6f * kth_largest_f<NT, 4 * kMaxChi>(
                                     [&](int j) {
                                         return sweep == 0 ? (float)(__ldcg(d.snorm + j) * sc2)
                                                           : __ldcg(diag + (size_t)(j / NB) * NB * NB + (j % NB) * (NB + 1));
                                     },
                                     c, kk);
                // every CTA has read the norms before a pair of this sweep changes them, or
                // their limits, and with them the sweep that ends the pass, could differ
                if (sweep > 0 && !op_barrier(sw, G, gen, timeout_ns)) goto timeout;
            }
            lm.lim = fmaxf(lm.lim, (float)cutoff_floor(d, (double)c));   // rows of unit mean square norm
            if (rank == 0 && threadIdx.x == 0) atomicExch(&sw[kSwQueue + ((sweep + 1) & 1)], 0u);
            int next = 0;
            for (;;) {
                int qpos = next++;   // an op with one CTA takes all pairs in order
                if (G > 1) {
                    if (threadIdx.x == 0) S.pair = (int)atomicAdd(&sw[kSwQueue + (sweep & 1)], 1u);
                    __syncthreads();
                    qpos = S.pair;
                }
                if (qpos >= (nbp - 1) * npair) break;
                const int r = qpos / npair, i = qpos % npair;
                const int x0 = tour_player(i, r, nbp), x1 = tour_player(nbp - 1 - i, r, nbp);
                const int P = min(x0, x1), Q = max(x0, x1);
                const unsigned R = (unsigned)(sweep * (nbp - 1) + r);   // rounds of this launch before
                __syncthreads();   // S.pair read, the previous pair done
                if (threadIdx.x == 0) {
                    S.conv = G == 1 || wait_blocks(sw + kSwVer, P, Q, nb, R, &sw[1], timeout_ns);
                    S.any = 0;
                }
                if (threadIdx.x < NP) {
                    const int blk = threadIdx.x < NB ? P : Q, row = blk * NB + (threadIdx.x % NB);
                    S.rid[threadIdx.x] = blk < nb && row < c ? row : -1;
                }
                __syncthreads();
                if (!S.conv) goto timeout;
                const bool first = r == 0, lone = Q >= nb;   // lone: the second block is empty
                st.any = 0;
                do {
                    if (lone && !first) break;   // a block that sits this round out
                    float* G0 = S.G[0];
                    float own[2 * NB * NB / NT];   // the blocks' own Gram matrices
                    if (!first) {
#pragma unroll
                        for (int k = 0; k < 2 * NB * NB / NT; ++k) {
                            const int e = threadIdx.x + k * NT;
                            own[k] = __ldcg(diag + (size_t)(e < NB * NB ? P : Q) * NB * NB + e % (NB * NB));
                        }
                    }
                    if (lone) {
                        for (int e = threadIdx.x; e < NP * NP; e += NT) G0[e] = 0.0f;
                    } else {
                        gram_block(S, G0, W, ld, L, 0, NB, warp, lane);
                    }
                    if (first) {
                        __syncthreads();
                        gram_block(S, G0, W, ld, L, 0, 0, warp, lane);
                        if (!lone) {
                            __syncthreads();
                            gram_block(S, G0, W, ld, L, NB, NB, warp, lane);
                        }
                    } else {
                        __syncthreads();
#pragma unroll
                        for (int k = 0; k < 2 * NB * NB / NT; ++k) {
                            const int e = threadIdx.x + k * NT;
                            const int h = e / (NB * NB), x = (e / NB) % NB, y = e % NB;
                            if (x != y) G0[(h * NB + x) * NP + h * NB + y] = own[k];
                        }
                        if (threadIdx.x < NP) {
                            float s = 0.0f;
#pragma unroll
                            for (int w = 0; w < NWARP; ++w) s += S.norm[w][threadIdx.x];
                            G0[threadIdx.x * (NP + 1)] = s;
                        }
                    }
                    __syncthreads();
                    // the pair's rotations, one barrier per step
                    const int s0 = first ? 0 : kIntra, s1 = lone ? kIntra : kSteps;
                    int cur = 0;
                    if (warp == 0) {
                        const uchar2 pq = S.tab[s0][lane];   // the first step's rotations
                        S.ring[s0 & 1][lane] = rotation(G0[pq.x * (NP + 1)], G0[pq.y * (NP + 1)],
                                                        G0[pq.x * NP + pq.y], lm, st);
                    }
                    MCols mc;
#pragma unroll
                    for (int k = 0; k < MC; ++k) {
                        const int col = (warp - GW) * MC + k;
                        mc.x[k] = lane == col ? 1.0f : 0.0f;
                        mc.y[k] = NB + lane == col ? 1.0f : 0.0f;
                    }
                    Look next_pairs = look(S, s0, s1, lane);
                    uchar2 pq = S.tab[s0][lane];
                    __syncthreads();
                    for (int s = s0; s < s1; ++s) {
                        const float* src = S.G[cur];
                        float* dst = S.G[cur ^ 1];
                        if (warp == 0) {
                            if (s + 1 < s1) lead_step(S, src, s, next_pairs, lane, lm, st);
                            next_pairs = look(S, s + 1, s1, lane);
                        } else if (warp < GW) {
                            gram_step(S, src, dst, s, pq, warp, lane);
                            pq = S.tab[min(s + 1, kSteps - 1)][lane];
                        } else {
                            m_step(S, mc, s, lane);
                        }
                        cur ^= 1;
                        __syncthreads();
                    }
                    if (warp >= GW) {
#pragma unroll
                        for (int k = 0; k < MC; ++k) {
                            const int col = (warp - GW) * MC + k;
                            S.M[col * MS + lane] = mc.x[k];
                            S.M[col * MS + NB + lane] = mc.y[k];
                        }
                    }
                    if (warp == 0 && __any_sync(0xffffffffu, st.any) && lane == 0) S.any = 1;
                    // the blocks' own Gram matrices for their next pairs
                    for (int e = threadIdx.x; e < 2 * NB * NB; e += NT) {
                        const int h = e / (NB * NB), x = (e / NB) % NB, y = e % NB;
                        const int blk = h ? Q : P;
                        if (blk < nb)
                            __stcg(diag + (size_t)blk * NB * NB + x * NB + y, S.G[cur][(h * NB + x) * NP + h * NB + y]);
                    }
                    __syncthreads();
                    if (S.any) apply_m(S, W, L, Z, c, ld, warp, lane);
                } while (false);
                // the pair's rows are stored: its blocks leave round r
                __threadfence();
                __syncthreads();
                if (threadIdx.x == 0) {
                    if (P < nb) st_release(&sw[kSwVer + P], R + 1);
                    if (Q < nb) st_release(&sw[kSwVer + Q], R + 1);
                }
            }
            if (warp == 0) {
                const int n = __reduce_add_sync(0xffffffffu, st.count);
                const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(st.rho2));
                if (lane == 0 && n > 0) {
                    atomicAdd(&sw[8 + sweep], (unsigned)n);
                    atomicMax(&sw[8 + kMaxSweepsCap + sweep], m);
                }
            }
            if (!op_barrier(sw, G, gen, timeout_ns)) goto timeout;
            // done when fewer than c/4 pairs still rotate (a few pairs sit at FP32's
            // resolution forever), or when the largest relative off-orthogonality
            // rotated away was at most pre_rho (default 1e-3): the rows are then
            // orthogonal to ~pre_rho^2, near FP32's rounding level for these inner
            // products, and further sweeps only chase rounding
            if (threadIdx.x == 0)
                S.conv = ld_acquire(&sw[8 + sweep]) <= (unsigned)(c / 4) ||
                         __uint_as_float(ld_acquire(&sw[8 + kMaxSweepsCap + sweep])) <= pre_rho2;
            __syncthreads();
            conv = S.conv;
            used = sweep + 1;
        }
        if (rank == 0 && threadIdx.x == 0) {
            if (d.sweeps_out) *d.sweeps_out += used << 16;   // FP32 sweeps in the high half
            if (d.rf) {   // the refinement starts (refine.cu)
                d.rf->state = c > 1 ? kRefineActive : kRefineLeft;
                d.rf->order = 0;
                d.rf->thr = 0.0;
            }
            if (d.pre_ok)
                *d.pre_ok = used > 0 && __uint_as_float(ld_acquire(&sw[8 + kMaxSweepsCap + used - 1])) <= pre_rho2;
        }
    }
    return;
timeout:
    if (threadIdx.x == 0) atomicOr(d.status, (int)MPDO_ST_TIMEOUT);
}

}  // namespace

cudaError_t jacobi32_max_resident(int* per_sm) {
    cudaError_t e =
        cudaFuncSetAttribute(jacobi32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, jacobi32_kernel, NT, sizeof(Smem));
}

cudaError_t launch_jacobi32(const OpDesc* d_desc, const int* d_cta_op, const int* d_cta_rank, const int* d_group,
                            unsigned* d_sync, int grid, int max_sweeps, unsigned long long timeout_ns, int ld,
                            cudaStream_t st, double pre_rho) {
    if (grid <= 0) return cudaSuccess;
    float pre_rho2 = (float)(pre_rho * pre_rho);
    void* args[] = {(void*)&d_desc, (void*)&d_cta_op,   (void*)&d_cta_rank, (void*)&d_group, (void*)&d_sync,
                    (void*)&max_sweeps, (void*)&timeout_ns, (void*)&ld,     (void*)&pre_rho2};
    return cudaLaunchCooperativeKernel((const void*)jacobi32_kernel, dim3(grid), dim3(NT), args, sizeof(Smem), st);
}

}  // namespace mpdo

// One Trotter step as a CUDA graph (mpdo_trotter_step_graph).
//
// mpdo_trotter_step reads the new bond dimensions back to the host after every
// chunk of ops, to size the next chunk's launches exactly.  Here nothing goes
// back to the host inside a step: every chunk starts with a planner kernel that
// reads the bond dimensions on the device and writes the dimension fields of
// the chunk's op descriptors, the co-resident CTA plans of the cooperative QR
// and Jacobi launches (the host plan's proportional-to-work rule; the launch
// has every resident CTA and the unassigned ones return at once); the
// tensor-core products build their problem shapes from the descriptors on the
// device as well, and every other launch has a capacity-sized grid
// whose CTAs outside an op's shape return at once.  The step is captured once
// per layout (op list and workspaces) and replayed; ranks are collected on the
// device.
#include <mpdo.h>

#include <algorithm>
#include <new>
#include <vector>

#include "ctx.h"
#include "internal.h"

using namespace mpdo;

namespace mpdo {

namespace {

// Shares R co-resident CTAs among the ops of a chunk in proportion to their
// work, each op between 1 and cap_s CTAs (the host plan's rule; none for cap_s = 0).  out: [R] op
// of each CTA (-1: unused, the CTA returns at once), [R] rank within the op,
// [nops] CTAs per op.  Returns 0, or 1 if R < nops.
// Called by a whole CTA; G: [nops] in shared memory.
__device__ int plan_ctas(const double* work, const int* cap, int nops, int R, int* out, int* G) {
    __shared__ double s_wsum;
    __shared__ int s_total;
    __syncthreads();   // work and cap are there, G is free
    if (threadIdx.x == 0) {
        double wsum = 0.0;
        for (int s = 0; s < nops; ++s) wsum += cap[s] > 0 ? work[s] : 0.0;
        s_wsum = fmax(wsum, 1.0);
        s_total = 0;
    }
    __syncthreads();
    for (int s = threadIdx.x; s < nops; s += blockDim.x) {
        int g = 0;
        if (cap[s] > 0) {
            g = (int)floor((double)R * work[s] / s_wsum);
            g = max(1, min(cap[s], g));
            const int passes = (cap[s] + g - 1) / g;
            g = (cap[s] + passes - 1) / passes;
        }
        G[s] = g;
        if (g > 0) atomicAdd(&s_total, g);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        while (s_total > R) {
            int arg = 0;
            for (int s = 1; s < nops; ++s)
                if (G[s] > G[arg]) arg = s;
            if (G[arg] <= 1) break;
            G[arg]--;
            s_total--;
        }
    }
    __syncthreads();
    const int total = s_total;
    if (total > R) return 1;
    for (int s = threadIdx.x; s < nops; s += blockDim.x) {
        int t = 0;
        for (int u = 0; u < s; ++u) t += G[u];
        out[2 * R + s] = G[s];
        for (int g = 0; g < G[s]; ++g, ++t) {
            out[t] = s;
            out[R + t] = g;
        }
    }
    for (int t = total + threadIdx.x; t < R; t += blockDim.x) {
        out[t] = -1;
        out[R + t] = 0;
    }
    return 0;
}

constexpr int kMaxChunk = 1024;

__global__ void __launch_bounds__(256) plan_chunk_kernel(OpDesc* descs, int nops, const int* dims, int N, int Rj,
                                                         int Rq, int* cta64, int* cta32, int* ctaqr, int* ctaq32, int Rq32, int precond, int q32,
                                                         int mixed, int blocked,
                                                         const int* jb_table, int chi_cap, const int* lp, int n_lp,
                                                         int* error) {
    __shared__ double work[kMaxChunk];
    __shared__ int cap[kMaxChunk];
    for (int s = threadIdx.x; s < nops; s += blockDim.x) {
        OpDesc& d = descs[s];
        const int* dm = dims + (size_t)d.b * (N + 1);
        d.cl = dm[d.p];
        d.cm = dm[d.p + 1];
        d.cr = dm[d.p + 2];
        d.m = 4 * d.cl;
        d.n = 4 * d.cr;
        d.c = min(d.m, d.n);
        d.plain = q32 && !mixed;   // the rule of run_chunk: all bonds of the instance's layer
        for (int i = 0; d.plain && i < n_lp; ++i) d.plain = 4 * min(dm[lp[i]], dm[lp[i] + 2]) <= kPlainRows;
        d.transposed = q32 && !d.plain && d.m > d.n;
        d.W0 = d.plain ? d.W : d.W0_staged;
        d.L = d.transposed ? d.m : d.n;
        d.jb = jacobi_block_rows(d.transposed ? d.L + d.c : d.L, d.c, 8);
        if (jb_table && !d.transposed) {   // autotuned rows per block of this (chi_l, chi_r) class
            const int t = jb_table[(size_t)d.cl * (chi_cap + 1) + d.cr];
            if (t > 0) d.jb = t;
        }
    }
    __shared__ int G[kMaxChunk];
    int bad = 0;
    for (int s = threadIdx.x; s < nops; s += blockDim.x) {   // the thread's own descriptors
        const OpDesc& d = descs[s];
        work[s] = (double)d.c * d.c * (double)d.L;
        cap[s] = jacobi_pairs_per_round(d.c, d.jb);
    }
    bad |= plan_ctas(work, cap, nops, Rj, cta64, G);
    if (precond) {
        __syncthreads();
        for (int s = threadIdx.x; s < nops; s += blockDim.x) cap[s] = jacobi_pairs_per_round(descs[s].c, kJacobiB32);
        bad |= plan_ctas(work, cap, nops, Rj, cta32, G);
    }
    __syncthreads();
    for (int s = threadIdx.x; s < nops; s += blockDim.x) {
        const OpDesc& d = descs[s];
        work[s] = (double)d.m * d.n * d.c;
        cap[s] = q32 && !d.plain ? 0 : max(1, (d.n + kQrWarps - 1) / kQrWarps);
    }
    if (!blocked) bad |= plan_ctas(work, cap, nops, Rq, ctaqr, G);
    if (q32) {
        __syncthreads();
        for (int s = threadIdx.x; s < nops; s += blockDim.x) cap[s] = descs[s].plain ? 0 : qr32_max_ctas(descs[s].c);
        bad |= plan_ctas(work, cap, nops, Rq32, ctaq32, G);
    }
    if (bad) *error = 1;
}

// klog[b * n_ops + op] = the rank the op chose
__global__ void klog_kernel(const OpDesc* descs, int nops, int n_ops, int* klog) {
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < nops; s += gridDim.x * blockDim.x) {
        const OpDesc& d = descs[s];
        klog[(size_t)d.b * n_ops + d.op] = *d.k_out;
    }
}

struct Chunk {
    int nops = 0;
    OpDesc* d_desc = nullptr;
    int *d_cta64 = nullptr, *d_cta32 = nullptr, *d_ctaqr = nullptr, *d_ctaq32 = nullptr;
    int* d_lp = nullptr;   // path positions of the layer's ops
    int n_lp = 0;
    bool stages = true;    // whether any of its bonds can grow over kPlainRows rows
};

}  // namespace

struct GraphState {
    long long layout = -1;
    cudaStream_t cap_st = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    std::vector<std::vector<Chunk>> chunks;   // per layer
    int* d_klog = nullptr;                    // [B][n_ops] ranks of the last replayed step
    int* d_error = nullptr;
    int Rj = 0, Rq = 0, Rq32 = 0;
};

namespace {

void release(GraphState* g) {
    if (g->exec) cudaGraphExecDestroy(g->exec);
    if (g->graph) cudaGraphDestroy(g->graph);
    g->exec = nullptr;
    g->graph = nullptr;
    for (auto& L : g->chunks)
        for (auto& ch : L) {
            void* ptrs[] = {ch.d_desc, ch.d_cta64, ch.d_cta32, ch.d_ctaqr, ch.d_ctaq32, ch.d_lp};
            for (void* p : ptrs)
                if (p) cudaFree(p);
        }
    g->chunks.clear();
    if (g->d_klog) cudaFree(g->d_klog);
    if (g->d_error) cudaFree(g->d_error);
    g->d_klog = nullptr;
    g->d_error = nullptr;
    g->layout = -1;
}

// queue one step on stream st (captured)
int enqueue_step(mpdo_ctx* c, GraphState* g, cudaStream_t st) {
    const int cap = c->cap, ld = c->ld;
    const unsigned long long timeout_ns = (unsigned long long)c->cfg.barrier_timeout_ms * 1000000ull;
    const bool blocked = c->mixed && c->cfg.qr_blocked && qrb_fits(cap);
    for (auto& L : g->chunks)
        for (auto& ch : L) {
            const int nops = ch.nops;
            const bool q32 = use_qr32(c), staged = c->precond && ch.stages;
            plan_chunk_kernel<<<1, 256, 0, st>>>(ch.d_desc, nops, c->d_dims, c->N, g->Rj, g->Rq, ch.d_cta64,
                                                 ch.d_cta32, ch.d_ctaqr, ch.d_ctaq32, g->Rq32,
                                                 c->precond ? 1 : 0, q32 ? 1 : 0, c->mixed ? 1 : 0, blocked ? 1 : 0,
                                                 c->d_jb_table, cap, ch.d_lp, ch.n_lp, g->d_error);
            CU(cudaGetLastError());
            CU(cudaMemsetAsync(c->d_sweeps, 0, sizeof(int) * nops, st));
            if (c->precond) {
                CU(launch_oz_ops(ch.d_desc, nops, OZ_MERGE, cap, c->oz_s, false, timeout_ns, st));
                CU(launch_gate_weight(ch.d_desc, nops, cap, st));
            } else {
                CU(launch_merge_gate(ch.d_desc, nops, cap, st));
            }
            const size_t sync_bytes = sizeof(unsigned) * jacobi_sync_words(nops);
            CU(cudaMemsetAsync(c->d_sync, 0, sync_bytes, st));
            if (blocked) {
                CU(launch_qr_blocked(ch.d_desc, nops, cap, c->d_oz, timeout_ns, st, 0));
            } else {
                if (!q32 || !c->mixed)   // mixed contexts have no plain ops
                    CU(launch_qr(ch.d_desc, ch.d_ctaqr, ch.d_ctaqr + g->Rq, ch.d_ctaqr + 2 * g->Rq, c->d_sync, g->Rq,
                                 timeout_ns, ld, st));
                if (q32 && staged) {
                    CU(cudaMemsetAsync(c->d_sync, 0, sync_bytes, st));
                    CU(launch_qr32(ch.d_desc, ch.d_ctaq32, ch.d_ctaq32 + g->Rq32, ch.d_ctaq32 + 2 * g->Rq32, c->d_sync,
                                   g->Rq32, timeout_ns, ld, st));
                    CU(launch_orthogonalise(c, ch.d_desc, nops, OZ_FIRST, false, st));
                }
            }
            if (staged) {
                CU(cudaMemsetAsync(c->d_sync, 0, sync_bytes, st));
                CU(launch_jacobi(ch.d_desc, nops, ch.d_cta32, ch.d_cta32 + g->Rj, ch.d_cta32 + 2 * g->Rj, c->d_sync,
                                 g->Rj, kMaxSweepsCap / 2, 0.0, timeout_ns, ld, true, st, precond_rho(c)));
                CU(launch_svd_products(c, ch.d_desc, nops, fp64_jacobi_tol(c), q32, st));
            }
            CU(cudaMemsetAsync(c->d_sync, 0, sync_bytes, st));
            CU(launch_jacobi(ch.d_desc, nops, ch.d_cta64, ch.d_cta64 + g->Rj, ch.d_cta64 + 2 * g->Rj, c->d_sync, g->Rj,
                             c->cfg.jacobi_max_sweeps, fp64_jacobi_tol(c), timeout_ns, ld, false, st, precond_rho(c)));
            CU(launch_truncate(ch.d_desc, nops, cap, st));
            if (c->precond)
                CU(launch_oz_ops(ch.d_desc, nops, OZ_RECON, cap, c->oz_s, false, timeout_ns, st));
            else
                CU(launch_reconstruct(ch.d_desc, nops, cap, st));
            klog_kernel<<<(nops + 127) / 128, 128, 0, st>>>(ch.d_desc, nops, c->n_ops, g->d_klog);
            CU(cudaGetLastError());
        }
    CU(launch_trace_normalize(c->d_sites, sites_f32(c), c->d_dims, c->N, c->B, cap, c->cfg.force_trace, c->d_trace,
                              c->d_status, st));
    return MPDO_OK;
}

int build_graph(mpdo_ctx* c, GraphState* g) {
    release(g);
    if (!g->cap_st) CU(cudaStreamCreateWithFlags(&g->cap_st, cudaStreamNonBlocking));
    g->Rj = c->jacobi_resident;
    g->Rq = c->qr_resident;
    g->Rq32 = c->qr32_resident;
    CU(dalloc(&g->d_klog, (size_t)c->B * c->n_ops));
    CU(dalloc(&g->d_error, 1));
    CU(cudaMemsetAsync(g->d_error, 0, sizeof(int), c->st));
    g->chunks.assign(c->layers.size(), {});
    for (int li = 0; li < (int)c->layers.size(); ++li) {
        const std::vector<Item> items = layer_items(c, li);
        const size_t cs = (size_t)chunk_ops(c);
        for (size_t s0 = 0; s0 < items.size(); s0 += cs) {
            const int nops = (int)std::min(cs, items.size() - s0);
            if (nops > kMaxChunk || nops > std::min(g->Rj, std::min(g->Rq, g->Rq32)))
                return fail(MPDO_ECAPACITY, "graph step: more ops in one chunk than co-resident CTAs");
            Chunk ch;
            ch.nops = nops;
            std::vector<OpDesc> h(nops);
            for (int s = 0; s < nops; ++s) fill_desc(c, items[s0 + s], s, false, h[s]);
            std::vector<int> lp;
            for (const Op& o : c->layers[li]) lp.push_back(o.p);
            ch.n_lp = (int)lp.size();
            // Instances of chi_max <= kPlainRows / 4 leave the stages out whatever their bonds
            // are: a chunk of them is captured without (chi 4, one chain of 10: 5.1 -> 4.6 ms
            // for two steps, sixteen: 6.3 -> 5.3 ms).
            ch.stages = c->mixed;
            for (int s = 0; s < nops; ++s)
                for (int p : lp)
                    ch.stages = ch.stages || (p > 0 && p + 2 < c->N && 4 * c->chi_max[items[s0 + s].b] > kPlainRows);
            CU(dalloc(&ch.d_lp, lp.size()));
            CU(cudaMemcpyAsync(ch.d_lp, lp.data(), sizeof(int) * lp.size(), cudaMemcpyHostToDevice, c->st));
            CU(dalloc(&ch.d_desc, (size_t)nops));
            CU(dalloc(&ch.d_cta64, (size_t)2 * g->Rj + nops));
            CU(dalloc(&ch.d_ctaqr, (size_t)2 * g->Rq + nops));
            if (c->precond) CU(dalloc(&ch.d_cta32, (size_t)2 * g->Rj + nops));
            if (c->precond) CU(dalloc(&ch.d_ctaq32, (size_t)2 * g->Rq32 + nops));
            CU(cudaMemcpyAsync(ch.d_desc, h.data(), sizeof(OpDesc) * nops, cudaMemcpyHostToDevice, c->st));
            CU(cudaStreamSynchronize(c->st));
            g->chunks[li].push_back(ch);
        }
    }
    CU(cudaStreamSynchronize(c->st));
    CU(cudaStreamBeginCapture(g->cap_st, cudaStreamCaptureModeThreadLocal));
    int rc = enqueue_step(c, g, g->cap_st);
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamEndCapture(g->cap_st, &graph);
    if (rc) {
        if (graph) cudaGraphDestroy(graph);
        return rc;
    }
    if (e != cudaSuccess) return fail(MPDO_ECUDA, std::string("graph capture: ") + cudaGetErrorString(e));
    g->graph = graph;
    CU(cudaGraphInstantiate(&g->exec, g->graph, 0));
    g->layout = c->layout;
    return MPDO_OK;
}

}  // namespace

void graph_free(GraphState* g) {
    if (!g) return;
    release(g);
    if (g->cap_st) cudaStreamDestroy(g->cap_st);
    delete g;
}

}  // namespace mpdo

extern "C" int mpdo_trotter_step_graph(mpdo_ctx* c, int n_steps) {
    if (!c) return fail(MPDO_EINVAL, "ctx is NULL");
    CU(cudaSetDevice(c->dev));
    if (!c->built) return fail(MPDO_ESTATE, "mpdo_build_gates must come first");
    if (n_steps < 0) return fail(MPDO_EINVAL, "n_steps must be >= 0");
    if (c->forced_steps > 0) return fail(MPDO_EINVAL, "forced ranks are not supported by the graph step");
    if (!c->graph) {
        c->graph = new (std::nothrow) GraphState();
        if (!c->graph) return fail(MPDO_ENOMEM, "host allocation failed");
    }
    GraphState* g = c->graph;
    if (g->layout != c->layout || !g->exec) {
        int rc = build_graph(c, g);
        if (rc) return rc;
    }
    // The captured step has the slice products alone: a loaded state whose gauge they would
    // not resolve takes host-planned steps until its bonds have been through an SVD (one
    // step, unless a bond has no op).  So do steps all of whose bonds leave the SVD's stages
    // out, while those are captured: the host-planned step does not launch them (see
    // build_graph for what that takes).
    int first = 0;
    auto small = [&] {
        bool any = false;
        for (const auto& L : g->chunks)
            for (const Chunk& ch : L) any = any || ch.stages;
        return any && !c->mixed && use_qr32(c) && 4 * *std::max_element(c->h_dims.begin(), c->h_dims.end()) <= kPlainRows;
    };
    int rc = refresh_gauge(c);
    if (rc) return rc;
    ++c->gen;
    c->rank_steps = n_steps;
    c->rank_log.assign((size_t)c->B * n_steps * c->n_ops, 0);
    for (; first < n_steps && (wide_any(c) || small()); ++first)
        if ((rc = host_step(c, first))) return rc;
    const size_t per = (size_t)c->B * c->n_ops;
    int* d_all = nullptr;
    CU(dalloc(&d_all, std::max<size_t>(1, per * (n_steps - first))));
    for (int step = 0; step < n_steps - first; ++step) {
        cudaError_t e = cudaGraphLaunch(g->exec, c->st);
        if (e != cudaSuccess) {
            cudaFree(d_all);
            return fail(MPDO_ECUDA, std::string("graph launch: ") + cudaGetErrorString(e));
        }
        e = cudaMemcpyAsync(d_all + per * step, g->d_klog, sizeof(int) * per, cudaMemcpyDeviceToDevice, c->st);
        if (e != cudaSuccess) {
            cudaFree(d_all);
            return fail(MPDO_ECUDA, std::string("rank copy: ") + cudaGetErrorString(e));
        }
    }
    std::vector<int> all(per * (n_steps - first)), err(1);
    cudaError_t e1 = cudaMemcpyAsync(all.data(), d_all, sizeof(int) * all.size(), cudaMemcpyDeviceToHost, c->st);
    cudaError_t e2 = cudaMemcpyAsync(err.data(), g->d_error, sizeof(int), cudaMemcpyDeviceToHost, c->st);
    cudaError_t e3 = cudaMemcpyAsync(c->h_dims.data(), c->d_dims, sizeof(int) * c->h_dims.size(),
                                     cudaMemcpyDeviceToHost, c->st);
    cudaError_t e4 = cudaStreamSynchronize(c->st);
    cudaFree(d_all);
    for (cudaError_t e : {e1, e2, e3, e4})
        if (e != cudaSuccess) return fail(MPDO_ECUDA, std::string("graph step: ") + cudaGetErrorString(e));
    if (err[0]) return fail(MPDO_ECAPACITY, "graph step: more ops in flight than co-resident CTAs");
    for (int step = first; step < n_steps; ++step)
        for (int b = 0; b < c->B; ++b)
            for (int op = 0; op < c->n_ops; ++op)
                c->rank_log[((size_t)b * n_steps + step) * c->n_ops + op] =
                    all[per * (step - first) + (size_t)b * c->n_ops + op];
    return check_status_code(c);
}

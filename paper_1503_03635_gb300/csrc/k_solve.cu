// k_solve.cu -- phases (ii) and (iii) plus assignment and objective:
//   radius solve (Eq. 1 at epsilon -> 0 from predicated HIP estimates),
//   key ordinals (r_f, pi_f), greedy-MIS rounds on the implicit conflict
//   graph H-bar (Section 4.3, Algorithm 6), nearest-open-facility BFS and
//   the objective (Section 3.1).
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <vector>

#include "fl_internal.cuh"

namespace fl {

static int grid_for(int64_t items, int per_block) {
    int64_t b = (items + per_block - 1) / per_block;
    if (b < 1) b = 1;
    if (b > 152 * 32) b = 152 * 32;
    return (int)b;
}

// ------------------------------------------------------------------ frontier propagation

// Seeds: X[s] = min(X[s], val(s)); s joins the frontier when it decreases.
// With `reach`, a seed that held no value below `limit` records reach_val.
template <class V>
__global__ void k_inject(const int32_t* __restrict__ src, int64_t n_src, uint8_t* __restrict__ reach,
                         uint32_t reach_val, V limit, const uint32_t* __restrict__ lo_of, V* __restrict__ X,
                         uint32_t* __restrict__ stamp, uint32_t sv, int32_t* __restrict__ fr,
                         unsigned long long* __restrict__ n_fr) {
    __shared__ BlockAppend<8> sh;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t bb = (int64_t)blockIdx.x * blockDim.x; bb < n_src; bb += stride) {
        const int64_t i = bb + threadIdx.x;
        bool fresh = false;
        int32_t s = 0;
        if (i < n_src) {
            s = src[i];
            const V val = lo_of ? lo_of[s] : (uint32_t)s;
            const V old = atomicMin(&X[s], val);
            if (val < old) {
                if (reach && old >= limit) reach[s] = (uint8_t)reach_val;
                fresh = atomicExch(&stamp[s], sv) != sv;
            }
        }
        long long at = block_append<8>(fresh, n_fr, sh);
        if (at >= 0) fr[at] = s;
    }
}

// ------------------------------------------------------------------ multi-source BFS
// Level-synchronous BFS from a source list; X[v] = (dist << 32) | label, and
// atomicMin keeps the smallest label among the sources at the smallest
// distance.  label/dist = -1 where no source is reachable.

__global__ void k_unpack_bfs(const unsigned long long* __restrict__ X, int64_t n, int32_t* __restrict__ label,
                             int32_t* __restrict__ dist) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        unsigned long long x = X[v];
        bool none = x == ~0ULL;
        if (label) label[v] = none ? -1 : (int32_t)(x & 0xffffffffULL);
        if (dist) dist[v] = none ? -1 : (int32_t)(x >> 32);
    }
}

int msbfs(fl_graph* g, const int32_t* src_list, int64_t n_src, int32_t* label, int32_t* dist, DBuf& X,
          DBuf& stampb, DBuf* fr, DBuf& frval, int cls) {
    const int64_t n = g->n;
    cudaStream_t st = g->stream;
    if (!g->lists_ready) {
        FL_TRY(build_work_lists(g));
        g->lists_ready = 1;
    }
    if (runs_resident(g)) return msbfs_resident(g, src_list, n_src, label, dist, frval, X, cls);
    FL_TRY(dalloc(X, (size_t)n * 16));
    FL_TRY(dalloc(stampb, (size_t)n * 4));
    FL_TRY(dalloc(fr[0], (size_t)n * 4));
    FL_TRY(dalloc(fr[1], (size_t)n * 4));
    FL_TRY(dalloc(frval, (size_t)n * 8 + 64));
    Relax r;
    r.X[0] = X.p;
    r.X[1] = X.as<unsigned long long>() + n;
    r.fr[0] = fr[0].as<int32_t>();
    r.fr[1] = fr[1].as<int32_t>();
    r.frval = frval.p;
    r.stamp = stampb.as<uint32_t>();
    r.cnt = reinterpret_cast<unsigned long long*>(frval.as<char>() + (size_t)n * 8);
    r.h_cnt = &g->h_ctr->aux3;
    r.limit = ~0ULL;
    r.settle = true;  // level-synchronous: a vertex's first value is its final one
    FL_TRY(relax_begin(g, r));
    FL_CUDA(cudaMemsetAsync(r.X[0], 0xff, (size_t)n * 8, st));
    FL_CUDA(cudaMemsetAsync(r.stamp, 0, (size_t)n * 4, st));
    FL_CUDA(cudaMemsetAsync(r.cnt, 0, 64, st));
    if (n_src > 0) {
        // labels are the sources' rank ids: ties go to the smallest original
        // (or part-local) facility id whatever the internal numbering
        const uint32_t* label_of = g->rid.p ? g->rid.as<uint32_t>() : nullptr;
        FL_LAUNCH(cls, k_inject<<<grid_for(n_src, 256), 256, 0, st>>>(
                           src_list, n_src, nullptr, 0u, ~0ULL, label_of, X.as<unsigned long long>(), r.stamp, 1u,
                           r.fr[0], &r.cnt[0]));
        FL_CUDA(cudaGetLastError());
    }
    r.n_front = n_src;
    r.sv_prev = 1;
    const int64_t cap = g->sched.level_cap > 0 ? g->sched.level_cap : n + 2;
    for (uint32_t level = 0; r.n_front > 0; ++level) {
        if ((int64_t)level >= cap) FL_FAIL(FL_ETIMEOUT, "BFS reached its level cap");
        FL_TRY(relax_round(g, r, 1ULL << 32, level + 2, cls));
    }
    FL_LAUNCH(cls, k_unpack_bfs<<<grid_for(n, 256), 256, 0, st>>>(
                       static_cast<unsigned long long*>(r.X[r.cur]), n, label, dist));
    FL_CUDA(cudaGetLastError());
    return FL_OK;
}

// ------------------------------------------------------------------ BFS as one CUDA graph
// The same BFS with its level loop on the device: a CUDA graph whose
// conditional WHILE node repeats one pull level and a kernel that advances
// the level, ending the loop when a level reaches no vertex.  Values are
// updated in place: a vertex reached at level L gets stamp L, and level L
// reads only neighbours stamped L - 1, whose values are final, so no level
// sees a value written in the same level.  The level count is capped (n + 2
// levels); at the cap the loop stops with an error flag (FL_ETIMEOUT).  One
// graph launch and one synchronisation replace a launch sequence and a
// synchronisation per level.

namespace {

struct GbfsState {
    uint32_t level;
    uint32_t pad;
    unsigned long long reached;
    unsigned long long error;
};

__device__ __forceinline__ bool gbfs_front(const uint32_t* __restrict__ stamp, int32_t u, uint32_t prev) {
    return __ldg(&stamp[u]) == prev;
}

// Vertices of at most kSmallDeg neighbours: a thread each.
__global__ void __launch_bounds__(256) k_gbfs_small(const int32_t* __restrict__ list, int64_t n_list,
                                                    const int64_t* __restrict__ rowp,
                                                    const int32_t* __restrict__ cols, unsigned long long* X,
                                                    uint32_t* stamp, GbfsState* st, unsigned long long add) {
    const uint32_t L = st->level;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long cnt = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_list; i += stride) {
        const int32_t v = list[i];
        if (X[v] != ~0ULL) continue;
        unsigned long long m = ~0ULL;
        for (int64_t e = rowp[v]; e < rowp[v + 1]; ++e) {
            const int32_t u = __ldg(&cols[e]);
            if (gbfs_front(stamp, u, L - 1)) m = umin64(m, X[u]);
        }
        if (m != ~0ULL) {
            X[v] = m + add;
            stamp[v] = L;
            ++cnt;
        }
    }
    if (cnt) atomicAdd(&st->reached, cnt);
}

// Other vertices: a group of G lanes each (8 for the middle degrees, 32 for
// hubs), 32 / G vertices per warp; every lane of a warp runs every pass (the
// group reductions are warp shuffles).
template <int G>
__global__ void __launch_bounds__(256) k_gbfs_group(const int32_t* __restrict__ list, int64_t n_list,
                                                    const int64_t* __restrict__ rowp,
                                                    const int32_t* __restrict__ cols, unsigned long long* X,
                                                    uint32_t* stamp, GbfsState* st, unsigned long long add) {
    constexpr int kPerWarp = 32 / G;
    const uint32_t L = st->level;
    const int lane = lane_id(), sub = lane & (G - 1);
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned long long cnt = 0;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w * kPerWarp < n_list; w += warps) {
        const int64_t i = w * kPerWarp + lane / G;
        const int32_t v = i < n_list ? list[i] : 0;
        const bool work = i < n_list && X[v] == ~0ULL;
        unsigned long long m = ~0ULL;
        if (work)
            for (int64_t e = rowp[v] + sub; e < rowp[v + 1]; e += G) {
                const int32_t u = __ldg(&cols[e]);
                if (gbfs_front(stamp, u, L - 1)) m = umin64(m, X[u]);
            }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) m = umin64(m, __shfl_xor_sync(kFull, m, o, G));
        if (work && sub == 0 && m != ~0ULL) {
            X[v] = m + add;
            stamp[v] = L;
            ++cnt;
        }
    }
    if (cnt) atomicAdd(&st->reached, cnt);
}

// Sources: level 1, value = the source's label (distance 0).
__global__ void k_gbfs_sources(const int32_t* __restrict__ src, int64_t n_src, const uint32_t* __restrict__ lo_of,
                               unsigned long long* __restrict__ X, uint32_t* __restrict__ stamp) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_src; i += stride) {
        const int32_t s = src[i];
        atomicMin(&X[s], (unsigned long long)(lo_of ? lo_of[s] : (uint32_t)s));
        stamp[s] = 1u;
    }
}

// End of a level: stop when it reached no vertex (or at the level cap, with
// the error flag), else go on with the next level.
__global__ void k_gbfs_next(GbfsState* st, uint32_t cap, cudaGraphConditionalHandle h) {
    if (st->reached == 0) {
        cudaGraphSetConditional(h, 0);
        return;
    }
    if (st->level >= cap) {
        st->error = 1;
        cudaGraphSetConditional(h, 0);
        return;
    }
    st->level += 1;
    st->reached = 0;
    cudaGraphSetConditional(h, 1);
}

int graph_grid(int64_t items, int per_block) {
    int64_t b = (items + per_block - 1) / per_block;
    if (b < 1) b = 1;
    if (b > 152 * 32) b = 152 * 32;
    return (int)b;
}

}  // namespace

void graph_bfs_release(GraphBfs* c) {
    if (c->exec) cudaGraphExecDestroy(c->exec);
    if (c->graph) cudaGraphDestroy(c->graph);
    c->exec = nullptr;
    c->graph = nullptr;
    dfree(c->state);
}

int msbfs_graph(fl_graph* g, const int32_t* src_list, int64_t n_src, int32_t* label, int32_t* dist, DBuf& X,
                DBuf& stampb, int cls) {
    const int64_t n = g->n;
    cudaStream_t st = g->stream;
    if (!g->lists_ready) {
        FL_TRY(build_work_lists(g));
        g->lists_ready = 1;
    }
    GraphBfs* c = g->gbfs;
    FL_TRY(dalloc(X, (size_t)n * 8));
    FL_TRY(dalloc(stampb, (size_t)n * 4));
    FL_TRY(dalloc(c->state, sizeof(GbfsState)));
    unsigned long long* Xp = X.as<unsigned long long>();
    uint32_t* stamp = stampb.as<uint32_t>();
    GbfsState* state = c->state.as<GbfsState>();
    const unsigned long long add = 1ULL << 32;
    const uint32_t cap = (uint32_t)std::min<int64_t>(g->sched.level_cap > 0 ? g->sched.level_cap + 1 : n + 2,
                                                     0x7fffffff);
    // (re)build the graph when its buffers or sizes changed
    const void* key[4] = {Xp, stamp, state, g->small_list.p};
    const int64_t key_n[4] = {n, g->n_small + ((int64_t)cap << 32), g->n_mid, g->n_hubs};
    bool same = c->exec != nullptr;
    for (int i = 0; i < 4; ++i) same = same && c->key[i] == key[i] && c->key_n[i] == key_n[i];
    if (!same) {
        if (c->exec) cudaGraphExecDestroy(c->exec);
        if (c->graph) cudaGraphDestroy(c->graph);
        c->exec = nullptr;
        c->graph = nullptr;
        FL_CUDA(cudaGraphCreate(&c->graph, 0));
        cudaGraphConditionalHandle h;
        FL_CUDA(cudaGraphConditionalHandleCreate(&h, c->graph, 1, cudaGraphCondAssignDefault));
        cudaGraphNodeParams p = {};
        p.type = cudaGraphNodeTypeConditional;
        p.conditional.handle = h;
        p.conditional.type = cudaGraphCondTypeWhile;
        p.conditional.size = 1;
        cudaGraphNode_t node;
        FL_CUDA(cudaGraphAddNode(&node, c->graph, nullptr, nullptr, 0, &p));
        cudaGraph_t body = p.conditional.phGraph_out[0];
        cudaStream_t cs;
        FL_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
        cudaError_t e = cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed);
        if (e == cudaSuccess) {
            const int64_t* rowp = g->rowp.as<int64_t>();
            const int32_t* cols = g->cols.as<int32_t>();
            if (g->n_small > 0)
                k_gbfs_small<<<graph_grid(g->n_small, 256), 256, 0, cs>>>(g->small_list.as<int32_t>(), g->n_small,
                                                                          rowp, cols, Xp, stamp, state, add);
            if (g->n_mid > 0)
                k_gbfs_group<8><<<graph_grid((g->n_mid + 3) / 4, 8), 256, 0, cs>>>(
                    g->mid_list.as<int32_t>(), g->n_mid, rowp, cols, Xp, stamp, state, add);
            if (g->n_hubs > 0)
                k_gbfs_group<32><<<graph_grid(g->n_hubs, 8), 256, 0, cs>>>(g->hub_list.as<int32_t>(), g->n_hubs,
                                                                           rowp, cols, Xp, stamp, state, add);
            k_gbfs_next<<<1, 1, 0, cs>>>(state, cap, h);
            cudaGraph_t captured = body;
            e = cudaStreamEndCapture(cs, &captured);
        }
        cudaStreamDestroy(cs);
        if (e != cudaSuccess) return status_of(e, "graph BFS capture", __FILE__, __LINE__);
        FL_CUDA(cudaGraphInstantiate(&c->exec, c->graph, 0));
        for (int i = 0; i < 4; ++i) {
            c->key[i] = key[i];
            c->key_n[i] = key_n[i];
        }
    }
    FL_CUDA(cudaMemsetAsync(Xp, 0xff, (size_t)n * 8, st));
    FL_CUDA(cudaMemsetAsync(stamp, 0, (size_t)n * 4, st));
    const GbfsState init = {2u, 0u, 0ULL, 0ULL};  // sources are level 1; the loop starts at level 2
    FL_CUDA(cudaMemcpyAsync(state, &init, sizeof(init), cudaMemcpyHostToDevice, st));
    if (n_src > 0) {
        // labels are the sources' rank ids, as in msbfs
        const uint32_t* label_of = g->rid.p ? g->rid.as<uint32_t>() : nullptr;
        FL_LAUNCH(cls, k_gbfs_sources<<<grid_for(n_src, 256), 256, 0, st>>>(src_list, n_src, label_of, Xp, stamp));
        FL_CUDA(cudaGetLastError());
        cudaError_t le = cudaSuccess;
        FL_LAUNCH(cls, le = cudaGraphLaunch(c->exec, st));
        FL_CUDA(le);
    }
    FL_LAUNCH(cls, k_unpack_bfs<<<grid_for(n, 256), 256, 0, st>>>(Xp, n, label, dist));
    FL_CUDA(cudaGetLastError());
    GbfsState out;
    FL_CUDA(cudaMemcpyAsync(&out, state, sizeof(out), cudaMemcpyDeviceToHost, st));
    FL_CUDA(cudaStreamSynchronize(st));
    if (out.error) FL_FAIL(FL_ETIMEOUT, "graph BFS reached its level cap");
    return FL_OK;
}

// ------------------------------------------------------------------ radius (phase ii)

__global__ void k_check_costs(const double* __restrict__ cost, int64_t n, Counters* ctr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        double c = cost[v];
        bool ok = (c > 0.0 && c < INFINITY) || c == INFINITY;  // rejects NaN, <= 0, -inf
        if (!ok) atomicOr(&ctr->error, 1ULL);
    }
}

// Radius of facility f with opening cost c (Eq. 1 at eps -> 0): W_h =
// (#counted client entries of the hop-h group) x weight; N_j = N_{j-1} + W_j;
// G_{j+1} = G_j + N_j; r = j + (c - G_j) / N_j at the first j < L with
// G_{j+1} >= c, else L + (c - G_L) / N_L (L = last hop of the ADS of f), +inf
// if N_L = 0.  Every operation is one IEEE-754 op in this order (no
// contraction).
//
// A warp takes 32 consecutive vertices.  It reads the entries of one facility
// after the other, 32 ids per load and a window of kRadWindow entries of two
// facilities in flight; each ballot of the client flags is one word of the
// facility's client bits, kept by the facility's own lane.  Then every lane
// walks the recurrence over its own groups (a group's clients are a popcount
// of its bits), so that one FP64 instruction serves 32 facilities: at some two
// FP64 lanes per SM and cycle a warp per facility, walking on all its lanes,
// was bound by them and by the chain of four dependent loads per facility.
// Facilities that found their root read no further window.  Whole calls, a
// warp per facility against this: query at 4.2 M facilities 11.24 -> 8.72 ms
// (the kernel 4.52 -> 0.57), 16 instances of 262 k vertices 12.61 -> 8.50 ms
// (5.05 -> 0.59), R-MAT 20 solve 11.81 -> 11.08 ms.
constexpr int kRadWords = 4;
constexpr int kRadWindow = 32 * kRadWords;  // a group has at most 32 entries

// R > 1 (batches on one resident graph): R instances, instance i's costs,
// client mask and radii at offset i*n; the warps of one vertex block's R
// instances are adjacent, so its ADS rows are read from DRAM once.
template <bool kMulti>
__global__ void __launch_bounds__(256) k_radius(int64_t n, int64_t R, const double* __restrict__ cost,
                                                const uint8_t* __restrict__ client,
                                                const int64_t* __restrict__ gofs, const int64_t* __restrict__ eofs,
                                                const uint32_t* __restrict__ ginfo, const double* __restrict__ gwt,
                                                const int32_t* __restrict__ eid, double* __restrict__ r_out) {
    const int lane = lane_id();
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t nb = (n + 31) >> 5;
    for (int64_t t = (((int64_t)blockIdx.x * blockDim.x) + threadIdx.x) >> 5; t < nb * R; t += warps) {
        const int64_t blk = kMulti ? t / R : t;
        const int64_t io = kMulti ? (t - blk * R) * n : 0;  // instance offset
        const uint8_t* __restrict__ cl_of = client + io;
        const int64_t v = (blk << 5) + lane;
        const double c = v < n ? cost[io + v] : INFINITY;
        bool todo = c < INFINITY, root = false;
        int64_t gi = 0, ge = 0, e = 0;
        int left = 0, L = 0, j = 0;
        uint32_t info = 0;
        double wt = 0.0, N = 0.0, G = 0.0;
        if (todo) {
            gi = gofs[v];
            ge = gofs[v + 1];
            e = eofs[v];
            left = (int)min(eofs[v + 1] - e, (int64_t)INT32_MAX);
            info = ginfo[gi];
            wt = gwt[gi];
            L = (int)(ginfo[ge - 1] & 0xffffu);
        }
        while (const unsigned live = __ballot_sync(kFull, todo)) {
            uint32_t bits[kRadWords + 1];
#pragma unroll
            for (int q = 0; q <= kRadWords; ++q) bits[q] = 0u;
            for (unsigned rest = live; rest;) {
                const int b0 = __ffs(rest) - 1;
                rest &= rest - 1;
                const int b1 = rest ? __ffs(rest) - 1 : 32;
                rest &= rest - 1;
                const int32_t* __restrict__ p0 = eid + __shfl_sync(kFull, e, b0);
                const int32_t* __restrict__ p1 = eid + __shfl_sync(kFull, e, b1 & 31);
                const int n0 = __shfl_sync(kFull, left, b0);
                const int n1l = __shfl_sync(kFull, left, b1 & 31);
                const int n1 = b1 < 32 ? n1l : 0;
                int32_t id0[kRadWords], id1[kRadWords];
#pragma unroll
                for (int q = 0; q < kRadWords; ++q) {
                    const int at = 32 * q + lane;
                    id0[q] = at < n0 ? __ldg(&p0[at]) : -1;
                    id1[q] = at < n1 ? __ldg(&p1[at]) : -1;
                }
                bool f0[kRadWords], f1[kRadWords];
#pragma unroll
                for (int q = 0; q < kRadWords; ++q) {
                    f0[q] = id0[q] >= 0 && __ldg(&cl_of[id0[q]]) != 0;
                    f1[q] = id1[q] >= 0 && __ldg(&cl_of[id1[q]]) != 0;
                }
#pragma unroll
                for (int q = 0; q < kRadWords; ++q) {
                    const unsigned w0 = __ballot_sync(kFull, f0[q]), w1 = __ballot_sync(kFull, f1[q]);
                    if (lane == b0) bits[q] = w0;
                    if (lane == b1) bits[q] = w1;
                }
            }
            int off = 0;  // entries of the window walked
            while (todo) {
                const int hop = (int)(info & 0xffffu), cnt = (int)((info >> 16) & 0xffu), counted = (int)(info >> 24);
                if (off + cnt > kRadWindow) break;  // the group ends in the next window
                const double w = wt;
                if (++gi < ge) {
                    info = ginfo[gi];
                    wt = gwt[gi];
                }
                uint32_t lo = 0, hi = 0;
#pragma unroll
                for (int q = 0; q < kRadWords; ++q)
                    if ((off >> 5) == q) {
                        lo = bits[q];
                        hi = bits[q + 1];
                    }
                const uint32_t own = __funnelshift_r(lo, hi, off & 31);
                const int clients = __popc(own & (counted >= 32 ? ~0u : (1u << counted) - 1u));
                off += cnt;
                for (; j < hop; ++j) {  // hops without new entries: W_j = 0
                    const double Gn = __dadd_rn(G, N);
                    if (Gn >= c) break;
                    G = Gn;
                }
                if (j < hop) {
                    root = true;
                    todo = false;
                    break;
                }
                N = __dadd_rn(N, __dmul_rn((double)clients, w));
                if (j < L) {
                    const double Gn = __dadd_rn(G, N);
                    if (Gn >= c) {
                        root = true;
                        todo = false;
                        break;
                    }
                    G = Gn;
                }
                ++j;
                if (gi >= ge) {  // the last group: its hop is L
                    j = L;
                    root = N > 0.0;
                    todo = false;
                }
            }
            e += off;
            left -= off;
        }
        if (v < n) r_out[io + v] = root ? __dadd_rn((double)j, __ddiv_rn(__dsub_rn(c, G), N)) : INFINITY;
    }
}

// The solve's opening costs are finite and > 0, or +inf (not a facility).
int check_costs(fl_solve* s) {
    fl_graph* g = s->g;
    cudaStream_t st = g->stream;
    FL_CUDA(cudaMemsetAsync(g->ctr.p, 0, sizeof(Counters), st));
    FL_LAUNCH(kProfRadius, k_check_costs<<<grid_for(g->n, 256), 256, 0, st>>>(s->cost.as<double>(), g->n, g->ctr.as<Counters>()));
    FL_CUDA(cudaGetLastError());
    FL_TRY(read_counters(g));
    if (g->h_ctr->error) FL_FAIL(FL_EINVAL, "open_cost must be finite and > 0 for facilities, +inf otherwise");
    return FL_OK;
}

int compute_radii(fl_solve* s) {
    fl_graph* g = s->g;
    cudaStream_t st = g->stream;
    FL_TRY(check_costs(s));
    FL_LAUNCH(kProfRadius, k_radius<false><<<grid_for((g->n + 31) / 32, 8), 256, 0, st>>>(g->n, 1, s->cost.as<double>(), s->client.as<uint8_t>(),
                                               g->gofs.as<int64_t>(), g->eofs.as<int64_t>(), g->ginfo.as<uint32_t>(),
                                               g->gwt.as<double>(), g->eid.as<int32_t>(), s->radii.as<double>()));
    FL_CUDA(cudaGetLastError());
    return FL_OK;
}

// Radii of R instances on the built graph src (batches): cost, client and
// radii are R*n arrays, instance-major.  Runs on g's stream with g's
// counters (src is only read).
int compute_radii_multi(const fl_graph* src, fl_graph* g, int64_t R, const double* cost, const uint8_t* client,
                        double* radii) {
    cudaStream_t st = g->stream;
    const int64_t n = src->n;
    FL_CUDA(cudaMemsetAsync(g->ctr.p, 0, sizeof(Counters), st));
    FL_LAUNCH(kProfRadius, k_check_costs<<<grid_for(n * R, 256), 256, 0, st>>>(cost, n * R, g->ctr.as<Counters>()));
    FL_CUDA(cudaGetLastError());
    FL_TRY(read_counters(g));
    if (g->h_ctr->error) FL_FAIL(FL_EINVAL, "open_cost must be finite and > 0 for facilities, +inf otherwise");
    FL_LAUNCH(kProfRadius, k_radius<true><<<grid_for((n + 31) / 32 * R, 8), 256, 0, st>>>(
                               n, R, cost, client, src->gofs.as<int64_t>(), src->eofs.as<int64_t>(),
                               src->ginfo.as<uint32_t>(), src->gwt.as<double>(), src->eid.as<int32_t>(), radii));
    FL_CUDA(cudaGetLastError());
    return FL_OK;
}

// ------------------------------------------------------------------ keys (r_f, pi_f)

// Up to kRankMax candidates are ordered by counting (k_count_keys), more by the
// radix sort.
constexpr int64_t kRankMax = 16384;
constexpr int64_t kTieRun = 64;  // longer runs of equal keys are not put in order by one thread

__global__ void k_candidates(const double* __restrict__ r, int64_t n, uint64_t seed,
                             IdMap ids, uint64_t* __restrict__ hi,
                             uint64_t* __restrict__ lo, uint32_t* __restrict__ val, uint8_t* __restrict__ state,
                             Counters* ctr) {
    // which radius bits vary: OR of the words and of their complements, per
    // block in shared memory, then one global OR per block
    __shared__ unsigned long long bits[2];
    if (threadIdx.x < 2) bits[threadIdx.x] = 0;
    __syncthreads();
    __shared__ BlockAppend<8> sh;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t bb = (int64_t)blockIdx.x * blockDim.x; bb < n; bb += stride) {
        int64_t f = bb + threadIdx.x;
        bool cand = false;
        double rf = 0.0;
        if (f < n) {
            rf = r[f];
            cand = rf < INFINITY;
            state[f] = cand ? 0 : 3;
        }
        long long at = block_append<8>(cand, &ctr->aux0, sh);
        const uint64_t h = cand ? (uint64_t)__double_as_longlong(rf) : 0;  // r >= 0: bit order = numeric order
        if (at >= 0) {
            hi[at] = h;
            if (at < kRankMax) lo[at] = facility_priority(seed, rank_id(ids, f));
            val[at] = (uint32_t)f;
        }
        if (__ballot_sync(kFull, cand)) {
            uint64_t w[2] = {h, cand ? ~h : 0};
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const unsigned a = __reduce_or_sync(kFull, (unsigned)w[q]);
                const unsigned b = __reduce_or_sync(kFull, (unsigned)(w[q] >> 32));
                w[q] = ((uint64_t)b << 32) | a;
            }
            if (lane_id() == 0)
                for (int q = 0; q < 2; ++q)
                    if (w[q] & ~bits[q]) atomicOr(&bits[q], (unsigned long long)w[q]);
        }
    }
    __syncthreads();
    if (threadIdx.x < 2 && bits[threadIdx.x]) atomicOr(threadIdx.x ? &ctr->key_orn : &ctr->key_or, bits[threadIdx.x]);
}

// Few candidates: each one's place in key order is the number of keys below
// its own.  A block counts for 64 candidates, two per lane, over its share of
// the keys (blockIdx.y of gridDim.y shares), staged in shared memory a tile at
// a time; its warps share the tile (every lane reads the same key: a
// broadcast).  Equal keys (parts of a batch with equal part-local ids) keep
// their input order.  Quadratic, but no pass over memory but the keys: bound by
// integer compares, one borrow chain over (radius, priority, index) each, and
// by how evenly the blocks fill the SMs (10^4 keys: 101 us with one share of
// all keys, 157 blocks on 152 SMs, and compares word by word; 41 us now).
constexpr int kRankTile = 512;

// -1 when (hi, lo, at) is below (h, l, i), else 0.
__device__ __forceinline__ int key_below(uint64_t hi, uint64_t lo, unsigned at, uint64_t h, uint64_t l, unsigned i) {
    int r;
    asm("{\n\t"
        ".reg .u32 t, a, b, c, d;\n\t"
        "sub.cc.u32 t, %1, %2;\n\t"
        "mov.b64 {a, b}, %3;\n\t"
        "mov.b64 {c, d}, %4;\n\t"
        "subc.cc.u32 t, a, c;\n\t"
        "subc.cc.u32 t, b, d;\n\t"
        "mov.b64 {a, b}, %5;\n\t"
        "mov.b64 {c, d}, %6;\n\t"
        "subc.cc.u32 t, a, c;\n\t"
        "subc.cc.u32 t, b, d;\n\t"
        "subc.u32 %0, 0, 0;\n\t"
        "}"
        : "=r"(r)
        : "r"(at), "r"(i), "l"(lo), "l"(l), "l"(hi), "l"(h));
    return r;
}

__global__ void __launch_bounds__(256) k_count_keys(const uint64_t* __restrict__ hi, const uint64_t* __restrict__ lo,
                                                    int m, unsigned* __restrict__ place) {
    __shared__ ulonglong2 key[kRankTile];
    __shared__ int below[64];
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const int i0 = blockIdx.x * 64 + lane, i1 = i0 + 32;
    const uint64_t h0 = i0 < m ? hi[i0] : 0, l0 = i0 < m ? lo[i0] : 0;
    const uint64_t h1 = i1 < m ? hi[i1] : 0, l1 = i1 < m ? lo[i1] : 0;
    const int t0 = (int)((int64_t)m * blockIdx.y / gridDim.y), t1 = (int)((int64_t)m * (blockIdx.y + 1) / gridDim.y);
    int c0 = 0, c1 = 0;
    if (threadIdx.x < 64) below[threadIdx.x] = 0;
    for (int t = t0; t < t1; t += kRankTile) {
        const int cnt = min(kRankTile, t1 - t);
        __syncthreads();
        for (int j = threadIdx.x; j < cnt; j += 256) key[j] = make_ulonglong2(hi[t + j], lo[t + j]);
        __syncthreads();
#pragma unroll 4
        for (int j = warp; j < cnt; j += 8) {
            const ulonglong2 k = key[j];
            c0 -= key_below(k.x, k.y, (unsigned)(t + j), h0, l0, (unsigned)i0);
            c1 -= key_below(k.x, k.y, (unsigned)(t + j), h1, l1, (unsigned)i1);
        }
    }
    atomicAdd(&below[lane], c0);
    atomicAdd(&below[lane + 32], c1);
    __syncthreads();
    if (threadIdx.x < 64 && blockIdx.x * 64 + threadIdx.x < m)
        atomicAdd(&place[blockIdx.x * 64 + threadIdx.x], (unsigned)below[threadIdx.x]);
}

__global__ void k_place_keys(const unsigned* __restrict__ place, const uint32_t* __restrict__ val, int m,
                             uint32_t* __restrict__ sorted) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m) sorted[place[i]] = val[i];
}

__device__ __forceinline__ uint64_t priority_of(uint64_t seed, const IdMap& ids, uint32_t f) {
    return facility_priority(seed, rank_id(ids, (int64_t)f));
}

// Keys sorted by the bits from `shift` up (and, with kByPrio, by the top half
// of the priority below them): put each run that these bits leave equal in
// the order of the whole key (r_f, pi_f), one thread per run.  A run longer
// than `longest` is left alone and reported.
template <bool kByPrio>
__global__ void k_order_runs(uint64_t* key, uint32_t* val, int64_t m, int shift, int64_t longest, uint64_t seed,
                             IdMap ids, Counters* ctr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    auto same = [&](int64_t i, int64_t j) {
        if ((key[i] >> shift) != (key[j] >> shift)) return false;
        return !kByPrio || (priority_of(seed, ids, val[i]) >> 32) == (priority_of(seed, ids, val[j]) >> 32);
    };
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i + 1 < m; i += stride) {
        if (!same(i, i + 1) || (i > 0 && same(i - 1, i))) continue;
        int64_t end = i + 2;
        while (end < m && end - i <= longest && same(i, end)) ++end;
        if (end - i > longest) {
            atomicOr(&ctr->key_ties, 1ULL);
            continue;
        }
        for (int64_t a = i + 1; a < end; ++a) {
            const uint64_t k = key[a];
            const uint32_t v = val[a];
            const uint64_t p = priority_of(seed, ids, v);
            int64_t b = a;
            for (; b > i; --b) {
                const uint64_t kb = key[b - 1];
                const uint32_t vb = val[b - 1];
                if (kb < k || (kb == k && priority_of(seed, ids, vb) <= p)) break;
                key[b] = kb;
                val[b] = vb;
            }
            key[b] = k;
            val[b] = v;
        }
    }
}

// Are neighbours with equal radii out of the order of their priorities?
__global__ void k_tie_order(const uint64_t* __restrict__ key, const uint32_t* __restrict__ val, int64_t m,
                            uint64_t seed, IdMap ids, Counters* ctr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    bool bad = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i + 1 < m; i += stride)
        bad |= key[i] == key[i + 1] && priority_of(seed, ids, val[i]) > priority_of(seed, ids, val[i + 1]);
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&ctr->key_ties, 2ULL);
}

// Half of the priorities: their bits from `shift` up.
__global__ void k_prio_keys(const uint32_t* __restrict__ val, int64_t m, uint64_t seed, IdMap ids, int shift,
                            uint32_t* __restrict__ key) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride)
        key[i] = (uint32_t)(priority_of(seed, ids, val[i]) >> shift);
}

__global__ void k_radius_keys(const uint32_t* __restrict__ val, int64_t m, const double* __restrict__ r,
                              uint64_t* __restrict__ key) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride)
        key[i] = (uint64_t)__double_as_longlong(r[val[i]]);
}

__global__ void k_ordinals(const uint32_t* __restrict__ sorted_f, int64_t m, const double* __restrict__ r,
                           const int32_t* __restrict__ ecc_ub, uint32_t* __restrict__ ord,
                           int32_t* __restrict__ fac_by_ord, int32_t* __restrict__ bcap, int32_t* __restrict__ ulist,
                           unsigned long long* __restrict__ bmax) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int32_t mx = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) {
        int32_t f = (int32_t)sorted_f[i];
        ord[f] = (uint32_t)i;
        fac_by_ord[i] = f;
        ulist[i] = f;
        // ball radius floor(r_f), capped by an eccentricity bound (same ball)
        double fl = floor(r[f]);
        int32_t cap = ecc_ub[f];
        int32_t b = fl >= (double)cap ? cap : (int32_t)fl;
        bcap[f] = b;
        mx = max(mx, b);
    }
    // the largest ball radius: one atomic per block
    __shared__ int s_max;
    if (threadIdx.x == 0) s_max = 0;
    __syncthreads();
    mx = (int32_t)__reduce_max_sync(kFull, (unsigned)mx);
    if (lane_id() == 0 && mx > 0) atomicMax(&s_max, mx);
    __syncthreads();
    if (threadIdx.x == 0 && s_max > 0) atomicMax(bmax, (unsigned long long)s_max);
}

// ------------------------------------------------------------------ MIS rounds (phase iii)

// Bucket sizes by ball radius, the largest radius, and (for a graph made of
// parts) each part's largest radius, gathered per block in shared memory (radii
// and parts beyond its tables go to the global counts at once): the undecided
// are in key order, so a warp holds most radii and parts, and its atomics on a
// few words took 120 us for 4.2 M facilities in 16 parts.
constexpr int kBuckets = 1024;
constexpr int kPartTab = 1024;

__global__ void __launch_bounds__(256) k_bucket_count(const int32_t* __restrict__ ulist, int64_t n_u,
                                                      const int32_t* __restrict__ bcap, int32_t* __restrict__ bcount,
                                                      unsigned long long* __restrict__ tmax,
                                                      const int32_t* __restrict__ vpart, int32_t* __restrict__ part_T,
                                                      int64_t n_parts) {
    __shared__ int s_cnt[kBuckets];
    __shared__ int s_part[kPartTab];
    __shared__ int s_max;
    for (int i = threadIdx.x; i < kBuckets; i += blockDim.x) s_cnt[i] = 0;
    if (vpart)
        for (int i = threadIdx.x; i < kPartTab; i += blockDim.x) s_part[i] = -1;
    if (threadIdx.x == 0) s_max = 0;
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int32_t mx = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_u; i += stride) {
        const int32_t f = ulist[i];
        const int32_t b = bcap[f];
        mx = max(mx, b);
        if (b < kBuckets) atomicAdd(&s_cnt[b], 1);
        else atomicAdd(&bcount[b], 1);
        if (vpart) {
            const int32_t p = vpart[f];
            if (p >= kPartTab) atomicMax(&part_T[p], b);
            else if (s_part[p] < b) atomicMax(&s_part[p], b);
        }
    }
    mx = (int32_t)__reduce_max_sync(kFull, (unsigned)mx);
    if (lane_id() == 0) atomicMax(&s_max, mx);
    __syncthreads();
    if (threadIdx.x == 0) atomicMax(tmax, (unsigned long long)s_max);
    for (int i = threadIdx.x; i < min(s_max + 1, kBuckets); i += blockDim.x)
        if (s_cnt[i]) atomicAdd(&bcount[i], s_cnt[i]);
    if (vpart)
        for (int i = threadIdx.x; i < kPartTab && i < n_parts; i += blockDim.x)
            if (s_part[i] >= 0) atomicMax(&part_T[i], s_part[i]);
}

// Facilities to their bucket's range: a block counts kScatter per thread by
// bucket, reserves its places with one atomic per bucket and writes them.
constexpr int kScatter = 8;

__global__ void __launch_bounds__(256) k_bucket_scatter(const int32_t* __restrict__ ulist, int64_t n_u,
                                                        const int32_t* __restrict__ bcap,
                                                        int32_t* __restrict__ cursor, int32_t* __restrict__ ubuck) {
    __shared__ int s_cnt[kBuckets];  // counts, then first places
    __shared__ int s_top;
    const int64_t tile = (int64_t)blockDim.x * kScatter;
    for (int64_t t = blockIdx.x * tile; t < n_u; t += gridDim.x * tile) {
        __syncthreads();
        for (int i = threadIdx.x; i < kBuckets; i += blockDim.x) s_cnt[i] = 0;
        if (threadIdx.x == 0) s_top = 0;
        __syncthreads();
        int32_t f[kScatter], b[kScatter], at[kScatter];
        int top = 0;
#pragma unroll
        for (int j = 0; j < kScatter; ++j) {
            const int64_t i = t + (int64_t)j * blockDim.x + threadIdx.x;
            f[j] = i < n_u ? ulist[i] : -1;
            b[j] = f[j] >= 0 ? bcap[f[j]] : -1;
            at[j] = 0;
            if (b[j] >= kBuckets) at[j] = atomicAdd(&cursor[b[j]], 1);
            else if (b[j] >= 0) at[j] = atomicAdd(&s_cnt[b[j]], 1);
            if (b[j] < kBuckets) top = max(top, b[j]);
        }
        top = (int)__reduce_max_sync(kFull, (unsigned)top);
        if (lane_id() == 0) atomicMax(&s_top, top);
        __syncthreads();
        for (int i = threadIdx.x; i <= s_top; i += blockDim.x)
            if (s_cnt[i]) s_cnt[i] = atomicAdd(&cursor[i], s_cnt[i]);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kScatter; ++j)
            if (f[j] >= 0) ubuck[(b[j] < kBuckets ? s_cnt[b[j]] : 0) + at[j]] = f[j];
    }
}

// Gather seeds: every client covered in this round's cover sweep (values C)
// starts the gather (values X, all unset) with 0 if already claimed, else 1 +
// (smallest key of an undecided facility covering it); mval keeps that smallest
// key for the claim step.
__global__ void k_gather_seed(const int32_t* __restrict__ touched, const unsigned long long* __restrict__ n_touched,
                              const uint8_t* __restrict__ client, const uint8_t* __restrict__ claimed,
                              const uint32_t* __restrict__ C, uint32_t* __restrict__ X, uint32_t* __restrict__ mval,
                              uint32_t* __restrict__ stamp, uint32_t sv, int32_t* __restrict__ fr,
                              unsigned long long* __restrict__ n_fr) {
    __shared__ BlockAppend<8> sh;
    const int64_t n = (int64_t)*n_touched;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t bb = (int64_t)blockIdx.x * blockDim.x; bb < n; bb += stride) {
        int64_t i = bb + threadIdx.x;
        bool seed = false;
        int32_t v = 0;
        if (i < n) {
            v = touched[i];
            if (client[v]) {
                const uint32_t m = C[v];
                mval[v] = m;
                X[v] = claimed[v] ? 0u : m + 1u;
                stamp[v] = sv;
                seed = true;
            }
        }
        long long at = block_append<8>(seed, n_fr, sh);
        if (at >= 0) fr[at] = v;
    }
}

// Facilities whose ball radius is b read the minimum over their ball after
// b gather rounds: 0 -> a client of the ball is claimed (dead); own key + 1
// -> smallest key among all conflicting undecided facilities (joins S).
__global__ void k_decide(const int32_t* __restrict__ fl, int64_t m, const uint32_t* __restrict__ X,
                         const uint32_t* __restrict__ ord, uint8_t* __restrict__ state, Counters* ctr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) {
        int32_t f = fl[i];
        const uint32_t x = X[f];
        if (x == 0xffffffffu) atomicOr(&ctr->error, 8ULL);  // a candidate's ball holds no client (cannot happen)
        else if (x == 0) state[f] = 2;
        else if (x == ord[f] + 1u) state[f] = 1;
    }
}

// Clients of this round's winners' balls become claimed; with `kr`, each
// newly claimed client is a seed (kr = 1) of the round's kill sweep, and
// *n_new counts them.
__global__ void k_claim(const int32_t* __restrict__ touched, const unsigned long long* __restrict__ n_touched,
                        const uint8_t* __restrict__ client, uint8_t* __restrict__ claimed,
                        const uint32_t* __restrict__ mval, const int32_t* __restrict__ fac_by_ord,
                        const uint8_t* __restrict__ state, uint8_t* __restrict__ kr,
                        unsigned long long* __restrict__ n_new) {
    const int64_t n = (int64_t)*n_touched;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned fresh = 0;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
        const int64_t i = base + lane_id();
        bool now = false;
        if (i < n) {
            const int32_t v = touched[i];
            if (client[v] && !claimed[v] && state[fac_by_ord[mval[v]]] == 1) {
                claimed[v] = 1;
                if (kr) kr[v] = 1;
                now = true;
            }
        }
        fresh += __popc(__ballot_sync(kFull, now));
    }
    block_count(lane_id() == 0 ? fresh : 0u, n_new);
}

// Kill sweep decision: an undecided facility with a client claimed in this
// round within its ball radius (kr[f] = 1 + that distance <= B_f + 1) can no
// longer join S.
__global__ void k_kill(const int32_t* __restrict__ ulist, int64_t n_u, const uint8_t* __restrict__ kr,
                       const int32_t* __restrict__ bcap, uint8_t* __restrict__ state) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_u; i += stride) {
        const int32_t f = ulist[i];
        const uint32_t k = kr[f];
        if (k != 0 && (int64_t)k <= (int64_t)bcap[f] + 1) state[f] = 2;
    }
}

__global__ void k_compact_undecided(const int32_t* __restrict__ ulist, int64_t n_u, const uint8_t* __restrict__ state,
                                    int32_t* __restrict__ out, unsigned long long* __restrict__ n_out) {
    __shared__ BlockAppend<8> sh;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t bb = (int64_t)blockIdx.x * blockDim.x; bb < n_u; bb += stride) {
        int64_t i = bb + threadIdx.x;
        int32_t f = i < n_u ? ulist[i] : 0;
        bool keep = i < n_u && state[f] == 0;
        long long at = block_append<8>(keep, n_out, sh);
        if (at >= 0) out[at] = f;
    }
}

__global__ void k_open_list(const uint8_t* __restrict__ state, int64_t n, uint8_t* __restrict__ open,
                            int32_t* __restrict__ list, unsigned long long* __restrict__ n_list) {
    __shared__ BlockAppend<8> sh;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t bb = (int64_t)blockIdx.x * blockDim.x; bb < n; bb += stride) {
        int64_t v = bb + threadIdx.x;
        bool is_open = v < n && state[v] == 1;
        if (v < n) open[v] = is_open ? 1 : 0;
        long long at = block_append<8>(is_open, n_list, sh);
        if (at >= 0) list[at] = (int32_t)v;
    }
}

// Candidates (finite r_f) sorted by the key (r_f, pi_f): *sorted holds their
// ids in key order, s->state is 0 for a candidate and 3 otherwise.
//
// Many candidates: radix sort by the leading bits of r_f that vary, as many
// as tell most of them apart (log2 m + 16), then put the few short runs that
// are left in order.  Costs that repeat give runs of equal radii of any
// length: then the top half of pi_f is sorted first and r_f by all its varying
// bits after it (each pass keeps the order of the one before), and again the
// runs that are left are put in order.  Those are a few candidates long, but
// in a union of many parts a local id has the same pi_f in all of them: a run
// above kTieRun is left as it is if it holds one priority, or else (two local
// ids that agree in the top half) everything is sorted by the whole of pi_f.
// 40,000 equal parts of 40 vertices: 40 ms a batch with the runs put in order by
// one thread each, 6.9 now; 100,000 of 20 vertices 89 and 7.5.
//
// known: the number of candidates when the caller has it (else -1); a few known
// ones are ordered without a look by the host.
int sort_candidates(fl_solve* s, int64_t* m_out, const uint32_t** sorted, int64_t known) {
    fl_graph* g = s->g;
    const int64_t n = g->n;
    cudaStream_t st = g->stream;
    FL_TRY(dalloc(s->state, (size_t)n));
    FL_TRY(dalloc(s->key_hi, (size_t)n * 8));
    FL_TRY(dalloc(s->key_lo, (size_t)n * 8));
    FL_TRY(dalloc(s->key_val, (size_t)n * 4));
    FL_TRY(dalloc(s->key_alt, (size_t)n * 12));
    SortPairs<uint64_t> p;
    p.key[0] = s->key_hi.as<uint64_t>();
    p.key[1] = s->key_alt.as<uint64_t>();
    p.val[0] = s->key_val.as<uint32_t>();
    p.val[1] = reinterpret_cast<uint32_t*>(p.key[1] + n);
    Counters* ctr = g->ctr.as<Counters>();
    FL_CUDA(cudaMemsetAsync(g->ctr.p, 0, sizeof(Counters), st));
    const IdMap ids = idmap_of(g);
    FL_LAUNCH(kProfKeys, k_candidates<<<grid_for(n, 256), 256, 0, st>>>(s->radii.as<double>(), n, g->seed, ids,
                                                   p.key[0], s->key_lo.as<uint64_t>(), p.val[0],
                                                   s->state.as<uint8_t>(), ctr));
    const bool told = known >= 0 && known <= kRankMax;
    if (!told) FL_TRY(read_counters(g));
    const int64_t m = told ? known : (int64_t)g->h_ctr->aux0;
    s->n_cand = m;
    *m_out = m;
    *sorted = p.val[0];
    if (m <= 1) return FL_OK;
    if (m <= kRankMax) {
        unsigned* place = reinterpret_cast<unsigned*>(p.key[1]);
        const int groups = (int)((m + 63) / 64);
        FL_CUDA(cudaMemsetAsync(place, 0, (size_t)m * 4, st));
        FL_LAUNCH(kProfKeys, k_count_keys<<<dim3(groups, count_shares(m)), 256, 0, st>>>(
                                 p.key[0], s->key_lo.as<uint64_t>(), (int)m, place));
        FL_LAUNCH(kProfKeys, k_place_keys<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(place, p.val[0], (int)m,
                                                                                      p.val[1]));
        FL_CUDA(cudaGetLastError());
        *sorted = p.val[1];
        return FL_OK;
    }
    const uint64_t varying = g->h_ctr->key_or & g->h_ctr->key_orn;
    int shift[kSortDigits];
    int lg = 0;
    while ((1LL << lg) < m) ++lg;
    bool ties = varying == 0;
    if (!ties) {
        const int nd = digit_windows(varying, lg + 16, shift);
        FL_TRY(sort_pairs(p, m, shift, nd, st, g->scratch, kProfKeys, &ctr->error));
        FL_LAUNCH(kProfKeys, k_order_runs<false><<<grid_for(m, 256), 256, 0, st>>>(p.key[p.cur], p.val[p.cur], m,
                                                                                  shift[0], 16, g->seed, ids, ctr));
        FL_CUDA(cudaGetLastError());
        FL_TRY(read_counters(g));
        if (g->h_ctr->error) FL_FAIL(FL_ETIMEOUT, "candidate keys: a sort's wait ran out");
        ties = g->h_ctr->key_ties != 0;
    }
    // stable passes by the halves of the priority (both, or the top one), then by the radius
    auto sort_ties = [&](bool both) -> int {
        SortPairs<uint32_t> q;
        q.key[0] = s->key_lo.as<uint32_t>();
        q.key[1] = q.key[0] + n;
        q.val[0] = p.val[p.cur];
        q.val[1] = p.val[p.cur ^ 1];
        for (int half = both ? 0 : 1; half < 2; ++half) {
            FL_LAUNCH(kProfKeys, k_prio_keys<<<grid_for(m, 256), 256, 0, st>>>(q.val[q.cur], m, g->seed, ids, 32 * half,
                                                                               q.key[q.cur]));
            FL_TRY(sort_pairs(q, m, shift, digit_windows(0xffffffffULL, 0, shift), st, g->scratch, kProfKeys,
                              &ctr->error));
        }
        p.val[0] = q.val[q.cur];
        p.val[1] = q.val[q.cur ^ 1];
        p.cur = 0;
        FL_LAUNCH(kProfKeys, k_radius_keys<<<grid_for(m, 256), 256, 0, st>>>(p.val[0], m, s->radii.as<double>(),
                                                                             p.key[0]));
        return sort_pairs(p, m, shift, digit_windows(varying, 0, shift), st, g->scratch, kProfKeys, &ctr->error);
    };
    if (ties) {
        FL_TRY(sort_ties(false));
        FL_CUDA(cudaMemsetAsync(&ctr->key_ties, 0, 8, st));
        FL_LAUNCH(kProfKeys, k_order_runs<true><<<grid_for(m, 256), 256, 0, st>>>(p.key[p.cur], p.val[p.cur], m, 0,
                                                                                 kTieRun, g->seed, ids, ctr));
        FL_CUDA(cudaGetLastError());
        FL_TRY(read_counters(g));
        if (g->h_ctr->error) FL_FAIL(FL_ETIMEOUT, "candidate keys: a sort's wait ran out");
        if (g->h_ctr->key_ties) {  // long runs
            FL_LAUNCH(kProfKeys, k_tie_order<<<grid_for(m, 256), 256, 0, st>>>(p.key[p.cur], p.val[p.cur], m, g->seed,
                                                                              ids, ctr));
            FL_CUDA(cudaGetLastError());
            FL_TRY(read_counters(g));
            if (g->h_ctr->key_ties & 2ULL) {
                FL_TRY(sort_ties(true));
                FL_TRY(read_counters(g));
            }
            if (g->h_ctr->error) FL_FAIL(FL_ETIMEOUT, "candidate keys: a sort's wait ran out");
        }
    }
    *sorted = p.val[p.cur];
    return FL_OK;
}

// Keys: candidates sorted by (r_f, pi_f) -> ordinals, ball radii and the list
// of the undecided (s->ulist).  cnt = the counters behind s->frval, cleared:
// cnt[0], cnt[1] frontier counts; cnt[2] changed count (dense rounds); cnt[3]
// undecided; cnt[4] largest ball radius; cnt[5] open list; cnt[6] touched.
// All scratch is solve-owned and grow-only: a cudaFree per solve would
// synchronise the whole device (and stall other solves on other streams).
static int candidate_keys(fl_solve* s, int64_t known, int64_t* m, unsigned long long** cnt) {
    fl_graph* g = s->g;
    const int64_t n = g->n;
    cudaStream_t st = g->stream;
    FL_TRY(dalloc(s->ord, (size_t)n * 4));
    FL_TRY(dalloc(s->fac_by_ord, (size_t)n * 4));
    FL_TRY(dalloc(s->bcap, (size_t)n * 4));
    FL_TRY(dalloc(s->state, (size_t)n));
    FL_TRY(dalloc(s->frval, (size_t)n * 8 + 64));
    FL_TRY(dalloc(s->ulist, (size_t)n * 4 * 2));
    FL_TRY(dalloc(s->open, (size_t)n));
    s->mis_log.clear();
    *cnt = reinterpret_cast<unsigned long long*>(s->frval.as<char>() + (size_t)n * 8);
    const uint32_t* sorted = nullptr;
    FL_TRY(sort_candidates(s, m, &sorted, known));
    FL_CUDA(cudaMemsetAsync(*cnt, 0, 64, st));
    if (*m > 0) {
        FL_LAUNCH(kProfKeys, k_ordinals<<<grid_for(*m, 256), 256, 0, st>>>(
                                 sorted, *m, s->radii.as<double>(), g->ecc_ub.as<int32_t>(), s->ord.as<uint32_t>(),
                                 s->fac_by_ord.as<int32_t>(), s->bcap.as<int32_t>(), s->ulist.as<int32_t>(),
                                 &(*cnt)[4]));
    }
    FL_CUDA(cudaGetLastError());
    return FL_OK;
}

// The selection of `known` candidates on a graph with work items, queued
// without a look by the host: its open set goes into acc (uint8, OR) and its
// outcome into *outcome when the device gets there (mis_resident_queue).
// *queued = false: not for this path.
int open_facilities_queued(fl_solve* s, int64_t known, uint8_t* acc, int* outcome, bool* queued) {
    *queued = false;
    if (!s->g->lists_ready || !runs_resident(s->g) || known > kRankMax) return FL_OK;
    int64_t m = 0;
    unsigned long long* cnt = nullptr;
    FL_TRY(candidate_keys(s, known, &m, &cnt));
    FL_TRY(mis_resident_queue(s, m, acc, outcome));
    *queued = true;
    return FL_OK;
}

int open_facilities(fl_solve* s) {
    fl_graph* g = s->g;
    const int64_t n = g->n;
    cudaStream_t st = g->stream;
    int64_t m = 0;
    unsigned long long* cnt = nullptr;
    FL_TRY(candidate_keys(s, -1, &m, &cnt));
    int32_t* ulist[2] = {s->ulist.as<int32_t>(), s->ulist.as<int32_t>() + n};
    if (!g->lists_ready) {
        FL_TRY(build_work_lists(g));
        g->lists_ready = 1;
    }
    if (runs_resident(g)) {
        bool done = false;
        FL_TRY(mis_resident(s, m, &done));
        if (done) return FL_OK;
    }
    FL_TRY(dalloc(s->claimed, (size_t)n));
    FL_TRY(dalloc(s->X, (size_t)n * 16));          // two value buffers of the cover, two of the gather
    FL_TRY(dalloc(s->stamp, (size_t)n * 4));
    FL_TRY(dalloc(s->mval, (size_t)n * 4));
    FL_TRY(dalloc(s->fr[0], (size_t)n * 4));
    FL_TRY(dalloc(s->fr[1], (size_t)n * 4));
    FL_TRY(dalloc(s->touched, (size_t)n * 4));
    FL_TRY(dalloc(s->ubuck, (size_t)n * 4));
    FL_TRY(dalloc(s->reach, (size_t)n));
    FL_TRY(dalloc(s->kill, (size_t)n));
    unsigned long long bmax = 0;
    FL_CUDA(cudaMemcpyAsync(&bmax, &cnt[4], 8, cudaMemcpyDeviceToHost, st));
    FL_CUDA(cudaMemsetAsync(s->claimed.p, 0, (size_t)n, st));
    FL_CUDA(cudaMemsetAsync(s->stamp.p, 0, (size_t)n * 4, st));
    FL_CUDA(cudaStreamSynchronize(st));
    DBuf& bcount_d = s->bcount;
    FL_TRY(dalloc(bcount_d, (bmax + 2) * 4 * 2));
    int32_t* bcount = bcount_d.as<int32_t>();
    int32_t* cursor = bcount + (bmax + 2);
    std::vector<int32_t> hcount(bmax + 2), hoff(bmax + 2);

    // values are keys (ordinals), all ones where unset
    uint32_t* const val = s->X.as<uint32_t>();
    Relax r;
    r.narrow = true;
    r.limit = 0xffffffffULL;
    r.fr[0] = s->fr[0].as<int32_t>();
    r.fr[1] = s->fr[1].as<int32_t>();
    r.frval = s->frval.p;
    r.stamp = s->stamp.as<uint32_t>();
    r.cnt = cnt;
    r.h_cnt = &g->h_ctr->aux3;
    FL_TRY(relax_begin(g, r));
    // a graph made of parts (batches): each part's gather sweep stops after
    // its own largest ball radius
    const int32_t* vpart = g->n_parts > 0 ? g->vpart.as<int32_t>() : nullptr;
    int32_t* part_T = nullptr;
    if (vpart) {
        FL_TRY(dalloc(s->part_T, (size_t)g->n_parts * 4));
        part_T = s->part_T.as<int32_t>();
    }
    int32_t* touched = s->touched.as<int32_t>();
    uint8_t* reach = s->reach.as<uint8_t>();
    uint8_t* kill = s->kill.as<uint8_t>();
    // rows of the round log: (greedy round, kind, step, frontier in, pulled, microseconds);
    // kind 0 cover round, 1 gather round, 2 bucket size (step = ball radius), 3 greedy-round total,
    // 4 kill-sweep round (frontier = marks made)
    using clock = std::chrono::steady_clock;
    auto log_row = [&](int64_t rd, int64_t kind, int64_t step, int64_t front, int64_t dense, double us) {
        const int64_t row[6] = {rd, kind, step, front, dense, (int64_t)us};
        s->mis_log.insert(s->mis_log.end(), row, row + 6);
    };
    auto timed_round = [&](int64_t rd, int64_t kind, int64_t step, uint32_t svr) -> int {
        const int64_t front = r.n_front;
        const auto t0 = clock::now();
        FL_TRY(relax_round(g, r, 0ULL, svr, kProfMis));
        log_row(rd, kind, step, front, r.last_dense ? 1 : 0,
                std::chrono::duration<double, std::micro>(clock::now() - t0).count());
        return FL_OK;
    };
    uint32_t sv = 0;  // frontier stamp values, unique per round
    int64_t n_u = m;
    int cu = 0;
    int64_t rounds = 0;
    while (n_u > 0) {
        if (++rounds > m + 1) FL_FAIL(FL_ETIMEOUT, "greedy MIS did not converge");
        const auto round_t0 = clock::now();
        // bucket the undecided facilities by ball radius
        FL_CUDA(cudaMemsetAsync(bcount, 0, (bmax + 1) * 4, st));
        FL_CUDA(cudaMemsetAsync(&cnt[4], 0, 8, st));
        if (part_T) FL_CUDA(cudaMemsetAsync(part_T, 0xff, (size_t)g->n_parts * 4, st));  // -1: no undecided facility
        FL_LAUNCH(kProfMis, k_bucket_count<<<std::min(grid_for(n_u, 256), 152 * 4), 256, 0, st>>>(
                                ulist[cu], n_u, s->bcap.as<int32_t>(), bcount, &cnt[4], vpart, part_T,
                                g->n_parts));
        FL_CUDA(cudaGetLastError());
        unsigned long long T64 = 0;
        FL_CUDA(cudaMemcpyAsync(&T64, &cnt[4], 8, cudaMemcpyDeviceToHost, st));
        FL_CUDA(cudaMemcpyAsync(hcount.data(), bcount, (bmax + 1) * 4, cudaMemcpyDeviceToHost, st));
        FL_CUDA(cudaStreamSynchronize(st));
        const int T = (int)T64;
        int32_t acc = 0;
        for (int b = 0; b <= T; ++b) {
            hoff[b] = acc;
            acc += hcount[b];
            if (hcount[b] > 0) log_row(rounds, 2, b, hcount[b], 0, 0.0);
        }
        // Gather pruning: the cover records reach = 1 + max_f (B_f - d(v, f))
        // (T minus the time its first wave arrived); gather round b needs only
        // vertices with B_f - d(v, f) >= b for some f, the others sit out.
        const bool prune = T < 255;
        if (prune) FL_CUDA(cudaMemsetAsync(reach, 0, (size_t)n, st));
        FL_CUDA(cudaMemcpyAsync(cursor, hoff.data(), (T + 1) * 4, cudaMemcpyHostToDevice, st));
        FL_LAUNCH(kProfMis, k_bucket_scatter<<<grid_for(n_u, 256 * kScatter), 256, 0, st>>>(
                                ulist[cu], n_u, s->bcap.as<int32_t>(), cursor, s->ubuck.as<int32_t>()));
        FL_CUDA(cudaGetLastError());
        const int32_t* ub = s->ubuck.as<int32_t>();

        // ---- cover: X[c] = smallest key of an undecided f with d(c, f) <= B_f.
        // Facility f starts at time T - B_f; all waves stop at time T.
        r.X[0] = val;
        r.X[1] = val + n;
        r.cur = 0;
        auto now = [&]() { return static_cast<uint32_t*>(r.X[r.cur]); };
        FL_CUDA(cudaMemsetAsync(val, 0xff, (size_t)n * 4, st));
        FL_CUDA(cudaMemsetAsync(cnt, 0, 24, st));
        r.n_front = 0;
        r.list_valid = true;
        const uint32_t sv0 = sv;
        r.sv_prev = sv0 + 1;
        r.prune = Prune();
        r.prune.reach = prune ? reach : nullptr;
        for (int t = 0; t <= T; ++t) {
            const int b = T - t;
            if (hcount[b] > 0) {
                FL_TRY(relax_prepare_list(g, r, kProfMis));
                FL_LAUNCH(kProfMis, k_inject<<<grid_for(hcount[b], 256), 256, 0, st>>>(
                                        ub + hoff[b], hcount[b], r.prune.reach, (uint32_t)b + 1u, 0xffffffffu,
                                        s->ord.as<uint32_t>(), now(), r.stamp, sv0 + 1 + t, r.fr[r.fc],
                                        &r.cnt[r.fc]));
                FL_CUDA(cudaGetLastError());
                r.n_front += hcount[b];
            }
            r.prune.reach_val = (uint32_t)(T - t);  // first reached at time t + 1
            // the last round: nothing relays a value past time T, and of the
            // values at time T only the clients' are read (gather seeds and
            // claims), so the other vertices sit it out (left unreached, they
            // have the same effect on the gather and kill sweeps as slack 0)
            r.prune.only = (prune && t == T - 1) ? s->client.as<uint8_t>() : nullptr;
            if (t < T && r.n_front > 0) FL_TRY(timed_round(rounds, 0, t, sv0 + 2 + t));
            else if (t < T) r.sv_prev = sv0 + 2 + t;
        }
        r.prune = Prune();
        sv = sv0 + T + 2;
        const uint32_t* cover = now();
        FL_TRY(relax_collect_set(g, cover, touched, &cnt[6], kProfMis));

        // ---- gather: min over Ball(f) of (claimed ? 0 : cover + 1), read at radius B_f
        r.X[0] = val + 2 * n;
        r.X[1] = val + 3 * n;
        r.cur = 0;
        FL_CUDA(cudaMemsetAsync(r.X[0], 0xff, (size_t)n * 4, st));
        FL_CUDA(cudaMemsetAsync(cnt, 0, 24, st));
        r.fc = 0;
        const uint32_t sg0 = ++sv;
        FL_LAUNCH(kProfMis, k_gather_seed<<<152 * 8, 256, 0, st>>>(touched, &cnt[6], s->client.as<uint8_t>(),
                                                                   s->claimed.as<uint8_t>(), cover, now(),
                                                                   s->mval.as<uint32_t>(), r.stamp, sg0, r.fr[0],
                                                                   &r.cnt[0]));
        FL_CUDA(cudaGetLastError());
        FL_CUDA(cudaMemcpyAsync(r.h_cnt, &r.cnt[0], 8, cudaMemcpyDeviceToHost, st));
        FL_CUDA(cudaStreamSynchronize(st));
        r.n_front = (int64_t)*r.h_cnt;
        r.list_valid = true;
        r.sv_prev = sg0;
        if (hcount[0] > 0)
            FL_LAUNCH(kProfMis, k_decide<<<grid_for(hcount[0], 256), 256, 0, st>>>(
                                    ub + hoff[0], hcount[0], now(), s->ord.as<uint32_t>(),
                                    s->state.as<uint8_t>(), g->ctr.as<Counters>()));
        r.part_limit = part_T;
        r.prune.need = prune ? reach : nullptr;
        for (int b = 1; b <= T; ++b) {
            r.part_round = b;
            r.prune.round = (uint32_t)b;
            if (r.n_front > 0) FL_TRY(timed_round(rounds, 1, b, sg0 + b));
            else r.sv_prev = sg0 + b;
            if (hcount[b] > 0)
                FL_LAUNCH(kProfMis, k_decide<<<grid_for(hcount[b], 256), 256, 0, st>>>(
                                        ub + hoff[b], hcount[b], now(), s->ord.as<uint32_t>(),
                                        s->state.as<uint8_t>(), g->ctr.as<Counters>()));
        }
        sv = sg0 + T + 1;
        r.part_limit = nullptr;
        r.prune = Prune();
        FL_CUDA(cudaGetLastError());

        // ---- claim the balls of this round's winners; keep the undecided
        if (prune) FL_CUDA(cudaMemsetAsync(kill, 0, (size_t)n, st));
        FL_CUDA(cudaMemsetAsync(&cnt[7], 0, 8, st));
        FL_LAUNCH(kProfMis, k_claim<<<152 * 8, 256, 0, st>>>(s->touched.as<int32_t>(), &cnt[6], s->client.as<uint8_t>(),
                                         s->claimed.as<uint8_t>(), s->mval.as<uint32_t>(),
                                         s->fac_by_ord.as<int32_t>(), s->state.as<uint8_t>(),
                                         prune ? kill : nullptr, &cnt[7]));
        FL_CUDA(cudaMemsetAsync(&cnt[3], 0, 8, st));
        FL_LAUNCH(kProfMis, k_compact_undecided<<<grid_for(n_u, 256), 256, 0, st>>>(ulist[cu], n_u, s->state.as<uint8_t>(),
                                                               ulist[cu ^ 1], &cnt[3]));
        FL_CUDA(cudaGetLastError());
        unsigned long long nu = 0, n_claimed = 0;
        FL_CUDA(cudaMemcpyAsync(&nu, &cnt[3], 8, cudaMemcpyDeviceToHost, st));
        FL_CUDA(cudaMemcpyAsync(&n_claimed, &cnt[7], 8, cudaMemcpyDeviceToHost, st));
        FL_TRY(read_counters(g));
        if (g->h_ctr->error) FL_FAIL(FL_ECUDA, "greedy MIS: inconsistent gather state");
        cu ^= 1;
        // ---- kill sweep: an undecided facility whose ball holds a client
        // claimed in this round is adjacent in H-bar to a facility of S and
        // can never join it.  The next round's gather would find the claim
        // too, but only after a cover sweep in which the dead facility still
        // competes; removing it now lets its neighbours decide a round earlier
        // (the result stays the lexicographically-first MIS).  A bounded
        // marking BFS from the newly claimed clients, pruned like the gather.
        if (prune && nu > 0 && n_claimed > 0) {
            for (int b = 1; b <= T; ++b) {
                const auto t0 = clock::now();
                int64_t marked = 0;
                FL_TRY(mark_round(g, r, kill, reach, (uint32_t)b, kProfMis, &marked));
                log_row(rounds, 4, b, marked, 1, std::chrono::duration<double, std::micro>(clock::now() - t0).count());
                if (marked == 0) break;
            }
            FL_LAUNCH(kProfMis, k_kill<<<grid_for((int64_t)nu, 256), 256, 0, st>>>(ulist[cu], (int64_t)nu, kill,
                                                                                  s->bcap.as<int32_t>(),
                                                                                  s->state.as<uint8_t>()));
            FL_CUDA(cudaMemsetAsync(&cnt[3], 0, 8, st));
            FL_LAUNCH(kProfMis, k_compact_undecided<<<grid_for((int64_t)nu, 256), 256, 0, st>>>(
                                    ulist[cu], (int64_t)nu, s->state.as<uint8_t>(), ulist[cu ^ 1], &cnt[3]));
            FL_CUDA(cudaGetLastError());
            FL_CUDA(cudaMemcpyAsync(&nu, &cnt[3], 8, cudaMemcpyDeviceToHost, st));
            FL_CUDA(cudaStreamSynchronize(st));
            cu ^= 1;
        }
        log_row(rounds, 3, T, n_u, n_u - (int64_t)nu,
                std::chrono::duration<double, std::micro>(clock::now() - round_t0).count());
        n_u = (int64_t)nu;
    }
    s->mis_rounds = rounds;
    // open set
    FL_CUDA(cudaMemsetAsync(&cnt[5], 0, 8, st));
    FL_LAUNCH(kProfMis, k_open_list<<<grid_for(n, 256), 256, 0, st>>>(s->state.as<uint8_t>(), n, s->open.as<uint8_t>(),
                                                  s->ulist.as<int32_t>(), &cnt[5]));
    FL_CUDA(cudaGetLastError());
    unsigned long long no = 0;
    FL_CUDA(cudaMemcpyAsync(&no, &cnt[5], 8, cudaMemcpyDeviceToHost, st));
    FL_CUDA(cudaStreamSynchronize(st));
    s->n_open = (int64_t)no;
    return FL_OK;
}

// ------------------------------------------------------------------ assignment + objective

int assign_clients(fl_solve* s) {
    fl_graph* g = s->g;
    FL_TRY(dalloc(s->assign, (size_t)g->n * 4));
    FL_TRY(dalloc(s->dist, (size_t)g->n * 4));
    // the open list was left in ulist by open_facilities
    if (g->sched.graph_bfs)
        return msbfs_graph(g, s->ulist.as<int32_t>(), s->n_open, s->assign.as<int32_t>(), s->dist.as<int32_t>(),
                           s->X, s->stamp, kProfBfs);
    return msbfs(g, s->ulist.as<int32_t>(), s->n_open, s->assign.as<int32_t>(), s->dist.as<int32_t>(), s->X,
                 s->stamp, s->fr, s->frval, kProfBfs);
}

constexpr int kObjBlocks = 152 * 4;

// Opening cost of the open facilities (per block, a fixed tree), distance sum
// and unserved clients.  A thread takes four consecutive vertices (the buffers
// are the solve's own, 256-byte aligned), so that its loads are in flight
// together, and a block adds up its counts before the atomics (a thread's own
// atomics on two words took 105 us at 2^20 vertices, now 7).
__global__ void __launch_bounds__(256) k_objective(int64_t n, const uint8_t* __restrict__ open,
                                                   const double* __restrict__ cost,
                                                   const uint8_t* __restrict__ client,
                                                   const int32_t* __restrict__ dist, double* __restrict__ partial,
                                                   unsigned long long* __restrict__ sums) {
    __shared__ double red[256];
    __shared__ unsigned long long s_sum[2];
    if (threadIdx.x < 2) s_sum[threadIdx.x] = 0;
    double acc = 0.0;
    unsigned long long ds = 0;
    unsigned un = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; 4 * q < n; q += stride) {
        const int64_t v = 4 * q;
        uint8_t op[4], cl[4];
        int32_t d[4];
        if (v + 4 <= n) {
            const uchar4 a = reinterpret_cast<const uchar4*>(open)[q], b = reinterpret_cast<const uchar4*>(client)[q];
            const int4 c = reinterpret_cast<const int4*>(dist)[q];
            op[0] = a.x, op[1] = a.y, op[2] = a.z, op[3] = a.w;
            cl[0] = b.x, cl[1] = b.y, cl[2] = b.z, cl[3] = b.w;
            d[0] = c.x, d[1] = c.y, d[2] = c.z, d[3] = c.w;
        } else {
            for (int j = 0; j < 4; ++j) {
                const bool in = v + j < n;
                op[j] = in ? open[v + j] : 0;
                cl[j] = in ? client[v + j] : 0;
                d[j] = in ? dist[v + j] : 0;
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (op[j]) acc += cost[v + j];
            if (cl[j]) {
                if (d[j] < 0) ++un;
                else ds += (unsigned long long)d[j];
            }
        }
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int s2 = 128; s2 > 0; s2 >>= 1) {
        if ((int)threadIdx.x < s2) red[threadIdx.x] += red[threadIdx.x + s2];
        __syncthreads();
    }
    un = __reduce_add_sync(kFull, un);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ds += __shfl_xor_sync(kFull, ds, o);
    if (lane_id() == 0) {
        atomicAdd(&s_sum[0], ds);
        atomicAdd(&s_sum[1], (unsigned long long)un);
    }
    __syncthreads();
    if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
    if (threadIdx.x < 2 && s_sum[threadIdx.x]) atomicAdd(&sums[threadIdx.x], s_sum[threadIdx.x]);
}

int objective(fl_solve* s, double* obj, int64_t* dist_sum, int64_t* n_unserved) {
    fl_graph* g = s->g;
    cudaStream_t st = g->stream;
    DBuf& tmp = s->obj_tmp;
    FL_TRY(dalloc(tmp, kObjBlocks * 8 + 64));
    double* partial = tmp.as<double>();
    unsigned long long* sums = reinterpret_cast<unsigned long long*>(partial + kObjBlocks);
    int rc = FL_OK;
    std::vector<double> hp(kObjBlocks);
    unsigned long long hs[2] = {0, 0};
    cudaError_t e = cudaMemsetAsync(sums, 0, 16, st);
    if (e == cudaSuccess) {
        FL_LAUNCH(kProfOther, k_objective<<<kObjBlocks, 256, 0, st>>>(g->n, s->open.as<uint8_t>(), s->cost.as<double>(),
                                                s->client.as<uint8_t>(), s->dist.as<int32_t>(), partial, sums));
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(hp.data(), partial, kObjBlocks * 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(hs, sums, 16, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) rc = status_of(e, "objective", __FILE__, __LINE__);

    if (rc) return rc;
    double open_cost = 0.0;
    for (int b = 0; b < kObjBlocks; ++b) open_cost += hp[b];
    *obj = open_cost + (double)hs[0];
    *dist_sum = (int64_t)hs[0];
    *n_unserved = (int64_t)hs[1];
    return FL_OK;
}

}  // namespace fl

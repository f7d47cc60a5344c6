// k_relax.cu -- synchronous min-propagation rounds over the CSR, used by the
// multi-source BFS (assignment, eccentricity bound) and by the cover / gather
// sweeps of the greedy MIS ("send to all vertices within distance d", §4.5).
//
// One round: every vertex v takes X'[v] = min(X[v], min_{u in N(v)} X[u] + add),
// reading only values of the previous round, so a value moves exactly one hop
// per round.  Only the frontier (the vertices whose value changed in the
// previous round) can lower a value.  Push rounds walk the frontier list
// (k_snap_front + k_push_low / k_push_segs, in place on one buffer, the
// frontier's values snapshotted first); pull rounds write the second buffer
// (every vertex reads its frontier neighbours, found in a bitmap; no atomics
// except per hub segment) and flag changed vertices with the next round's
// stamp.  Hub edge lists are split into fl_graph::seg-edge segments in both.
#include <algorithm>
#include <cstdio>

#include "fl_internal.cuh"

namespace fl {

namespace {

int grid_for(int64_t items, int per_block) {
    int64_t b = (items + per_block - 1) / per_block;
    if (b < 1) b = 1;
    if (b > 152 * 32) b = 152 * 32;
    return (int)b;
}

__device__ __forceinline__ bool in_front(const uint32_t* __restrict__ bm, int32_t u) {
    return (__ldg(&bm[u >> 5]) >> (u & 31)) & 1u;
}


// Frontier bitmap of a pull round: bit v = (stamp[v] == sv).  Only neighbours
// whose value changed in the previous round can lower a value, so a pull
// reads the value of a neighbour only when its bit is set; the bitmap (n/8
// bytes) stays in L2 while the values do not.
//
// In a graph made of disjoint parts (batches) the parts with frontier vertices
// are flagged: a part without any has no vertex that can change, and pull
// rounds skip it.  A part whose limit is below `round` no longer
// needs its values (nothing of it reads them any more) and sits out too.
//
// A warp takes kBmWords words in a row, four words' loads at a time, and a block
// flags a part once: the flags share a line, and an access to it costs some 10 ns
// (4.2 M vertices in 16 parts, all with frontier vertices: 72 us with a flag per
// warp, 375 with a look at the flag before it, 10 now).
constexpr int kBmWords = 16;

__global__ void k_bitmap(const uint32_t* __restrict__ stamp, uint32_t sv, int64_t n, uint32_t* __restrict__ bm,
                         const int32_t* __restrict__ vpart, int32_t* __restrict__ part_cnt,
                         const int32_t* __restrict__ part_limit, int32_t round) {
    __shared__ int32_t s_flagged;  // the part that the block flagged last
    if (threadIdx.x == 0) s_flagged = -1;
    __syncthreads();
    const int lane = lane_id();
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t c = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; c * 32 * kBmWords < n; c += warps) {
        int32_t known = -1;  // the part looked up last, and whether it takes part
        bool live = false;
        const int64_t end = min((c + 1) * 32 * kBmWords, n);
        for (int64_t base = c * 32 * kBmWords; base < end; base += 128) {
            bool in[4];
            int32_t p[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int64_t v = base + 32 * j + lane;
                in[j] = v < end && __ldg(&stamp[v]) == sv;
                p[j] = vpart && v < end ? __ldg(&vpart[v]) : -1;
            }
            uint32_t mine = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (vpart && in[j] && p[j] != known) {
                    known = p[j];
                    live = !(part_limit && part_limit[known] < round);
                    if (live && atomicExch(&s_flagged, known) != known) part_cnt[known] = 1;
                }
                const unsigned w = __ballot_sync(kFull, in[j] && (!vpart || live));
                if (lane == j) mine = w;
            }
            if (lane < 4 && base + 32 * lane < end) bm[(base >> 5) + lane] = mine;
        }
    }
}

__device__ __forceinline__ bool part_idle(const int32_t* __restrict__ vpart, const int32_t* __restrict__ part_cnt,
                                          int32_t v) {
    return vpart && __ldg(&part_cnt[__ldg(&vpart[v])]) == 0;
}

__device__ __forceinline__ bool skipped(const Prune& pr, int32_t u) {
    return (pr.need && __ldg(&pr.need[u]) <= pr.round) || (pr.only && !__ldg(&pr.only[u]));
}

// Values are 64-bit for a BFS (distance << 32 | label) and 32-bit for the MIS
// sweeps, whose values are key ordinals below 2^31: half the bytes of every
// gather and of the copy per round, and a warp's 32 gathers touch fewer sectors
// of the hot head of X.  R-MAT scale 22, a dense gather round: k_pull_low 221 ->
// 192 us, k_pull_segs 125 -> 114 us; the whole query 8.29 -> 7.24 ms, a batch of 16
// solves on R-MAT scale 18 6.72 -> 5.93 ms.
// Values >= `limit` are ignored: unset entries.  With `settle`, a
// vertex holding a value below the limit is final and is skipped.
//
// Lowest value offered by the frontier neighbours cols[e], e in [e0, e1) with
// stride `step`, four edges per lane and pass: the four bitmap loads, then
// the value loads are independent, so each lane keeps up to four dependent-
// load chains in flight; the columns of the next pass are loaded at the start
// of a pass, so their DRAM latency overlaps this pass's bitmap and value loads.
//
// kAll: every neighbour's value is read, the bitmap is not.  A neighbour whose
// value did not change offers what it offered in an earlier round, so the
// result is the same; when most neighbours are in the frontier the bitmap only
// adds a second gather per edge to rounds that are bound by the gathers (L1
// wavefronts, 80 % of its peak).
template <bool kAll, class V>
__device__ __forceinline__ V pull_min(const int32_t* __restrict__ cols, int64_t e0, int64_t e1, int step,
                                      const uint32_t* __restrict__ bm, const V* __restrict__ X, V add, V limit, V m) {
    int32_t nx[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) nx[j] = e0 + j * step < e1 ? __ldcs(&cols[e0 + j * step]) : -1;
    for (int64_t e = e0; e < e1; e += 4 * step) {
        int32_t u[4];
        bool f[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) u[j] = nx[j];
        const int64_t en = e + 4 * step;
#pragma unroll
        for (int j = 0; j < 4; ++j) nx[j] = en + j * step < e1 ? __ldcs(&cols[en + j * step]) : -1;
#pragma unroll
        for (int j = 0; j < 4; ++j) f[j] = u[j] >= 0 && (kAll || in_front(bm, u[j]));
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (f[j]) {
                const V x = __ldg(&X[u[j]]);
                if (x < limit && x + add < m) m = x + add;
            }
        }
    }
    return m;
}

// Pull round over vertices of at most kSmallDeg neighbours: a thread per
// vertex, its neighbours loaded four at a time (column, bitmap and value
// loads each independent of the others), so that a warp keeps 32 vertices'
// chains in flight.
template <bool kAll, class V>
__global__ void __launch_bounds__(256) k_pull_small(const int32_t* __restrict__ list, int64_t n_list,
                                                    const int64_t* __restrict__ rowp,
                                                    const int32_t* __restrict__ cols, V add, V limit, bool settle,
                                                    const uint32_t* __restrict__ bm, const V* __restrict__ X,
                                                    V* __restrict__ Xn,
                                                    uint32_t* __restrict__ stamp, uint32_t sv,
                                                    unsigned long long* __restrict__ n_changed,
                                                    const int32_t* __restrict__ vpart,
                                                    const int32_t* __restrict__ part_cnt, Prune pr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned changed = 0;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n_list; base += stride) {
        const int64_t i = base + lane_id();
        const int32_t v = i < n_list ? list[i] : 0;
        const bool have = i < n_list && !part_idle(vpart, part_cnt, v) && !skipped(pr, v);
        const V own = have ? X[v] : (V)~(V)0;
        const bool work = have && !(settle && own < limit);
        const int64_t beg = work ? rowp[v] : 0, end = work ? rowp[v + 1] : 0;
        const V m = pull_min<kAll, V>(cols, beg, end, 1, bm, X, add, limit, own);
        const bool ch = work && m < own;
        if (ch) {
            Xn[v] = m;
            stamp[v] = sv;
            if (pr.reach && own >= limit) pr.reach[v] = (uint8_t)pr.reach_val;
        }
        changed += __popc(__ballot_sync(kFull, ch));
    }
    block_count(lane_id() == 0 ? changed : 0u, n_changed);
}

// Pull round over the other non-hub vertices: four vertices per warp, eight
// lanes per vertex striding over its neighbours; the lanes meet again at the
// reduction.
template <bool kAll, class V>
__global__ void __launch_bounds__(256) k_pull_low(const int32_t* __restrict__ list, int64_t n_list,
                                                  const int64_t* __restrict__ rowp, const int32_t* __restrict__ cols,
                                                  V add, V limit, bool settle,
                                                  const uint32_t* __restrict__ bm, const V* __restrict__ X,
                                                  V* __restrict__ Xn, uint32_t* __restrict__ stamp,
                                                  uint32_t sv, unsigned long long* __restrict__ n_changed,
                                                  const int32_t* __restrict__ vpart,
                                                  const int32_t* __restrict__ part_cnt, Prune pr) {
    const int lane = lane_id();
    const int sub = lane & 7;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned changed = 0;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w * 4 < n_list; w += warps) {
        const int64_t i = w * 4 + (lane >> 3);
        const int32_t v = i < n_list ? list[i] : 0;
        const bool have = i < n_list && !part_idle(vpart, part_cnt, v) && !skipped(pr, v);
        const V own = have ? X[v] : (V)~(V)0;
        const bool work = have && !(settle && own < limit);
        const int64_t beg = work ? rowp[v] : 0, end = work ? rowp[v + 1] : 0;
        V m = pull_min<kAll, V>(cols, beg + sub, end, 8, bm, X, add, limit, own);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) m = min(m, __shfl_xor_sync(kFull, m, o));
        const bool ch = work && sub == 0 && m < own;
        if (ch) {
            Xn[v] = m;
            stamp[v] = sv;
            if (pr.reach && own >= limit) pr.reach[v] = (uint8_t)pr.reach_val;
        }
        changed += __popc(__ballot_sync(kFull, ch));
    }
    block_count(lane == 0 ? changed : 0u, n_changed);
}

// Pull round over hubs: one warp per segment of fl_graph::seg edges.  Xn[v] starts as
// X[v]; the segments lower it with atomicMin and the one that lowers it first
// (it sees the old value) flags the hub.
template <bool kAll, class V>
__global__ void __launch_bounds__(256) k_pull_segs(const int32_t* __restrict__ seg_hub, int64_t n_seg,
                                                   const int64_t* __restrict__ hub_seg,
                                                   const int32_t* __restrict__ hub_list,
                                                   const int64_t* __restrict__ rowp, const int32_t* __restrict__ cols,
                                                   int seg, V add, V limit, bool settle,
                                                   const uint32_t* __restrict__ bm, const V* __restrict__ X,
                                                   V* __restrict__ Xn, uint32_t* __restrict__ stamp,
                                                   uint32_t sv, unsigned long long* __restrict__ n_changed,
                                                   const int32_t* __restrict__ vpart,
                                                   const int32_t* __restrict__ part_cnt, Prune pr) {
    const int lane = lane_id();
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t sidx = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; sidx < n_seg; sidx += warps) {
        const int32_t h = seg_hub[sidx];
        const int32_t v = hub_list[h];
        const V own = X[v];
        if ((settle && own < limit) || part_idle(vpart, part_cnt, v) || skipped(pr, v)) continue;
        const int64_t e0 = rowp[v] + (sidx - hub_seg[h]) * seg;
        const int64_t e1 = min(e0 + (int64_t)seg, rowp[v + 1]);
        V m = pull_min<kAll, V>(cols, e0 + lane, e1, 32, bm, X, add, limit, (V)~(V)0);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = min(m, __shfl_xor_sync(kFull, m, o));
        if (lane == 0 && m < own) {
            const V old = atomicMin(&Xn[v], m);
            if (old == own) {
                stamp[v] = sv;
                if (pr.reach && own >= limit) pr.reach[v] = (uint8_t)pr.reach_val;
                atomicAdd(n_changed, 1ULL);
            }
        }
    }
}

// Snapshot of a push frontier: frval[i] = X[fr[i]], the frontier's edge count
// into *edges, and each hub of the frontier tagged (hub_tag = tag, hub_val =
// its value) for the segment push.  hub_list is ascending.
template <class V>
__global__ void k_snap_front(const int32_t* __restrict__ fr, const unsigned long long* __restrict__ n_fr,
                             const V* __restrict__ X, V* __restrict__ frval,
                             unsigned long long* __restrict__ reset_next, const int64_t* __restrict__ rowp,
                             const int32_t* __restrict__ hub_list, int64_t n_hubs, int seg, uint32_t* __restrict__ hub_tag,
                             uint32_t tag, V* __restrict__ hub_val,
                             unsigned long long* __restrict__ edges) {
    const int64_t n = (int64_t)*n_fr;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    if (blockIdx.x == 0 && threadIdx.x == 0) *reset_next = 0;
    unsigned long long ed = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const int32_t v = fr[i];
        const V x = X[v];
        frval[i] = x;
        const int64_t d = rowp[v + 1] - rowp[v];
        ed += (unsigned long long)d;
        if (d > seg) {
            int64_t lo = 0, hi = n_hubs;  // first hub_list entry >= v
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (hub_list[mid] < v) lo = mid + 1;
                else hi = mid;
            }
            if (lo < n_hubs && hub_list[lo] == v) {
                hub_val[lo] = x;
                hub_tag[lo] = tag;
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ed += __shfl_xor_sync(kFull, ed, o);
    if (lane_id() == 0 && ed) atomicAdd(edges, ed);
}

// Push from the non-hub frontier vertices: a warp per vertex, read-before-
// atomicMin on the neighbours, stamp dedupe for the next frontier.
template <class V>
__global__ void __launch_bounds__(256) k_push_low(const int32_t* __restrict__ fr,
                                                  const V* __restrict__ frval,
                                                  const unsigned long long* __restrict__ n_fr,
                                                  const int64_t* __restrict__ rowp, const int32_t* __restrict__ cols,
                                                  int seg, V add, V limit, V* __restrict__ X,
                                                  uint32_t* __restrict__ stamp, uint32_t sv,
                                                  int32_t* __restrict__ fr_next, unsigned long long* __restrict__ n_next,
                                                  Prune pr) {
    const int lane = lane_id();
    const int64_t n = (int64_t)*n_fr;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = (((int64_t)blockIdx.x * blockDim.x) + threadIdx.x) >> 5; w < n; w += warps) {
        const int32_t v = fr[w];
        const int64_t beg = rowp[v], end = rowp[v + 1];
        if (end - beg > seg) continue;  // hubs: k_push_segs
        const V val = frval[w] + add;
        for (int64_t cb = beg; cb < end; cb += 32) {
            const int64_t e = cb + lane;
            bool fresh = false;
            int32_t u = 0;
            if (e < end) {
                u = cols[e];
                if (val < X[u] && !skipped(pr, u)) {
                    const V old = atomicMin(&X[u], val);
                    if (val < old) {
                        if (pr.reach && old >= limit) pr.reach[u] = (uint8_t)pr.reach_val;
                        fresh = atomicExch(&stamp[u], sv) != sv;
                    }
                }
            }
            const long long at = warp_append(fresh, n_next);
            if (at >= 0) fr_next[at] = u;
        }
    }
}

// Push from the frontier hubs (tagged by k_snap_front): a warp per segment.
template <class V>
__global__ void __launch_bounds__(256) k_push_segs(const int32_t* __restrict__ seg_hub, int64_t n_seg,
                                                   const int64_t* __restrict__ hub_seg,
                                                   const int32_t* __restrict__ hub_list,
                                                   const uint32_t* __restrict__ hub_tag, uint32_t tag,
                                                   const V* __restrict__ hub_val,
                                                   const int64_t* __restrict__ rowp, const int32_t* __restrict__ cols,
                                                   int seg, V add, V limit, V* __restrict__ X,
                                                   uint32_t* __restrict__ stamp, uint32_t sv,
                                                   int32_t* __restrict__ fr_next, unsigned long long* __restrict__ n_next,
                                                   Prune pr) {
    const int lane = lane_id();
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t sidx = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; sidx < n_seg; sidx += warps) {
        const int32_t h = seg_hub[sidx];
        if (hub_tag[h] != tag) continue;
        const int32_t v = hub_list[h];
        const V val = hub_val[h] + add;
        const int64_t e0 = rowp[v] + (sidx - hub_seg[h]) * seg;
        const int64_t e1 = min(e0 + (int64_t)seg, rowp[v + 1]);
        for (int64_t cb = e0; cb < e1; cb += 32) {
            const int64_t e = cb + lane;
            bool fresh = false;
            int32_t u = 0;
            if (e < e1) {
                u = cols[e];
                if (val < X[u] && !skipped(pr, u)) {
                    const V old = atomicMin(&X[u], val);
                    if (val < old) {
                        if (pr.reach && old >= limit) pr.reach[u] = (uint8_t)pr.reach_val;
                        fresh = atomicExch(&stamp[u], sv) != sv;
                    }
                }
            }
            const long long at = warp_append(fresh, n_next);
            if (at >= 0) fr_next[at] = u;
        }
    }
}

// Vertices flagged with stamp sv -> list.
__global__ void k_collect_stamped(const uint32_t* __restrict__ stamp, uint32_t sv, int64_t n,
                                  int32_t* __restrict__ out, unsigned long long* __restrict__ n_out) {
    __shared__ BlockAppend<8> sh;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t bb = (int64_t)blockIdx.x * blockDim.x; bb < n; bb += stride) {
        const int64_t v = bb + threadIdx.x;
        const bool in = v < n && stamp[v] == sv;
        const long long at = block_append<8>(in, n_out, sh);
        if (at >= 0) out[at] = (int32_t)v;
    }
}

constexpr int64_t kPushAlways = 4096;  // smaller frontiers push without counting their edges
// A pull reads every neighbour's value when frontier * kAllDiv >= the listed
// vertices.  R-MAT, 4.2 M vertices, a cover round of a query: 160 us (hub
// segments) and 268 us (the others) with the bitmap, 125 and 222 without; a
// round with 30 % of the vertices in the frontier 160 and 268 against 127 and
// 225.
constexpr int64_t kAllDiv = 4;

}  // namespace

// Vertices that a sweep reached (a value below the unset one) -> list.
__global__ void k_collect_set(const uint32_t* __restrict__ X, int64_t n, int32_t* __restrict__ out,
                              unsigned long long* __restrict__ n_out) {
    __shared__ BlockAppend<8> sh;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t bb = (int64_t)blockIdx.x * blockDim.x; bb < n; bb += stride) {
        const int64_t v = bb + threadIdx.x;
        const bool in = v < n && X[v] != 0xffffffffu;
        const long long at = block_append<8>(in, n_out, sh);
        if (at >= 0) out[at] = (int32_t)v;
    }
}

int relax_collect_set(fl_graph* g, const uint32_t* X, int32_t* out, unsigned long long* n_out, int cls) {
    FL_CUDA(cudaMemsetAsync(n_out, 0, 8, g->stream));
    FL_LAUNCH(cls, k_collect_set<<<grid_for(g->n, 256), 256, 0, g->stream>>>(X, g->n, out, n_out));
    FL_CUDA(cudaGetLastError());
    return FL_OK;
}

// Work lists and round scratch of g allocated ahead (so that a solve on a
// prefix view of g allocates nothing graph-owned).
int relax_reserve(fl_graph* g) {
    Relax r;
    return relax_begin(g, r);
}

int relax_begin(fl_graph* g, Relax& r) {
    if (!g->lists_ready) {
        FL_TRY(build_work_lists(g));
        g->lists_ready = 1;
    }
    r.dense_div = g->sched.dense_div;
    r.edge_div = g->sched.edge_div;
    const size_t bm_words = (size_t)(g->n + 63) / 32 + 2;
    const size_t off_tag = ((bm_words * 4 + 255) / 256) * 256;
    const size_t off_val = off_tag + (((size_t)g->n_hubs * 4 + 255) / 256) * 256;
    const size_t off_cnt = off_val + (((size_t)g->n_hubs * 8 + 255) / 256) * 256;
    const size_t off_part = off_cnt + 256;
    FL_TRY(dalloc(g->relax_aux, off_part + (size_t)(g->n_parts + 1) * 4));
    char* base = g->relax_aux.as<char>();
    r.bm = reinterpret_cast<uint32_t*>(base);
    r.hub_tag = reinterpret_cast<uint32_t*>(base + off_tag);
    r.hub_val = base + off_val;
    r.ecnt = reinterpret_cast<unsigned long long*>(base + off_cnt);
    r.part_cnt = reinterpret_cast<int32_t*>(base + off_part);
    if (g->n_hubs > 0) FL_CUDA(cudaMemsetAsync(r.hub_tag, 0, (size_t)g->n_hubs * 4, g->stream));
    FL_CUDA(cudaMemsetAsync(r.ecnt, 0, 256, g->stream));
    return FL_OK;
}

namespace {

// One synchronous round.  The caller keeps the frontier count on the host
// (r.n_front) and, for push rounds, a valid list in r.fr[r.fc] with its count
// in r.cnt[r.fc].  `sv` is the stamp of the frontier this round produces.
// A round pushes when its frontier is small (few vertices, or few edges);
// otherwise it pulls with the frontier bitmap.
template <class V>
int round_of(fl_graph* g, Relax& r, V add, uint32_t sv, int cls) {
    cudaStream_t st = g->stream;
    const int64_t n = g->n;
    const int64_t* rowp = g->rowp.as<int64_t>();
    const int32_t* cols = g->cols.as<int32_t>();
    const int32_t* hub_list = g->hub_list.as<int32_t>();
    bool dense = r.n_front * r.dense_div >= g->n_low + g->n_hubs;
    V* X = static_cast<V*>(r.X[r.cur]);
    V* frval = static_cast<V*>(r.frval);
    V* hub_val = static_cast<V*>(r.hub_val);
    const V limit = (V)r.limit;
    if (!dense) {
        if (!r.list_valid) {
            // rebuild the frontier list from the stamps of the previous round
            FL_CUDA(cudaMemsetAsync(&r.cnt[r.fc], 0, 8, st));
            FL_LAUNCH(cls, k_collect_stamped<<<grid_for(n, 256), 256, 0, st>>>(r.stamp, r.sv_prev, n, r.fr[r.fc],
                                                                              &r.cnt[r.fc]));
            r.list_valid = true;
        }
        FL_CUDA(cudaMemsetAsync(r.ecnt, 0, 8, st));
        FL_LAUNCH(cls, k_snap_front<<<grid_for(r.n_front, 256), 256, 0, st>>>(
                           r.fr[r.fc], &r.cnt[r.fc], X, frval, &r.cnt[r.fc ^ 1], rowp, hub_list, g->n_hubs, g->seg,
                           r.hub_tag, r.sv_prev, hub_val, r.ecnt));
        FL_CUDA(cudaGetLastError());
        if (r.n_front >= kPushAlways) {
            FL_CUDA(cudaMemcpyAsync(r.h_cnt, r.ecnt, 8, cudaMemcpyDeviceToHost, st));
            FL_CUDA(cudaStreamSynchronize(st));
            dense = (int64_t)*r.h_cnt * r.edge_div >= g->nnz;
        }
    }
    if (!dense) {
        FL_LAUNCH(cls, k_push_low<<<grid_for(r.n_front, 8), 256, 0, st>>>(r.fr[r.fc], frval, &r.cnt[r.fc], rowp, cols, g->seg,
                                                                         add, limit, X, r.stamp, sv, r.fr[r.fc ^ 1],
                                                                         &r.cnt[r.fc ^ 1], r.prune));
        if (g->n_seg > 0)
            FL_LAUNCH(cls, k_push_segs<<<grid_for(g->n_seg, 8), 256, 0, st>>>(
                               g->seg_hub.as<int32_t>(), g->n_seg, g->hub_seg.as<int64_t>(), hub_list, r.hub_tag,
                               r.sv_prev, hub_val, rowp, cols, g->seg, add, limit, X, r.stamp, sv, r.fr[r.fc ^ 1],
                               &r.cnt[r.fc ^ 1], r.prune));
        FL_CUDA(cudaGetLastError());
        r.fc ^= 1;
        r.list_valid = true;
        FL_CUDA(cudaMemcpyAsync(r.h_cnt, &r.cnt[r.fc], 8, cudaMemcpyDeviceToHost, st));
    } else {
        V* Xn = static_cast<V*>(r.X[r.cur ^ 1]);
        const int32_t* vpart = g->n_parts > 0 ? g->vpart.as<int32_t>() : nullptr;
        // most of the listed vertices changed: read every neighbour's value
        // (not in a BFS: its frontier leaves out the hubs, reached earlier, that
        // most edges lead to)
        const bool all = !r.settle && r.n_front * kAllDiv >= g->n_low + g->n_hubs;
        if (vpart) FL_CUDA(cudaMemsetAsync(r.part_cnt, 0, (size_t)g->n_parts * 4, st));
        if (vpart || !all)
            FL_LAUNCH(cls, k_bitmap<<<grid_for(n, 256 * kBmWords), 256, 0, st>>>(r.stamp, r.sv_prev, n, r.bm, vpart, r.part_cnt,
                                                                      vpart ? r.part_limit : nullptr, r.part_round));
        FL_CUDA(cudaMemcpyAsync(Xn, X, (size_t)n * sizeof(V), cudaMemcpyDeviceToDevice, st));
        FL_CUDA(cudaMemsetAsync(&r.cnt[2], 0, 8, st));
        auto small = all ? k_pull_small<true, V> : k_pull_small<false, V>;
        auto low = all ? k_pull_low<true, V> : k_pull_low<false, V>;
        auto segs = all ? k_pull_segs<true, V> : k_pull_segs<false, V>;
        if (g->n_small > 0)
            FL_LAUNCH(cls, small<<<grid_for(g->n_small, 256), 256, 0, st>>>(
                               g->small_list.as<int32_t>(), g->n_small, rowp, cols, add, limit, r.settle, r.bm, X,
                               Xn, r.stamp, sv, &r.cnt[2], vpart, r.part_cnt, r.prune));
        if (g->n_mid > 0)
            FL_LAUNCH(cls, low<<<grid_for((g->n_mid + 3) / 4, 8), 256, 0, st>>>(
                               g->mid_list.as<int32_t>(), g->n_mid, rowp, cols, add, limit, r.settle, r.bm, X, Xn,
                               r.stamp, sv, &r.cnt[2], vpart, r.part_cnt, r.prune));
        if (g->n_seg > 0)
            FL_LAUNCH(cls, segs<<<grid_for(g->n_seg, 8), 256, 0, st>>>(
                               g->seg_hub.as<int32_t>(), g->n_seg, g->hub_seg.as<int64_t>(), hub_list, rowp, cols, g->seg, add,
                               limit, r.settle, r.bm, X, Xn, r.stamp, sv, &r.cnt[2], vpart, r.part_cnt,
                               r.prune));
        FL_CUDA(cudaGetLastError());
        r.cur ^= 1;
        r.list_valid = false;
        FL_CUDA(cudaMemcpyAsync(r.h_cnt, &r.cnt[2], 8, cudaMemcpyDeviceToHost, st));
    }
    FL_CUDA(cudaStreamSynchronize(st));
    r.n_front = (int64_t)*r.h_cnt;
    r.sv_prev = sv;
    r.last_dense = dense;
    return FL_OK;
}

}  // namespace

int relax_round(fl_graph* g, Relax& r, unsigned long long add, uint32_t sv, int cls) {
    return r.narrow ? round_of<uint32_t>(g, r, (uint32_t)add, sv, cls) : round_of<unsigned long long>(g, r, add, sv, cls);
}

// ------------------------------------------------------------------ marking rounds
// A bounded BFS that only records whether a vertex lies within distance b of
// the seeds: kr[v] = 1 + its distance, 0 while it is farther than the rounds
// run so far (seeds carry 1).  Round b marks every unmarked vertex with
// need[v] > b that has a neighbour marked in an earlier round (kr in [1, b],
// read from a bitmap); a vertex stops reading its row at the first such
// neighbour, so a dense round costs far less than a min-propagation round.

namespace {

__global__ void k_mark_bitmap(const uint8_t* __restrict__ kr, int64_t n, uint32_t b, uint32_t* __restrict__ bm) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
        const int64_t v = base + lane_id();
        const uint32_t k = v < n ? kr[v] : 0u;
        const unsigned w = __ballot_sync(kFull, k != 0 && k <= b);
        if (lane_id() == 0) bm[base >> 5] = w;
    }
}

__device__ __forceinline__ bool unmarked_needed(const uint8_t* __restrict__ kr, const uint8_t* __restrict__ need,
                                                int32_t v, uint32_t b) {
    return kr[v] == 0 && (!need || __ldg(&need[v]) > b);
}

// Vertices of at most kSmallDeg neighbours: a thread each.
__global__ void __launch_bounds__(256) k_mark_small(const int32_t* __restrict__ list, int64_t n_list,
                                                    const int64_t* __restrict__ rowp,
                                                    const int32_t* __restrict__ cols,
                                                    const uint32_t* __restrict__ bm, uint8_t* __restrict__ kr,
                                                    const uint8_t* __restrict__ need, uint32_t b,
                                                    unsigned long long* __restrict__ n_marked) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned marked = 0;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n_list; base += stride) {
        const int64_t i = base + lane_id();
        const int32_t v = i < n_list ? list[i] : 0;
        bool hit = false;
        if (i < n_list && unmarked_needed(kr, need, v, b)) {
            const int64_t beg = rowp[v], end = rowp[v + 1];
            for (int64_t e = beg; e < end && !hit; e += 4) {
                int32_t u[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) u[j] = e + j < end ? __ldcs(&cols[e + j]) : -1;
#pragma unroll
                for (int j = 0; j < 4; ++j) hit |= u[j] >= 0 && in_front(bm, u[j]);
            }
            if (hit) kr[v] = (uint8_t)(b + 1);
        }
        marked += __popc(__ballot_sync(kFull, hit));
    }
    block_count(lane_id() == 0 ? marked : 0u, n_marked);
}

// Other non-hub vertices: eight lanes each (four per warp), 32 entries of a
// row per pass; a group leaves at the first pass that finds a marked neighbour.
__global__ void __launch_bounds__(256) k_mark_low(const int32_t* __restrict__ list, int64_t n_list,
                                                  const int64_t* __restrict__ rowp, const int32_t* __restrict__ cols,
                                                  const uint32_t* __restrict__ bm, uint8_t* __restrict__ kr,
                                                  const uint8_t* __restrict__ need, uint32_t b,
                                                  unsigned long long* __restrict__ n_marked) {
    const int lane = lane_id();
    const int sub = lane & 7;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    unsigned marked = 0;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w * 4 < n_list; w += warps) {
        const int64_t i = w * 4 + (lane >> 3);
        const int32_t v = i < n_list ? list[i] : 0;
        bool work = i < n_list && unmarked_needed(kr, need, v, b);
        const int64_t beg = work ? rowp[v] : 0, end = work ? rowp[v + 1] : 0;
        for (int64_t at = beg;; at += 32) {
            bool hit = false;
            if (work) {
                int32_t u[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int64_t e = at + sub + 8 * j;
                    u[j] = e < end ? __ldcs(&cols[e]) : -1;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) hit |= u[j] >= 0 && in_front(bm, u[j]);
            }
            const bool group_hit = (__ballot_sync(kFull, hit) >> (lane & ~7)) & 0xffu;
            if (work && group_hit) {
                if (sub == 0) {
                    kr[v] = (uint8_t)(b + 1);
                    ++marked;
                }
                work = false;
            }
            if (at + 32 >= end) work = false;
            if (!__any_sync(kFull, work)) break;
        }
    }
    block_count(marked, n_marked);
}

// Hubs: a warp per segment of fl_graph::seg entries; every segment that finds a marked
// neighbour marks the hub (the count may hold a hub more than once).
__global__ void __launch_bounds__(256) k_mark_segs(const int32_t* __restrict__ seg_hub, int64_t n_seg,
                                                   const int64_t* __restrict__ hub_seg,
                                                   const int32_t* __restrict__ hub_list,
                                                   const int64_t* __restrict__ rowp, const int32_t* __restrict__ cols,
                                                   int seg,
                                                   const uint32_t* __restrict__ bm, uint8_t* __restrict__ kr,
                                                   const uint8_t* __restrict__ need, uint32_t b,
                                                   unsigned long long* __restrict__ n_marked) {
    const int lane = lane_id();
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t sidx = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; sidx < n_seg; sidx += warps) {
        const int32_t h = seg_hub[sidx];
        const int32_t v = hub_list[h];
        if (!unmarked_needed(kr, need, v, b)) continue;
        const int64_t e0 = rowp[v] + (sidx - hub_seg[h]) * seg;
        const int64_t e1 = min(e0 + (int64_t)seg, rowp[v + 1]);
        for (int64_t at = e0; at < e1; at += 128) {
            bool hit = false;
            int32_t u[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int64_t e = at + lane + 32 * j;
                u[j] = e < e1 ? __ldcs(&cols[e]) : -1;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) hit |= u[j] >= 0 && in_front(bm, u[j]);
            if (__any_sync(kFull, hit)) {
                if (lane == 0) {
                    kr[v] = (uint8_t)(b + 1);
                    atomicAdd(n_marked, 1ULL);
                }
                break;
            }
        }
    }
}

}  // namespace

int mark_round(fl_graph* g, Relax& r, uint8_t* kr, const uint8_t* need, uint32_t b, int cls, int64_t* marked) {
    cudaStream_t st = g->stream;
    const int64_t* rowp = g->rowp.as<int64_t>();
    const int32_t* cols = g->cols.as<int32_t>();
    FL_CUDA(cudaMemsetAsync(&r.cnt[2], 0, 8, st));
    FL_LAUNCH(cls, k_mark_bitmap<<<grid_for(g->n, 256), 256, 0, st>>>(kr, g->n, b, r.bm));
    if (g->n_small > 0)
        FL_LAUNCH(cls, k_mark_small<<<grid_for(g->n_small, 256), 256, 0, st>>>(
                           g->small_list.as<int32_t>(), g->n_small, rowp, cols, r.bm, kr, need, b, &r.cnt[2]));
    if (g->n_mid > 0)
        FL_LAUNCH(cls, k_mark_low<<<grid_for((g->n_mid + 3) / 4, 8), 256, 0, st>>>(
                           g->mid_list.as<int32_t>(), g->n_mid, rowp, cols, r.bm, kr, need, b, &r.cnt[2]));
    if (g->n_seg > 0)
        FL_LAUNCH(cls, k_mark_segs<<<grid_for(g->n_seg, 8), 256, 0, st>>>(
                           g->seg_hub.as<int32_t>(), g->n_seg, g->hub_seg.as<int64_t>(), g->hub_list.as<int32_t>(),
                           rowp, cols, g->seg, r.bm, kr, need, b, &r.cnt[2]));
    FL_CUDA(cudaGetLastError());
    FL_CUDA(cudaMemcpyAsync(r.h_cnt, &r.cnt[2], 8, cudaMemcpyDeviceToHost, st));
    FL_CUDA(cudaStreamSynchronize(st));
    *marked = (int64_t)*r.h_cnt;
    return FL_OK;
}

// Add vertices to the current frontier list (sources or injections): X[s] =
// min(X[s], val(s)); s joins when it decreases.  Makes the list valid first.
int relax_prepare_list(fl_graph* g, Relax& r, int cls) {
    if (r.list_valid) return FL_OK;
    cudaStream_t st = g->stream;
    FL_CUDA(cudaMemsetAsync(&r.cnt[r.fc], 0, 8, st));
    FL_LAUNCH(cls, k_collect_stamped<<<grid_for(g->n, 256), 256, 0, st>>>(r.stamp, r.sv_prev, g->n, r.fr[r.fc],
                                                                          &r.cnt[r.fc]));
    FL_CUDA(cudaGetLastError());
    r.list_valid = true;
    return FL_OK;
}

}  // namespace fl

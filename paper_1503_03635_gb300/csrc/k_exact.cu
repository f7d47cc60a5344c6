// k_exact.cu -- exact neighbourhood sizes, their HIP estimates, and radii
// from exact client counts: the ground truth of the ADS accuracy study
// (Section 5.1, "Accuracy vs. k", Fig. 1) and an exact-radius mode of phase
// (ii) (Eq. 1 at epsilon -> 0 with the true number of clients at each
// distance in place of the HIP estimate).
//
// Exact sizes come from a bit-parallel breadth-first search.  One sweep
// serves 64 W sources; every vertex holds W words of source bits for
// "visited", "frontier" and "next".  W is 4, 8 or 16, the smallest that takes
// the sources left (graphs above kXWideN vertices: 4, for their scratch): a
// level's launches and its look by the host serve four times the sources at
// W = 16, and a neighbour is one 128-byte line instead of four 32-byte sectors
// in four sweeps.  A source stops when its question is
// answered -- ball sizes at the largest distance asked for or when its
// component is exhausted, a radius when the walk of Eq. 1 has its root --
// and its bit is masked out of every later level.  Each level runs in one of
// two directions (Beamer, Asanovic, Patterson, SC 2012), chosen from the
// frontier's row entries against the entries of rows that still need bits:
//   bottom-up: every vertex that some running source has not reached ORs
//     its neighbours' frontier words and keeps the new bits.  Rows longer
//     than 32 entries get a whole warp (32 / W neighbours x W words at a time,
//     several in flight, stopping once every needed bit is in); rows longer
//     than 256 are cut into work items of 256 entries, a warp each, that OR
//     into the row's next words (a warp, or a block, on the largest hub was
//     most of a level); shorter rows get W lanes, one word each.
//     A bottom-up level of 1000 sources on an R-MAT graph with 262 k vertices:
//     light 92 us, heavy 105, items 86 (a block per long row: 552).
//   top-down (sparse frontiers, e.g. the sources themselves): the frontier
//     rows, cut into work items of 256 entries (so a hub's row is spread
//     over many warps), OR their bits into the neighbours' next words
//     (atomicOr); one pass over all vertices then folds the new bits into
//     "visited" and counts them.
// Both directions count the new bits per source under the predicate and
// list the next frontier with its row entries.
#include <algorithm>
#include <cmath>

#include "fl_internal.cuh"

namespace fl {
namespace {

constexpr int kXMaxW = 16;      // 64-bit words of source bits per vertex, at most
// Larger graphs take W = 4: a sweep holds 24 W bytes per vertex until the graph is
// destroyed (96 B at W = 4, 384 at 16; 1.6 GB against 0.4 at 2^22 vertices).  The
// line is that limit on scratch, not where the speed turns: 1000 sources on R-MAT,
// W = 4 against 16, 2^20 + 1 vertices 4.3 / 2.8 ms, 2^21 9.7 / 7.8, 2^22 18.2 / 14.3.
constexpr int64_t kXWideN = 1 << 20;
constexpr int kXHeavy = 32;     // rows longer than this get a whole warp
constexpr int kXSeg = 256;      // entries of a work item
constexpr int kXHuge = kXSeg;   // rows longer than this are cut into work items
constexpr int kXBlocks = 152 * 8;
constexpr int kXLevelBlocks = 152 * 4;  // level kernels: each warp flushes its counts once

enum XMode { kXSizes = 0, kXRadius = 1 };

// State of one sweep (device).
template <int W>
struct XState {
    static constexpr int kS = 64 * W;  // sources
    unsigned long long active[W];    // sources still searching
    unsigned long long any[W];       // sources that reached a vertex at this level
    unsigned long long cnt[kS];      // this level's newly reached vertices under the predicate
    long long N[kS];                 // sizes: running ball size; radius: N_j
    long long G[kS], Gp[kS];         // radius: G_{j+1} and G_j of the walk
    unsigned long long rows, entries;  // rows scanned and their entries read (this sweep, cumulative)
    unsigned long long n_next;       // this level: vertices listed in the next frontier
    unsigned long long fr_edges;     // this level: row entries of the next frontier
    unsigned long long rem_edges;    // bottom-up level: row entries of vertices that still need bits
};

// Per-lane sums a level kernel flushes once.
struct XSums {
    unsigned long long rows = 0, entries = 0, fr_edges = 0, rem_edges = 0;
};

int blocks_for(int64_t items, int64_t per_block, int most = kXBlocks) {
    int64_t b = (items + per_block - 1) / per_block;
    if (b < 1) b = 1;
    if (b > most) b = most;
    return (int)b;
}

// Original ids -> internal ids, with range checks.
__global__ void k_x_map(const int32_t* __restrict__ src, int64_t n_src, const int32_t* __restrict__ inv, int64_t n,
                        int32_t* __restrict__ out, Counters* ctr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_src; i += stride) {
        const int32_t s = src[i];
        if (s < 0 || s >= n) {
            atomicOr(&ctr->error, 1ULL);
            out[i] = 0;
        } else {
            out[i] = inv ? inv[s] : s;
        }
    }
}

// Vertices with short rows (<= kXHeavy entries, isolated ones included), with
// long rows, and with rows above kXHuge entries (from the end of `heavy`).
__global__ void k_x_lists(const int64_t* __restrict__ rowp, int64_t n, int32_t* __restrict__ light,
                          int32_t* __restrict__ heavy, unsigned long long* n_light, unsigned long long* n_heavy,
                          unsigned long long* n_huge) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
        const int64_t v = base + lane_id();
        const bool valid = v < n;
        const int64_t deg = valid ? rowp[v + 1] - rowp[v] : 0;
        const long long a = warp_append(valid && deg <= kXHeavy, n_light);
        if (a >= 0) light[a] = (int32_t)v;
        const long long b = warp_append(valid && deg > kXHeavy && deg <= kXHuge, n_heavy);
        if (b >= 0) heavy[b] = (int32_t)v;
        const long long c = warp_append(valid && deg > kXHuge, n_huge);
        if (c >= 0) heavy[n - 1 - c] = (int32_t)v;
    }
}

// Facilities (finite cost) of an exact-radius solve; every radius starts at
// +inf; a cost that is NaN, <= 0 or -inf is an error.
__global__ void k_x_facilities(const double* __restrict__ cost, int64_t n, int32_t* __restrict__ fac,
                               double* __restrict__ radius, Counters* ctr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
        const int64_t v = base + lane_id();
        const bool valid = v < n;
        const double c = valid ? cost[v] : INFINITY;
        if (valid) {
            const bool ok = (c > 0.0 && c < INFINITY) || c == INFINITY;
            if (!ok) atomicOr(&ctr->error, 1ULL);
            radius[v] = INFINITY;
        }
        const long long at = warp_append(valid && c > 0.0 && c < INFINITY, &ctr->aux0);
        if (at >= 0) fac[at] = (int32_t)v;
    }
}

// Start of a sweep: the sources' own bits in "visited" and "frontier"
// (which the host cleared), the sources as the first frontier list, cleared
// counters.  One block of 64 W threads.
template <int W>
__global__ void k_x_seed(const int32_t* __restrict__ src, int64_t nb, const int64_t* __restrict__ rowp,
                         unsigned long long* __restrict__ vis, unsigned long long* __restrict__ cur,
                         int32_t* __restrict__ front, XState<W>* __restrict__ st) {
    const int s = threadIdx.x;
    st->cnt[s] = 0;
    st->N[s] = 0;
    st->G[s] = 0;
    st->Gp[s] = 0;
    if (s < W) {
        const int64_t m = nb - 64LL * s;  // sources in word s
        st->active[s] = m <= 0 ? 0ULL : (m >= 64 ? ~0ULL : ((1ULL << m) - 1ULL));
        st->any[s] = 0;
    }
    if (s == 0) {
        st->rows = st->entries = 0;
        st->n_next = (unsigned long long)nb;
        st->fr_edges = st->rem_edges = 0;
    }
    __syncthreads();
    if (s < nb) {
        const int32_t v = src[s];
        const unsigned long long bit = 1ULL << (s & 63);
        atomicOr(&vis[(int64_t)v * W + (s >> 6)], bit);
        atomicOr(&cur[(int64_t)v * W + (s >> 6)], bit);
        front[s] = v;  // a source listed twice is harmless
        atomicAdd(&st->fr_edges, (unsigned long long)(rowp[v + 1] - rowp[v]));
    }
}

// Shared memory of a level kernel: counts per source, bit b of word w at
// [b * W + w] (the lanes of a group count different words: no bank conflicts).
template <int W>
struct XShared {
    unsigned cnt[64 * W];
    unsigned long long any[W];
};

template <int W>
__device__ __forceinline__ void x_init(XShared<W>& sh) {
    for (int i = threadIdx.x; i < 64 * W; i += blockDim.x) sh.cnt[i] = 0;
    if (threadIdx.x < W) sh.any[threadIdx.x] = 0;
    __syncthreads();
}

// Per-bit counts of the words that a lane adds, as five bit planes (a carry
// chain of ten operations per word, where a ballot per bit took 64 for the
// warp): up to 31 words between two flushes.
struct XPlanes {
    unsigned long long p[5] = {0, 0, 0, 0, 0};
    int n = 0;
    __device__ __forceinline__ void add(unsigned long long x) {
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const unsigned long long c = p[i] & x;
            p[i] ^= x;
            x = c;
        }
        ++n;
    }
    // to the block's counts of word w; rot spreads the lanes that share w (all 32 lanes call)
    template <int W>
    __device__ __forceinline__ void flush(XShared<W>& sh, int w, int rot) {
        n = 0;
        if (!__any_sync(kFull, (p[0] | p[1] | p[2] | p[3] | p[4]) != 0)) return;
        for (int i = 0; i < 64; ++i) {
            const int b = (i + rot) & 63;
            const unsigned c = (unsigned)((p[0] >> b) & 1) | ((unsigned)((p[1] >> b) & 1) << 1) |
                               ((unsigned)((p[2] >> b) & 1) << 2) | ((unsigned)((p[3] >> b) & 1) << 3) |
                               ((unsigned)((p[4] >> b) & 1) << 4);
            if (c) atomicAdd(&sh.cnt[b * W + w], c);
        }
#pragma unroll
        for (int i = 0; i < 5; ++i) p[i] = 0;
    }
};

// End of a level kernel: the lanes' counts, the OR of the new bits (lane w
// mod W holds word w) and the level's sums.  Every thread of the block calls.
template <int W>
__device__ __forceinline__ void x_flush(XPlanes& c, unsigned long long any, XSums m, XShared<W>& sh, XState<W>* st) {
    const int lane = lane_id();
    const int q = lane / W;
    c.flush(sh, lane & (W - 1), q * (64 * W / 32) + q);
#pragma unroll
    for (int o = W; o < 32; o <<= 1) any |= __shfl_xor_sync(kFull, any, o);
    if (lane < W && any) atomicOr(&sh.any[lane], any);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        m.rows += __shfl_xor_sync(kFull, m.rows, o);
        m.entries += __shfl_xor_sync(kFull, m.entries, o);
        m.fr_edges += __shfl_xor_sync(kFull, m.fr_edges, o);
        m.rem_edges += __shfl_xor_sync(kFull, m.rem_edges, o);
    }
    if (lane == 0) {
        if (m.rows) atomicAdd(&st->rows, m.rows);
        if (m.entries) atomicAdd(&st->entries, m.entries);
        if (m.fr_edges) atomicAdd(&st->fr_edges, m.fr_edges);
        if (m.rem_edges) atomicAdd(&st->rem_edges, m.rem_edges);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 64 * W; i += blockDim.x)
        if (sh.cnt[i]) atomicAdd(&st->cnt[(i & (W - 1)) * 64 + i / W], (unsigned long long)sh.cnt[i]);
    if (threadIdx.x < W && sh.any[threadIdx.x]) atomicOr(&st->any[threadIdx.x], sh.any[threadIdx.x]);
}

// Does some lane of this lane's group of W hold true?  (mask: a ballot)
template <int W>
__device__ __forceinline__ bool group_any(unsigned mask) {
    constexpr unsigned kGroup = (1u << W) - 1u;
    return ((mask >> (lane_id() & ~(W - 1))) & kGroup) != 0;
}

// Bottom-up level for vertices with short rows: W lanes per vertex (lane w
// holds word w), 32 / W vertices per warp; the lanes of a group load the row's
// columns together and share them, so several neighbours' words are in flight.
template <int W>
__global__ void __launch_bounds__(256) k_x_light(const int32_t* __restrict__ list, int64_t n_list,
                                                 const int64_t* __restrict__ rowp, const int32_t* __restrict__ cols,
                                                 const unsigned long long* __restrict__ cur,
                                                 unsigned long long* __restrict__ nxt, unsigned long long* vis,
                                                 const uint8_t* __restrict__ pred, int32_t* __restrict__ next_front,
                                                 XState<W>* __restrict__ st) {
    __shared__ XShared<W> sh;
    x_init(sh);
    constexpr int kLoads = W == 4 ? 2 : 1;  // columns per lane and step
    const int lane = lane_id();
    const int w = lane & (W - 1), q = lane / W;
    const unsigned qm = ((1u << W) - 1u) << (lane & ~(W - 1));
    const unsigned long long act = st->active[w];
    XPlanes c;
    unsigned long long any = 0;
    XSums m;
    const int64_t stride = ((int64_t)gridDim.x * blockDim.x) / W;
    for (int64_t base = (((int64_t)blockIdx.x * blockDim.x) + (threadIdx.x & ~31)) / W; base < n_list;
         base += stride) {
        const int64_t i = base + q;
        const bool valid = i < n_list;
        const int32_t v = valid ? __ldg(&list[i]) : 0;
        const unsigned long long vw = valid ? vis[(int64_t)v * W + w] : ~0ULL;
        const unsigned long long need = act & ~vw;
        const unsigned nb = __ballot_sync(kFull, need != 0);
        unsigned long long nx = 0;
        int64_t deg = 0;
        if (group_any<W>(nb)) {  // some word of this vertex still needs bits
            const int64_t beg = __ldg(&rowp[v]), end = __ldg(&rowp[v + 1]);
            deg = end - beg;
            if (w == 0) {
                ++m.rows;
                m.entries += (unsigned long long)deg;
            }
            unsigned long long acc = 0;
            for (int64_t e0 = beg; e0 < end; e0 += kLoads * W) {
                int32_t u[kLoads];
#pragma unroll
                for (int l = 0; l < kLoads; ++l) u[l] = e0 + l * W + w < end ? __ldg(&cols[e0 + l * W + w]) : -1;
#pragma unroll
                for (int j = 0; j < kLoads * W; ++j) {
                    const int32_t x = __shfl_sync(qm, u[j / W], j & (W - 1), W);
                    if (x >= 0) acc |= __ldg(&cur[(int64_t)x * W + w]);
                }
            }
            nx = acc & need;
        }
        if (valid) {
            nxt[(int64_t)v * W + w] = nx;
            if (nx) vis[(int64_t)v * W + w] = vw | nx;
        }
        any |= nx;
        // the vertex joins the next frontier; or still needs bits afterwards
        const bool got = group_any<W>(__ballot_sync(kFull, nx != 0));
        const bool left = group_any<W>(__ballot_sync(kFull, (need & ~nx) != 0));
        const long long at = warp_append(w == 0 && got, &st->n_next);
        if (at >= 0) {
            next_front[at] = v;
            m.fr_edges += (unsigned long long)deg;
        }
        if (w == 0 && left) m.rem_edges += (unsigned long long)deg;
        c.add((valid && (!pred || pred[v])) ? nx : 0ULL);
        if (c.n == 31) c.flush(sh, w, q * (64 * W / 32) + q);
    }
    x_flush(c, any, m, sh, st);
}

// Bottom-up level for vertices with long rows: a warp per vertex, lane (t, w)
// reads word w of neighbours t, t + 32 / W, ..., kUnroll in flight; every 128
// entries the warp stops if its OR already holds every bit the vertex needs.
template <int W>
__global__ void __launch_bounds__(256) k_x_heavy(const int32_t* __restrict__ list, int64_t n_list,
                                                 const int64_t* __restrict__ rowp, const int32_t* __restrict__ cols,
                                                 const unsigned long long* __restrict__ cur,
                                                 unsigned long long* __restrict__ nxt, unsigned long long* vis,
                                                 const uint8_t* __restrict__ pred, int32_t* __restrict__ next_front,
                                                 XState<W>* __restrict__ st) {
    __shared__ XShared<W> sh;
    x_init(sh);
    constexpr int kT = 32 / W, kUnroll = W == 4 ? 4 : 8, kStep = kT * kUnroll;
    const int lane = lane_id();
    const int w = lane & (W - 1), t = lane / W;
    const unsigned long long act = st->active[w];
    XPlanes c;
    unsigned long long any = 0;
    XSums m;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = (((int64_t)blockIdx.x * blockDim.x) + threadIdx.x) >> 5; i < n_list; i += warps) {
        const int32_t v = __ldg(&list[i]);
        const unsigned long long vw = vis[(int64_t)v * W + w];
        const unsigned long long need = act & ~vw;
        unsigned long long nx = 0;
        int64_t deg = 0;
        if (__any_sync(kFull, need != 0)) {
            const int64_t beg = __ldg(&rowp[v]), end = __ldg(&rowp[v + 1]);
            deg = end - beg;
            int64_t stop = end;
            unsigned long long acc = 0;
            for (int64_t b0 = beg; b0 < end; b0 += kStep) {
                int32_t u[kUnroll];
#pragma unroll
                for (int j = 0; j < kUnroll; ++j) u[j] = b0 + kT * j + t < end ? __ldg(&cols[b0 + kT * j + t]) : -1;
#pragma unroll
                for (int j = 0; j < kUnroll; ++j)
                    if (u[j] >= 0) acc |= __ldg(&cur[(int64_t)u[j] * W + w]);
                if (((b0 - beg) & 127) == 128 - kStep) {
                    unsigned long long a = acc;
#pragma unroll
                    for (int o = W; o < 32; o <<= 1) a |= __shfl_xor_sync(kFull, a, o);
                    if (__all_sync(kFull, (a & need) == need)) {
                        acc = a;
                        stop = b0 + kStep < end ? b0 + kStep : end;
                        break;
                    }
                }
            }
#pragma unroll
            for (int o = W; o < 32; o <<= 1) acc |= __shfl_xor_sync(kFull, acc, o);
            nx = acc & need;
            if (lane == 0) {
                ++m.rows;
                m.entries += (unsigned long long)(stop - beg);
            }
        }
        if (t == 0) {
            nxt[(int64_t)v * W + w] = nx;
            if (nx) vis[(int64_t)v * W + w] = vw | nx;
        }
        any |= nx;
        const bool got = __any_sync(kFull, nx != 0);
        const bool left = __any_sync(kFull, (need & ~nx) != 0);
        const long long at = warp_append(lane == 0 && got, &st->n_next);
        if (at >= 0) {
            next_front[at] = v;
            m.fr_edges += (unsigned long long)deg;
        }
        if (lane == 0 && left) m.rem_edges += (unsigned long long)deg;
        // every lane holds its word's new bits; the first group counts them
        c.add(t == 0 && (!pred || pred[v]) ? nx : 0ULL);
        if (c.n == 31) c.flush(sh, w, 0);
    }
    x_flush(c, any, m, sh, st);
}

// Work items of the rows above kXHuge entries (vertex << 32 | segment): the rows'
// first segments, then the others (*n_more of them) in any order.  With few
// sources a row's first segment often brings all that it needs, and the items
// after it are passed over: one source on 2 x 2000 vertices, joined completely,
// 0.28 ms with a row's items side by side, 0.24 now (and one wait of the host less).
__global__ void k_x_huge_items(const int32_t* __restrict__ list, int64_t n_list, const int64_t* __restrict__ rowp,
                               unsigned long long* __restrict__ items, unsigned long long* __restrict__ n_more) {
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = (((int64_t)blockIdx.x * blockDim.x) + threadIdx.x) >> 5; i < n_list; i += warps) {
        const int32_t v = list[i];
        const unsigned long long item = (unsigned long long)(uint32_t)v << 32;
        const int more = (int)((rowp[v + 1] - rowp[v] + kXSeg - 1) / kXSeg) - 1;
        unsigned long long at = 0;
        if (lane_id() == 0) {
            items[i] = item;
            at = (unsigned long long)n_list + atomicAdd(n_more, (unsigned long long)more);
        }
        at = __shfl_sync(kFull, at, 0);
        for (int j = lane_id(); j < more; j += 32) items[at + j] = item | (unsigned)(j + 1);
    }
}

// Their next words start empty (W lanes per vertex).
template <int W>
__global__ void k_x_huge_clear(const int32_t* __restrict__ list, int64_t n_list,
                               unsigned long long* __restrict__ nxt) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n_list * W; t += stride)
        nxt[(int64_t)list[t / W] * W + (t & (W - 1))] = 0;
}

// Bottom-up level, the items: a warp each; lane (t, w) reads word w of
// neighbours t, t + 32 / W, ..., eight in flight.  An item whose row has every
// bit it needs is passed over.
template <int W>
__global__ void __launch_bounds__(256) k_x_huge(const unsigned long long* __restrict__ items, int64_t n_first,
                                                const unsigned long long* __restrict__ n_more,
                                                const int64_t* __restrict__ rowp, const int32_t* __restrict__ cols,
                                                const unsigned long long* __restrict__ cur, unsigned long long* nxt,
                                                const unsigned long long* __restrict__ vis, XState<W>* __restrict__ st) {
    constexpr int kT = 32 / W, kUnroll = 8, kStep = kT * kUnroll;
    const int lane = lane_id();
    const int w = lane & (W - 1), t = lane / W;
    const unsigned long long act = st->active[w];
    unsigned long long entries = 0;
    const int64_t n_items = n_first + (int64_t)*n_more;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = (((int64_t)blockIdx.x * blockDim.x) + threadIdx.x) >> 5; i < n_items; i += warps) {
        const unsigned long long it = __ldg(&items[i]);
        const int32_t v = (int32_t)(it >> 32);
        const unsigned long long need = act & ~__ldg(&vis[(int64_t)v * W + w]) & ~__ldcg(&nxt[(int64_t)v * W + w]);
        if (!__any_sync(kFull, need != 0)) continue;
        const int64_t row_end = __ldg(&rowp[v + 1]);
        const int64_t beg = __ldg(&rowp[v]) + (int64_t)(uint32_t)it * kXSeg;
        const int64_t end = beg + kXSeg < row_end ? beg + kXSeg : row_end;
        unsigned long long acc = 0;
        for (int64_t b0 = beg; b0 < end; b0 += kStep) {
            int32_t u[kUnroll];
#pragma unroll
            for (int j = 0; j < kUnroll; ++j) u[j] = b0 + kT * j + t < end ? __ldg(&cols[b0 + kT * j + t]) : -1;
#pragma unroll
            for (int j = 0; j < kUnroll; ++j)
                if (u[j] >= 0) acc |= __ldg(&cur[(int64_t)u[j] * W + w]);
        }
#pragma unroll
        for (int o = W; o < 32; o <<= 1) acc |= __shfl_xor_sync(kFull, acc, o);
        acc &= need;
        if (t == 0 && acc) atomicOr(&nxt[(int64_t)v * W + w], acc);
        entries += (unsigned long long)(end - beg);
    }
    if (lane == 0 && entries) atomicAdd(&st->entries, entries);
}

// ... and their vertices: what the warp kernels do after a row (W lanes per vertex).
template <int W>
__global__ void __launch_bounds__(256) k_x_huge_done(const int32_t* __restrict__ list, int64_t n_list,
                                                     const int64_t* __restrict__ rowp,
                                                     const unsigned long long* __restrict__ nxt,
                                                     unsigned long long* vis, const uint8_t* __restrict__ pred,
                                                     int32_t* __restrict__ next_front, XState<W>* __restrict__ st) {
    __shared__ XShared<W> sh;
    x_init(sh);
    const int lane = lane_id();
    const int w = lane & (W - 1), q = lane / W;
    const unsigned long long act = st->active[w];
    XPlanes c;
    unsigned long long any = 0;
    XSums m;
    const int64_t stride = ((int64_t)gridDim.x * blockDim.x) / W;
    for (int64_t base = (((int64_t)blockIdx.x * blockDim.x) + (threadIdx.x & ~31)) / W; base < n_list;
         base += stride) {
        const bool valid = base + q < n_list;
        const int32_t v = valid ? __ldg(&list[base + q]) : 0;
        const unsigned long long vw = valid ? vis[(int64_t)v * W + w] : ~0ULL;
        const unsigned long long need = act & ~vw;
        const unsigned long long nx = valid ? nxt[(int64_t)v * W + w] : 0ULL;
        const unsigned long long deg = valid ? (unsigned long long)(__ldg(&rowp[v + 1]) - __ldg(&rowp[v])) : 0ULL;
        if (nx) vis[(int64_t)v * W + w] = vw | nx;
        any |= nx;
        const bool had = group_any<W>(__ballot_sync(kFull, need != 0));
        const bool got = group_any<W>(__ballot_sync(kFull, nx != 0));
        const bool left = group_any<W>(__ballot_sync(kFull, (need & ~nx) != 0));
        const long long at = warp_append(w == 0 && got, &st->n_next);
        if (at >= 0) {
            next_front[at] = v;
            m.fr_edges += deg;
        }
        if (w == 0 && had) ++m.rows;
        if (w == 0 && left) m.rem_edges += deg;
        c.add((valid && (!pred || pred[v])) ? nx : 0ULL);
        if (c.n == 31) c.flush(sh, w, q * (64 * W / 32) + q);
    }
    x_flush(c, any, m, sh, st);
}

// Top-down level, step 1: the frontier rows as work items of at most
// kXSeg entries (vertex << 32 | segment), so that a hub's row is spread over
// many warps.  A vertex without running bits gives none.

template <int W>
__global__ void k_x_td_items(const int32_t* __restrict__ front, int64_t n_front, const int64_t* __restrict__ rowp,
                             const unsigned long long* __restrict__ cur, unsigned long long* __restrict__ items,
                             XState<W>* __restrict__ st) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int lane = lane_id();
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n_front; base += stride) {
        const int64_t i = base + lane;
        int segs = 0;
        int32_t u = 0;
        if (i < n_front) {
            u = __ldg(&front[i]);
            unsigned long long running = 0;
#pragma unroll
            for (int w = 0; w < W; ++w) running |= __ldg(&cur[(int64_t)u * W + w]) & st->active[w];
            const bool live = running != 0;
            const int64_t deg = __ldg(&rowp[u + 1]) - __ldg(&rowp[u]);
            segs = live ? (int)((deg + kXSeg - 1) / kXSeg) : 0;
        }
        const int incl = warp_incl_scan(segs);
        const int total = __shfl_sync(kFull, incl, 31);
        unsigned long long at = 0;
        if (lane == 31 && total) at = atomicAdd(&st->n_next, (unsigned long long)total);
        at = __shfl_sync(kFull, at, 31) + (unsigned long long)(incl - segs);
        for (int j = 0; j < segs; ++j) items[at + j] = ((unsigned long long)(uint32_t)u << 32) | (unsigned)j;
    }
}

// Step 2: a warp per work item, lane (t, w) takes word w of the row owner's
// running bits to entries t, t + 32 / W, ...: the bits a neighbour has not visited
// go into its next words (atomicOr; the host cleared them).
template <int W>
__global__ void __launch_bounds__(256) k_x_td(const unsigned long long* __restrict__ items,
                                              const int64_t* __restrict__ rowp, const int32_t* __restrict__ cols,
                                              const unsigned long long* __restrict__ cur,
                                              unsigned long long* __restrict__ nxt,
                                              const unsigned long long* __restrict__ vis,
                                              XState<W>* __restrict__ st) {
    constexpr int kT = 32 / W;
    const int lane = lane_id();
    const int w = lane & (W - 1), t = lane / W;
    const unsigned long long act = st->active[w];
    const int64_t n_items = (int64_t)st->n_next;
    unsigned long long rows = 0, entries = 0;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = (((int64_t)blockIdx.x * blockDim.x) + threadIdx.x) >> 5; i < n_items; i += warps) {
        const unsigned long long it = __ldg(&items[i]);
        const int32_t u = (int32_t)(it >> 32);
        const int64_t seg = (int64_t)(it & 0xffffffffULL);
        const unsigned long long bits = __ldg(&cur[(int64_t)u * W + w]) & act;
        const int64_t row_end = __ldg(&rowp[u + 1]);
        const int64_t beg = __ldg(&rowp[u]) + seg * kXSeg;
        const int64_t end = beg + kXSeg < row_end ? beg + kXSeg : row_end;
        if (lane == 0) {
            rows += seg == 0 ? 1 : 0;
            entries += (unsigned long long)(end - beg);
        }
#pragma unroll 4
        for (int64_t b0 = beg; b0 < end; b0 += kT) {
            const int64_t e = b0 + t;
            if (e < end) {
                const int32_t v = __ldg(&cols[e]);
                const unsigned long long nb = bits & ~__ldg(&vis[(int64_t)v * W + w]);
                if (nb) atomicOr(&nxt[(int64_t)v * W + w], nb);
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        rows += __shfl_xor_sync(kFull, rows, o);
        entries += __shfl_xor_sync(kFull, entries, o);
    }
    if (lane == 0 && rows) {
        atomicAdd(&st->rows, rows);
        atomicAdd(&st->entries, entries);
    }
}

// Step 3, over every vertex (W lanes per vertex): fold the new bits into
// "visited", count them, list the next frontier and its row entries.
template <int W>
__global__ void __launch_bounds__(256) k_x_td_finish(int64_t n, const int64_t* __restrict__ rowp,
                                                     const unsigned long long* __restrict__ nxt,
                                                     unsigned long long* vis, const uint8_t* __restrict__ pred,
                                                     int32_t* __restrict__ next_front, XState<W>* __restrict__ st) {
    __shared__ XShared<W> sh;
    x_init(sh);
    const int lane = lane_id();
    const int w = lane & (W - 1), q = lane / W;
    XPlanes c;
    unsigned long long any = 0;
    XSums m;
    const int64_t stride = ((int64_t)gridDim.x * blockDim.x) / W;
    for (int64_t base = (((int64_t)blockIdx.x * blockDim.x) + (threadIdx.x & ~31)) / W; base < n; base += stride) {
        const int64_t v = base + q;
        const bool valid = v < n;
        const unsigned long long nx = valid ? nxt[v * W + w] : 0ULL;
        const unsigned some = __ballot_sync(kFull, nx != 0);
        if (!some) continue;
        if (nx) vis[v * W + w] |= nx;
        any |= nx;
        const long long at = warp_append(w == 0 && group_any<W>(some), &st->n_next);
        if (at >= 0) {
            next_front[at] = (int32_t)v;
            m.fr_edges += (unsigned long long)(__ldg(&rowp[v + 1]) - __ldg(&rowp[v]));
        }
        c.add((valid && (!pred || pred[v])) ? nx : 0ULL);
        if (c.n == 31) c.flush(sh, w, q * (64 * W / 32) + q);
    }
    x_flush(c, any, m, sh, st);
}

// End of a level (one block of 64 W threads, thread s = source s of the
// sweep): fold the level's counts into each running source and stop the
// sources that are answered.  Level 0 is the source itself.
//   sizes:  N += (new vertices at this distance under the predicate);
//           row[level] = N; a source stops at level D or, filling the rest
//           of its row with N, at the first level that reaches nothing.
//   radius: the walk of Eq. 1: N_j = N_{j-1} + W_j, G_{j+1} = G_j + N_j;
//           r = j + (c - G_j) / N_j at the first j with G_{j+1} >= c; a
//           level that reaches nothing means j-1 was the eccentricity L and
//           r = L + (c - G_L) / N_L (+inf when N_L = 0).  N and G are exact
//           integers; each FP64 step is one IEEE operation.
template <int W>
__global__ void k_x_finish(XState<W>* __restrict__ st, int mode, int64_t level, const int32_t* __restrict__ src,
                           const uint8_t* __restrict__ pred, const double* __restrict__ cost, int64_t D,
                           int64_t* __restrict__ sizes, double* __restrict__ radius, Counters* ctr) {
    __shared__ unsigned s_bal[2 * W];
    const int s = threadIdx.x;
    const int w = s >> 6;
    const unsigned long long bit = 1ULL << (s & 63);
    bool act = (st->active[w] & bit) != 0;
    if (act) {
        const int32_t v = src[s];
        long long fresh;
        bool found;
        if (level == 0) {
            fresh = (!pred || pred[v]) ? 1 : 0;
            found = true;
        } else {
            fresh = (long long)st->cnt[s];
            found = (st->any[w] & bit) != 0;
        }
        if (mode == kXSizes) {
            const long long N = st->N[s] + fresh;
            st->N[s] = N;
            int64_t* row = sizes + (int64_t)s * (D + 1);
            row[level] = N;
            if (!found) {
                for (int64_t h = level + 1; h <= D; ++h) row[h] = N;
                act = false;
            } else if (level == D) {
                act = false;
            }
        } else {
            const double c = cost[v];
            double r = INFINITY;
            if (!found) {
                const long long N = st->N[s];
                if (N > 0) r = __dadd_rn((double)(level - 1), __ddiv_rn(__dsub_rn(c, (double)st->Gp[s]), (double)N));
                act = false;
            } else {
                const long long N = st->N[s] + fresh;
                const long long G = st->G[s];
                const long long Gn = G + N;
                st->N[s] = N;
                if ((double)Gn >= c) {
                    r = __dadd_rn((double)level, __ddiv_rn(__dsub_rn(c, (double)G), (double)N));
                    act = false;
                } else {
                    st->Gp[s] = G;
                    st->G[s] = Gn;
                }
            }
            if (!act) radius[v] = r;
        }
    }
    __syncthreads();  // every thread has read active, any and its count
    st->cnt[s] = 0;
    const unsigned bal = __ballot_sync(kFull, act);
    if (lane_id() == 0) s_bal[s >> 5] = bal;
    __syncthreads();
    if (s < W) {
        st->active[s] = (unsigned long long)s_bal[2 * s] | ((unsigned long long)s_bal[2 * s + 1] << 32);
        st->any[s] = 0;
    }
    if (s == 0) {
        unsigned long long tot = 0;
        for (int i = 0; i < 2 * W; ++i) tot += __popc(s_bal[i]);
        ctr->aux0 = tot;
        ctr->scanned = st->rows;
        ctr->cand_reads = st->entries;
        ctr->frontier = st->n_next;
        ctr->merges = st->fr_edges;
        ctr->aux3 = st->rem_edges;
        st->n_next = st->fr_edges = st->rem_edges = 0;
    }
}

// HIP estimates of the same sizes from the ADS (the predicated
// neighbourhood query of Section 3.3; the estimator of Section 4.5): a warp
// per source; out row h = sum over the groups at hop <= h, in hop order, of
// (counted entries under the predicate) x the group's weight.
__global__ void __launch_bounds__(256) k_x_estimates(const int32_t* __restrict__ src, int64_t n_src, int64_t D,
                                                     const uint8_t* __restrict__ pred,
                                                     const int64_t* __restrict__ gofs,
                                                     const int64_t* __restrict__ eofs,
                                                     const uint32_t* __restrict__ ginfo,
                                                     const double* __restrict__ gwt, const int32_t* __restrict__ eid,
                                                     double* __restrict__ out) {
    const int lane = lane_id();
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t s = (((int64_t)blockIdx.x * blockDim.x) + threadIdx.x) >> 5; s < n_src; s += warps) {
        const int32_t v = src[s];
        const int64_t g0 = gofs[v], g1 = gofs[v + 1];
        int64_t e = eofs[v];
        double* row = out + s * (D + 1);
        double N = 0.0;
        int64_t h = 0;
        for (int64_t gi = g0; gi < g1; ++gi) {
            const uint32_t info = ginfo[gi];
            const int64_t hop = (int64_t)(info & 0xffffu);
            const int cnt = (int)((info >> 16) & 0xffu);
            const int counted = (int)(info >> 24);
            if (hop > D) break;
            for (int64_t x = h + lane; x < hop; x += 32) row[x] = N;  // distances before this group
            h = hop;
            const bool in = lane < counted && (!pred || pred[eid[e + lane]]);
            const int m = __popc(__ballot_sync(kFull, in));
            N = __dadd_rn(N, __dmul_rn((double)m, gwt[gi]));
            e += cnt;
        }
        for (int64_t x = h + lane; x <= D; x += 32) row[x] = N;
    }
}

// Scratch of the sweeps of one call.
struct XScratch {
    unsigned long long* vis;
    unsigned long long* buf[2];
    int32_t *light, *heavy;
    const int32_t* huge;
    int32_t* front[2];
    unsigned long long* huge_items;  // of the huge rows, n_huge + *n_more
    unsigned long long* n_more;
    unsigned long long* items;       // of a top-down level
    size_t n_items;
    void* state;
    int64_t n_light, n_heavy, n_huge;
};

// One sweep of nb <= 64 W sources; rows: the sizes of its first source.
template <int W>
int run_sweep(fl_graph* g, const XScratch& x, int mode, int64_t nb, const int32_t* src, int64_t D,
              const uint8_t* pred, const double* cost, int64_t* rows, double* radius) {
    cudaStream_t st = g->stream;
    const int64_t n = g->n, nnz = g->nnz;
    const int cls = kProfExact;
    const size_t words = (size_t)n * W;
    const int kS = 64 * W;
    Counters* ctr = g->ctr.as<Counters>();
    const int64_t* rowp = g->rowp.as<int64_t>();
    const int32_t* cols = g->cols.as<int32_t>();
    XState<W>* xs = static_cast<XState<W>*>(x.state);
    unsigned long long* vis = x.vis;
    unsigned long long* buf[2] = {vis + words, vis + 2 * words};
    int32_t* front[2] = {x.front[0], x.front[1]};
    const int grid_l = blocks_for(x.n_light, 256 / W, kXLevelBlocks);
    const int grid_h = blocks_for(x.n_heavy, 8, kXLevelBlocks);  // 8 warps x 1 vertex
    // a bottom-up level rewrites the next words of every vertex; a
    // top-down level gets them cleared first
    FL_CUDA(cudaMemsetAsync(vis, 0, words * 8, st));
    FL_CUDA(cudaMemsetAsync(buf[0], 0, words * 8, st));
    int c = 0, fc = 0;
    FL_LAUNCH(cls, k_x_seed<W><<<1, kS, 0, st>>>(src, nb, rowp, vis, buf[0], front[0], xs));
    FL_LAUNCH(cls, k_x_finish<W><<<1, kS, 0, st>>>(xs, mode, 0, src, pred, cost, D, rows, radius, ctr));
    FL_CUDA(cudaGetLastError());
    FL_TRY(read_counters(g));
    int64_t n_front = (int64_t)g->h_ctr->frontier;
    int64_t fr_edges = (int64_t)g->h_ctr->merges;
    int64_t rem = nnz;  // entries of rows that may still need bits
    unsigned long long rows_prev = 0, entries_prev = 0;
    for (int64_t level = 1; g->h_ctr->aux0 > 0; ++level) {
        if (level > n + 1) FL_FAIL(FL_ETIMEOUT, "exact search did not finish");
        // top-down when the frontier's rows are much shorter than the
        // rows bottom-up would scan, and their work items fit
        const bool td = 2 * fr_edges < rem && n_front + fr_edges / kXSeg + 1 <= (int64_t)x.n_items;
        if (td) {
            FL_CUDA(cudaMemsetAsync(buf[c ^ 1], 0, words * 8, st));
            // work items (their count in st->n_next), then the pushes;
            // k_x_td_finish restarts n_next for the next frontier
            FL_LAUNCH(cls, k_x_td_items<W><<<blocks_for(n_front, 256), 256, 0, st>>>(front[fc], n_front, rowp,
                                                                                    buf[c], x.items, xs));
            const int64_t most = n_front + fr_edges / kXSeg;  // work items at most
            FL_LAUNCH(cls, k_x_td<W><<<blocks_for(most, 8), 256, 0, st>>>(x.items, rowp, cols, buf[c], buf[c ^ 1],
                                                                          vis, xs));
            FL_CUDA(cudaMemsetAsync(&xs->n_next, 0, 8, st));
            FL_LAUNCH(cls, k_x_td_finish<W><<<blocks_for(n, 256 / W, kXLevelBlocks), 256, 0, st>>>(
                               n, rowp, buf[c ^ 1], vis, pred, front[fc ^ 1], xs));
        } else {
            if (x.n_huge > 0) {
                FL_LAUNCH(cls, k_x_huge_clear<W><<<blocks_for(x.n_huge, 256 / W), 256, 0, st>>>(x.huge, x.n_huge,
                                                                                              buf[c ^ 1]));
                FL_LAUNCH(cls, k_x_huge<W><<<blocks_for(x.n_huge + nnz / kXSeg, 8), 256, 0, st>>>(
                                   x.huge_items, x.n_huge, x.n_more, rowp, cols, buf[c], buf[c ^ 1], vis, xs));
                FL_LAUNCH(cls, k_x_huge_done<W><<<blocks_for(x.n_huge, 256 / W, kXLevelBlocks), 256, 0, st>>>(
                                   x.huge, x.n_huge, rowp, buf[c ^ 1], vis, pred, front[fc ^ 1], xs));
            }
            if (x.n_heavy > 0)
                FL_LAUNCH(cls, k_x_heavy<W><<<grid_h, 256, 0, st>>>(x.heavy, x.n_heavy, rowp, cols, buf[c],
                                                                    buf[c ^ 1], vis, pred, front[fc ^ 1], xs));
            if (x.n_light > 0)
                FL_LAUNCH(cls, k_x_light<W><<<grid_l, 256, 0, st>>>(x.light, x.n_light, rowp, cols, buf[c],
                                                                    buf[c ^ 1], vis, pred, front[fc ^ 1], xs));
        }
        FL_LAUNCH(cls, k_x_finish<W><<<1, kS, 0, st>>>(xs, mode, level, src, pred, cost, D, rows, radius, ctr));
        FL_CUDA(cudaGetLastError());
        c ^= 1;
        fc ^= 1;
        FL_TRY(read_counters(g));
        const int64_t touched = (int64_t)g->h_ctr->frontier;
        // algorithmic bytes of the level, B = 8 W bytes of bits per vertex.
        // Bottom-up: every listed vertex reads its list id and visited words
        // and writes its next words (4 + 2 B); a scanned row reads two offsets
        // (16) and, per entry, the column and the neighbour's frontier words
        // (4 + B).  Top-down: a frontier vertex reads its list id, frontier
        // words and offsets (4 + B + 16); per entry the column and the
        // neighbour's visited words (4 + B); every vertex reads its next words
        // (B) and a newly reached one reads and writes its visited words, reads
        // its offsets and is listed (2 B + 16 + 4).
        const double B = 8.0 * W;
        const double d_rows = (double)(g->h_ctr->scanned - rows_prev);
        const double d_entries = (double)(g->h_ctr->cand_reads - entries_prev);
        rows_prev = g->h_ctr->scanned;
        entries_prev = g->h_ctr->cand_reads;
        g->prof.bytes[cls] += td ? (20.0 + B) * (double)n_front + (4.0 + B) * d_entries + B * (double)n +
                                       (20.0 + 2.0 * B) * (double)touched
                                 : (4.0 + 2.0 * B) * (double)n + 16.0 * d_rows + (4.0 + B) * d_entries;
        n_front = touched;
        fr_edges = (int64_t)g->h_ctr->merges;
        if (!td) rem = (int64_t)g->h_ctr->aux3;
    }
    return FL_OK;
}

// Sweeps over src[0, n_src) (internal ids).
int run_sweeps(fl_graph* g, int mode, int64_t n_src, const int32_t* src, int64_t D, const uint8_t* pred,
               const double* cost, int64_t* sizes, double* radius) {
    cudaStream_t st = g->stream;
    const int64_t n = g->n, nnz = g->nnz;
    // the smallest W that takes what is left
    auto width = [&](int64_t left) { return left <= 256 || n > kXWideN ? 4 : (left <= 512 ? 8 : 16); };
    const int w_max = width(n_src);
    constexpr int64_t kMost = 64 * kXMaxW;
    FL_TRY(dalloc(g->xbits, (size_t)n * w_max * 8 * 3));
    // int32 lists: light rows (n), heavy rows from the front and huge ones from
    // the back (n), two frontiers (n + kMost each: the first frontier lists the
    // sweep's sources, repeats included); then the top-down work items (uint64,
    // one per kXSeg entries of a frontier row: at most n + kMost + nnz / kXSeg),
    // those of the huge rows (at most 2 nnz / kXSeg), their number and the sweep state
    const size_t lists = ((size_t)(4 * n + 2 * kMost) * 4 + 255) & ~(size_t)255;
    XScratch x;
    x.n_items = (size_t)(n + kMost + nnz / kXSeg + 1);
    const size_t items_b = (x.n_items * 8 + 255) & ~(size_t)255;
    const size_t huge_b = ((size_t)(2 * (nnz / kXSeg) + 1) * 8 + 255) & ~(size_t)255;
    FL_TRY(dalloc(g->xaux, lists + items_b + huge_b + 256 + sizeof(XState<kXMaxW>)));
    x.vis = g->xbits.as<unsigned long long>();
    x.light = g->xaux.as<int32_t>();
    x.heavy = x.light + n;
    x.front[0] = x.light + 2 * n;
    x.front[1] = x.light + 3 * n + kMost;
    x.items = reinterpret_cast<unsigned long long*>(g->xaux.as<char>() + lists);
    x.huge_items = reinterpret_cast<unsigned long long*>(g->xaux.as<char>() + lists + items_b);
    x.state = g->xaux.as<char>() + lists + items_b + huge_b + 256;
    x.n_more = reinterpret_cast<unsigned long long*>(g->xaux.as<char>() + lists + items_b + huge_b);
    Counters* ctr = g->ctr.as<Counters>();
    FL_CUDA(cudaMemsetAsync(g->ctr.p, 0, sizeof(Counters), st));
    FL_LAUNCH(kProfExact, k_x_lists<<<blocks_for(n, 256), 256, 0, st>>>(g->rowp.as<int64_t>(), n, x.light, x.heavy,
                                                                      &ctr->aux0, &ctr->aux3, &ctr->frontier));
    FL_CUDA(cudaGetLastError());
    FL_TRY(read_counters(g));
    x.n_light = (int64_t)g->h_ctr->aux0;
    x.n_heavy = (int64_t)g->h_ctr->aux3;
    x.n_huge = (int64_t)g->h_ctr->frontier;
    x.huge = x.heavy + n - x.n_huge;
    if (x.n_huge > 0) {
        FL_CUDA(cudaMemsetAsync(x.n_more, 0, 8, st));
        FL_LAUNCH(kProfExact, k_x_huge_items<<<blocks_for(x.n_huge, 8), 256, 0, st>>>(
                                  x.huge, x.n_huge, g->rowp.as<int64_t>(), x.huge_items, x.n_more));
        FL_CUDA(cudaGetLastError());
    }
    for (int64_t b0 = 0; b0 < n_src;) {
        const int w = width(n_src - b0);
        const int64_t nb = std::min<int64_t>(n_src - b0, 64 * w);
        int64_t* rows = sizes ? sizes + b0 * (D + 1) : nullptr;
        auto sweep = w == 4 ? run_sweep<4> : (w == 8 ? run_sweep<8> : run_sweep<16>);
        FL_TRY(sweep(g, x, mode, nb, src + b0, D, pred, cost, rows, radius));
        b0 += nb;
    }
    return FL_OK;
}

}  // namespace

int map_sources(fl_graph* g, const int32_t* in, int64_t n_src, int32_t* out) {
    cudaStream_t st = g->stream;
    FL_CUDA(cudaMemsetAsync(g->ctr.p, 0, sizeof(Counters), st));
    FL_LAUNCH(kProfExact, k_x_map<<<blocks_for(n_src, 256), 256, 0, st>>>(
                              in, n_src, g->relabelled ? g->inv.as<int32_t>() : nullptr, g->n, out,
                              g->ctr.as<Counters>()));
    FL_CUDA(cudaGetLastError());
    FL_TRY(read_counters(g));
    if (g->h_ctr->error) FL_FAIL(FL_EINVAL, "source ids must lie in [0, n)");
    return FL_OK;
}

int exact_ball_sizes(fl_graph* g, int64_t n_src, const int32_t* src, int64_t D, const uint8_t* pred, int64_t* out) {
    if (n_src == 0) return FL_OK;
    return run_sweeps(g, kXSizes, n_src, src, D, pred, nullptr, out, nullptr);
}

int hip_ball_estimates(fl_graph* g, int64_t n_src, const int32_t* src, int64_t D, const uint8_t* pred, double* out) {
    if (n_src == 0) return FL_OK;
    FL_LAUNCH(kProfExact, k_x_estimates<<<blocks_for(n_src, 8), 256, 0, g->stream>>>(
                              src, n_src, D, pred, g->gofs.as<int64_t>(), g->eofs.as<int64_t>(),
                              g->ginfo.as<uint32_t>(), g->gwt.as<double>(), g->eid.as<int32_t>(), out));
    FL_CUDA(cudaGetLastError());
    return FL_OK;
}

int exact_radii(fl_solve* s) {
    fl_graph* g = s->g;
    cudaStream_t st = g->stream;
    const int64_t n = g->n;
    FL_TRY(dalloc(s->ulist, (size_t)n * 4 * 2));  // facility list (the MIS reuses the buffer later)
    int32_t* fac = s->ulist.as<int32_t>();
    FL_CUDA(cudaMemsetAsync(g->ctr.p, 0, sizeof(Counters), st));
    FL_LAUNCH(kProfExact, k_x_facilities<<<blocks_for(n, 256), 256, 0, st>>>(s->cost.as<double>(), n, fac,
                                                                            s->radii.as<double>(),
                                                                            g->ctr.as<Counters>()));
    FL_CUDA(cudaGetLastError());
    FL_TRY(read_counters(g));
    if (g->h_ctr->error) FL_FAIL(FL_EINVAL, "open_cost must be finite and > 0 for facilities, +inf otherwise");
    const int64_t m = (int64_t)g->h_ctr->aux0;
    if (m == 0) return FL_OK;
    return run_sweeps(g, kXRadius, m, fac, 0, s->client.as<uint8_t>(), s->cost.as<double>(), nullptr,
                      s->radii.as<double>());
}

}  // namespace fl

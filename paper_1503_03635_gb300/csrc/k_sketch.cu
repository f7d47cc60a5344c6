// k_sketch.cu -- phase (i): bottom-k sketches and ADS by hop-synchronous
// propagation (Section 3.3, Algorithm 2 for unweighted graphs), with HIP
// weights computed where each entry joins a sketch.
//
// Ranks enter a sketch only by their order, so the hops work on ordinals: the
// ranks r(v) are sorted once, and a vertex is known by the place of its rank
// (32 bits in place of 64 in every list, load, shuffle and compare, and the
// small ranks that the masks below cover are simply the ordinals below kUW).
// The rank itself is computed again where an HIP weight or an export needs it.
//
// Data layout (k <= 32):
//   ord[v]            ordinal of vertex v's rank (in a union: of its local id's)
//   ord_rid[o]        rank id of ordinal o
//   S[v*k + i]        current sketch of v, ascending ordinals, kNil padding
//   Scnt[v]           number of ordinals in S[v]
//   D[p][v*k + i]     entries v gained at the previous / current hop, kNil padding
//   Dcnt[p][v]        their number (0 = v is not in the frontier)
//   staging           one group slot per work item of every hop >= 1 (v, hop,
//                     counts, the sketch's k-th ordinal) and k entry slots
//                     (ordinals); compacted into the vertex-major ADS, with
//                     HIP weights and vertex ids, after the last hop
//
// Work decomposition of one hop.  A group of G lanes (G = 16 when k <= 16,
// else 32) owns one vertex: lane i holds S[v][i].  Non-hub vertices are
// processed directly (k_hop_vertices).  Hubs (degree > fl_graph::seg) are cut into
// segments of that many edges; each segment yields a partial bottom-k of its
// candidates in scratch (k_hop_hub_segments), and one group per hub merges
// the partials into the hub's sketch (k_hop_hubs).  Bottom-k of a union is the
// bottom-k of the union of bottom-k's, so the split does not change results.
//
// What bounds the hops: instructions in the list merges (hops 1-3 of an R-MAT
// graph, all of an Erdos-Renyi graph's), the chain column -> bitmap -> mask
// word in the mask and head merges.  Per build, against 64-bit ranks and
// half-warp groups that diverged: non-hub vertices of R-MAT 24 (k = 16) 49.2
// -> 32.1 ms, hub segments 9.8 -> 7.1; R-MAT 20 (k = 32) 5.4 -> 3.6; 64
// Erdos-Renyi graphs (k = 32) 14.9 -> 7.0.  With weights and ids left to the
// compaction and six blocks per SM in place of four (latency of the gathers):
// 25.5, 2.9 and 6.0 ms.  The sort of the ranks adds 0.3 ms
// at 2^20 vertices, 2.0 at 2^24.
#include <algorithm>
#include <cstdio>
#include <vector>

#include "fl_internal.cuh"

namespace fl {

// A staged group; its HIP weight is computed at the compaction from its
// sketch's k-th ordinal (kNil: fewer than k entries), kept beside it.
struct __align__(16) StgGroup {
    int32_t v;      // vertex
    int32_t gidx;   // index of this group among v's groups
    int32_t eidx;   // index of its first entry among v's entries
    uint32_t info;  // hop | cnt << 16 | counted << 24; 0 = empty slot
};

__host__ __device__ __forceinline__ uint32_t pack_info(int hop, int cnt, int counted) {
    return (uint32_t)hop | ((uint32_t)cnt << 16) | ((uint32_t)counted << 24);
}

constexpr int kMaxHops = 65535;
constexpr int64_t kCountMax = 16384;    // more ranks than this go through the radix sort

// ------------------------------------------------------------------ small-ordinal masks
// A sketch whose k-th ordinal is below kUW ("saturated") holds only ordinals
// below kUW, and so does every candidate that can still enter it: the sketch
// is a kUW-bit mask, and one hop is S_h(v) = lowest k bits of (S_{h-1}(v) |
// OR_{u in N(v)} D_{h-1}(u)), with D_{h-1}(u) kept as a mask beside its list.
// Candidates at or above kUW are above the k-th ordinal and drop out either
// way, so the mask update is the list merge exactly.  Masks are merged in
// 256-bit slices from the smallest ordinals up, stopping once k bits are kept:
// a sketch whose k-th ordinal lies in the first slice reads 32 bytes per
// neighbour.

constexpr int kSliceWords = 8;  // 32-bit words of a slice

// Lane l's word l mod 8 of the OR over the group of the lanes' slices: each
// exchange halves the words a lane still holds (8 shuffles for 16 lanes, 40
// for the OR of every word on every lane).
template <int G>
__device__ __forceinline__ uint32_t slice_or(const Lock<G>& g, const uint32_t (&w)[kSliceWords]) {
    uint32_t a[4], b[2];
    const bool h4 = (g.l & 4) != 0, h2 = (g.l & 2) != 0, h1 = (g.l & 1) != 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = (h4 ? w[i + 4] : w[i]) | g.shfl_xor(h4 ? w[i] : w[i + 4], 4);
#pragma unroll
    for (int i = 0; i < 2; ++i) b[i] = (h2 ? a[i + 2] : a[i]) | g.shfl_xor(h2 ? a[i] : a[i + 2], 2);
    uint32_t r = (h1 ? b[1] : b[0]) | g.shfl_xor(h1 ? b[0] : b[1], 1);
    r |= g.shfl_xor(r, 8);
    if (G == 32) r |= g.shfl_xor(r, 16);
    return r;
}

// The lane's entry `x` into its words of slice q.
__device__ __forceinline__ void slice_set(uint32_t (&w)[kSliceWords], uint32_t x, int q) {
    const uint32_t bit = (x >> 8) == (uint32_t)q ? 1u << (x & 31) : 0u;
#pragma unroll
    for (int i = 0; i < kSliceWords; ++i)
        if (((x >> 5) & 7) == (uint32_t)i) w[i] |= bit;
}

// Slice q of a merged mask (r: lane l holds word l mod 8): its lowest `left`
// bits go to the lanes base, base + 1, ... of sk.  Returns the bits taken.
template <int G>
__device__ __forceinline__ int slice_emit(const Lock<G>& g, uint32_t r, int q, int base, int left, uint32_t& sk) {
    const int c = __popc(r);
    int incl = c;
#pragma unroll
    for (int s = 1; s < 8; s <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, s, 8);
        if ((g.l & 7) >= s) incl += y;
    }
    const int take = min(g.shfl(incl, 7), left);
    const int j = g.l - base;
    int wl = 0;
#pragma unroll
    for (int s = 4; s > 0; s >>= 1)
        if (g.shfl(incl, wl + s - 1) <= j) wl += s;
    const uint32_t word = g.shfl(r, wl);
    const int before = g.shfl(incl - c, wl);
    if (j >= 0 && j < take) sk = (uint32_t)(q * 256 + wl * 32 + nth_set_bit(word, j - before));
    return max(take, 0);
}

// ------------------------------------------------------------------ per-hop inputs and outputs

// Per-group hop counters in shared memory, one slot per group, updated by
// the group's lane 0 without atomics and flushed once at the end of a kernel
// (counters in registers cost spills in the merge loops).  32-bit: a group
// adds at most 32 * kMaxSeg per vertex it processes (hub degrees go to the
// global counters directly) and, with the grids of the hop kernels, processes
// at most 2^31 / 77824 < 2^16 work items.
enum { kCFront, kCMerges, kCMerging, kCDelta, kCNew, kNCtr };  // in the order of flush_counters

// Shared memory of a hop kernel (256 threads).
struct HopShared {
    unsigned ctr[256 / 16][kNCtr];
    unsigned cand[8];            // per warp
    uint32_t x[8][32];           // per warp: merged candidates by place
    uint32_t mask[256 / 16][32];  // per group: a delta mask
};

// p = previous hop's buffers, read-only during a hop; c = this hop's.  Besides
// each vertex's delta list D (padded with kNil) and delta mask DM, two dense
// per-vertex words make the per-edge reads small and cache-friendly:
//   F[u]  the smallest ordinal u gained at the hop (kNil: none), the filter of
//         the list merge: a neighbour whose F is not below the vertex's k-th
//         ordinal cannot change its sketch;
//   H[u]  the bits of u's delta mask over the ordinals 0..63 (word 0 of DM);
// and W[v], the mask of v's own sketch once the sketch is full and its k-th
// ordinal is below 64 ("head" vertices; 0 otherwise).  A head vertex takes
// S_h(v) = lowest k bits of (W[v] | OR_u H[u]): every candidate that can still
// enter is below 64, so this is the list merge's result.  Frontier membership
// comes from a bitmap of the previous hop's frontier (n/8 bytes,
// cache-resident).
struct HopIO {
    const int64_t* __restrict__ rowp;
    const int32_t* __restrict__ cols;
    int k;
    int hop;
    int seg;                                 // longest row that is not a hub's, and edges per hub segment
    const uint32_t* __restrict__ ord;        // ordinal of each vertex
    uint32_t* __restrict__ S;
    uint8_t* __restrict__ Scnt;
    const uint32_t* __restrict__ Dp;
    uint32_t* __restrict__ Dc;
    uint8_t* __restrict__ Dcc;
    const uint32_t* __restrict__ Fp;
    uint32_t* __restrict__ Fc;
    const uint64_t* __restrict__ Hp;
    uint64_t* __restrict__ Hc;
    uint64_t* __restrict__ W;
    const uint32_t* __restrict__ bm;
    const uint64_t* __restrict__ DMp;  // slice-major: slice q of vertex v at [(q * n + v) * 4]
    uint64_t* __restrict__ DMc;
    int64_t n;
    int32_t* __restrict__ vg;
    int32_t* __restrict__ ve;
    uint32_t* __restrict__ stg_ent;
    uint32_t* __restrict__ stg_kth;
    StgGroup* __restrict__ stg_grp;
    Counters* ctr;
};

__device__ __forceinline__ bool in_bitmap(const uint32_t* __restrict__ bm, int32_t u) {
    return (__ldg(&bm[u >> 5]) >> (u & 31)) & 1u;
}

// Position of the n-th (0-based) set bit of a 64-bit word (n < popcount).
__device__ __forceinline__ int nth_bit64(uint64_t x, int n) {
    const unsigned lo = (unsigned)x;
    const int c = __popc(lo);
    return n < c ? nth_set_bit(lo, n) : 32 + nth_set_bit((unsigned)(x >> 32), n - c);
}

// The lowest k set bits of x.
__device__ __forceinline__ uint64_t lowest_k64(uint64_t x, int k) {
    return __popcll(x) <= k ? x : x & ((1ULL << nth_bit64(x, k)) - 1ULL);
}

// Word w of vertex v's delta mask in the slice-major layout (each 256-bit
// slice of all vertices is one dense array, so that the hot slices of
// high-degree vertices share cache lines).
__device__ __forceinline__ int64_t dm_word(int64_t n, int64_t v, int w) {
    return ((int64_t)(w >> 2) * n + v) * 4 + (w & 3);
}

// The lanes' shares of slice q of the delta masks of the neighbours in
// [e0, e1) that gained entries at the previous hop are ORed into w (four
// columns per lane in flight); `front`: the lane saw such a neighbour.
template <int G>
__device__ __forceinline__ void gather_slice(const Lock<G>& g, const HopIO& io, int64_t e0, int64_t e1, int q,
                                             uint32_t (&w)[kSliceWords], bool& front, unsigned& cand) {
    const uint64_t* __restrict__ slice = io.DMp + (int64_t)q * io.n * 4;
    for (int64_t e = e0 + g.l; e < e1; e += 4 * G) {
        int32_t u[4];
        bool in[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) u[j] = e + j * G < e1 ? __ldcs(&io.cols[e + j * G]) : -1;
#pragma unroll
        for (int j = 0; j < 4; ++j) in[j] = u[j] >= 0 && in_bitmap(io.bm, u[j]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (in[j]) {
                const uint4* p = reinterpret_cast<const uint4*>(slice + (int64_t)u[j] * 4);
                const uint4 a = __ldg(p), b = __ldg(p + 1);
                w[0] |= a.x;
                w[1] |= a.y;
                w[2] |= a.z;
                w[3] |= a.w;
                w[4] |= b.x;
                w[5] |= b.y;
                w[6] |= b.z;
                w[7] |= b.w;
                front = true;
                cand += 4u;
            }
        }
    }
}

// OR over the lane's share of the delta heads H[u] of the neighbours in
// [e0, e1) that are in the previous hop's frontier.
template <int G>
__device__ __forceinline__ uint64_t gather_heads(const Lock<G>& g, const HopIO& io, int64_t e0, int64_t e1,
                                                 bool& front, unsigned& cand) {
    uint64_t acc = 0;
    for (int64_t e = e0 + g.l; e < e1; e += 4 * G) {
        int32_t u[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) u[j] = e + j * G < e1 ? __ldcs(&io.cols[e + j * G]) : -1;
        bool in[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) in[j] = u[j] >= 0 && in_bitmap(io.bm, u[j]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (in[j]) {
                acc |= __ldg(&io.Hp[u[j]]);
                front = true;
                cand += 1u;
            }
        }
    }
    return acc;
}

// ------------------------------------------------------------------ hop 0

// Hop 0: S_0(v) = {ord(v)}.  (Hop 1 reads the neighbours' ordinals, so no
// hop-0 delta list or mask is stored; v's group at distance 0, the entry v
// alone, is written by the compaction.)
__global__ void k_rank_init(int64_t n, int k, const uint32_t* __restrict__ ord, uint32_t* __restrict__ S,
                            uint8_t* __restrict__ Scnt, int32_t* __restrict__ vg, int32_t* __restrict__ ve) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        S[v * k] = ord[v];
        Scnt[v] = 1;
        vg[v] = 1;
        ve[v] = 1;
    }
}

// ------------------------------------------------------------------ group sketch updates

// Absorb the candidates of CSR entries [e0, e1) (e0 >= e1: none): at hop 1 the
// neighbours' own ordinals, later the entries each neighbour gained at the
// previous hop.  Lane j of the group owns neighbour j of a chunk of G
// neighbours and loads its smallest new ordinal F[u] (independent loads into a
// dense array that also filter whole lists).  The lists of the neighbours that
// pass are loaded across the group, four in flight, and merged one after the
// other.  `front`: the lane saw a neighbour that gained entries.
template <int G>
__device__ __forceinline__ void gather_lists(const Lock<G>& g, const HopIO& io, int64_t e0, int64_t e1,
                                             Sketch<G>& s, bool& front, unsigned& cand, uint32_t* sx) {
    const int k = io.k;
    if (io.hop == 1) {
        front |= e0 < e1;
        for (int64_t cb = e0; warp_any(cb < e1); cb += 2 * G) {
            const int64_t e = cb + g.l;
            const int32_t u0 = e < e1 ? __ldcs(&io.cols[e]) : -1, u1 = e + G < e1 ? __ldcs(&io.cols[e + G]) : -1;
            const uint32_t x0 = u0 >= 0 ? __ldg(&io.ord[u0]) : kNil, x1 = u1 >= 0 ? __ldg(&io.ord[u1]) : kNil;
            absorb(g, k, x0, s, sx);
            absorb(g, k, x1, s, sx);
        }
        return;
    }
    // the next chunk's columns are loaded while this chunk merges
    int32_t u_next = e0 + g.l < e1 ? __ldcs(&io.cols[e0 + g.l]) : -1;
    for (int64_t cb = e0; warp_any(cb < e1); cb += G) {
        const int32_t u = u_next;
        const int64_t e = cb + G + g.l;
        u_next = e < e1 ? __ldcs(&io.cols[e]) : -1;
        const uint32_t first = u >= 0 ? __ldg(&io.Fp[u]) : kNil;
        front |= first != kNil;
        cand += first != kNil ? 1u : 0u;
        unsigned live = g.ballot(first < s.tau);
        while (warp_any(live != 0)) {
            uint32_t x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int j = live ? __ffs(live) - 1 : 0;
                const int32_t uj = g.shfl(u, j);
                x[q] = live && g.l < k ? __ldg(&io.Dp[(int64_t)uj * k + g.l]) : kNil;
                live &= live - 1;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                cand += x[q] != kNil ? 1u : 0u;
                merge_list(g, k, x[q], s, sx);
            }
            live &= g.ballot(first < s.tau);  // the filter tightened since
        }
    }
}

// Saturated merge, slice by slice from the smallest ordinals: src(q, w) ORs
// the candidates' shares of slice q into w, `old` is the lane's old entry.
// Lanes j < k receive the new sketch; groups that are not `on` keep theirs.
template <int G, class Src>
__device__ __forceinline__ void merge_slices(const Lock<G>& g, int k, bool on, Src src, uint32_t& sk) {
    const uint32_t old = sk;
    uint32_t nw = kNil;
    int left = on ? k : 0, base = 0;
    for (int q = 0; q < kUSlices && warp_any(left > 0); ++q) {
        uint32_t w[kSliceWords];
#pragma unroll
        for (int i = 0; i < kSliceWords; ++i) w[i] = 0u;
        if (left > 0) {
            slice_set(w, old, q);
            src(q, w);
        }
        const int c = slice_emit(g, slice_or(g, w), q, base, left, nw);
        base += c;
        left -= c;
    }
    if (on) sk = nw;
}

// Record a changed vertex's ADS group in staging slot `slot` and count it
// (lane 0 of the group).
template <int G>
__device__ __forceinline__ void stage_group(const HopIO& io, HopShared& sh, int32_t v, int64_t deg, int64_t slot,
                                            int dcnt, int counted, uint32_t kth) {
    StgGroup gr;
    gr.v = v;
    gr.gidx = io.vg[v];
    gr.eidx = io.ve[v];
    gr.info = pack_info(io.hop, dcnt, counted);
    io.vg[v] = gr.gidx + 1;
    io.ve[v] = gr.eidx + dcnt;
    io.stg_grp[slot] = gr;
    io.stg_kth[slot] = kth;
    unsigned* c = sh.ctr[threadIdx.x / G];
    c[kCFront] += 1u;
    c[kCNew] += (unsigned)dcnt;
    if (deg <= io.seg) {
        c[kCMerges] += (unsigned)deg;
        c[kCDelta] += (unsigned)(deg * dcnt);
    }
}

// Write the results of vertex v (groups that are `on`) after a list or slice
// merge: new sketch, the entries it gained (list, mask, head word, smallest
// one, for the next hop), its own head mask once the sketch is a head sketch,
// and its staged ADS group in work slot `slot`.  Returns the number of entries
// gained (0: the sketch is unchanged).
template <int G>
__device__ __forceinline__ int finish_vertex(const Lock<G>& g, const HopIO& io, HopShared& sh, bool on, int32_t v,
                                             int64_t deg, uint32_t old, uint32_t sk, int64_t slot) {
    const int k = io.k;
    const bool valid = g.l < k && sk != kNil;
    bool was_there;
    lock_find(g, old, sk, was_there);
    const unsigned newm = g.ballot(on && valid && !was_there);
    const int dcnt = __popc(newm);
    if (on && dcnt == 0 && g.l == 0) io.stg_grp[slot].info = 0;  // empty slot
    if (!warp_any(dcnt > 0)) return 0;
    const bool wr = dcnt > 0, is_new = (newm >> g.l) & 1u;
    uint32_t* m = sh.mask[threadIdx.x / G];
    m[g.l] = 0u;
    if (G == 16) m[g.l + 16] = 0u;
    __syncwarp();
    if (is_new && sk < (uint32_t)kUW) atomicOr(&m[sk >> 5], 1u << (sk & 31));
    __syncwarp();
    if (wr) {
        if (g.l < k) io.S[(int64_t)v * k + g.l] = sk;
        if (is_new) {
            const int at = __popc(newm & g.below());
            io.Dc[(int64_t)v * k + at] = sk;
            io.stg_ent[slot * k + at] = sk;
        }
        if (g.l < k && g.l >= dcnt) io.Dc[(int64_t)v * k + g.l] = kNil;
        if (g.l < kUWords)
            io.DMc[dm_word(io.n, v, g.l)] = ((uint64_t)m[2 * g.l + 1] << 32) | m[2 * g.l];
    }
    const int cnt_new = __popc(g.ballot(valid));
    const uint32_t kth = g.shfl(sk, k - 1);
    const uint32_t least = g.shfl(sk, wr ? __ffs(newm) - 1 : 0);
    // a full sketch whose k-th ordinal is below 64 becomes a head vertex
    const bool head = wr && cnt_new == k && kth < 64u;
    if (warp_any(head)) {
        const uint64_t own = lock_or64(g, valid && sk < 64u ? 1ULL << sk : 0ULL);
        if (head && g.l == 0) io.W[v] = own;
    }
    if (wr && g.l == 0) {
        io.Fc[v] = least;
        io.Hc[v] = ((uint64_t)m[1] << 32) | m[0];
        io.Scnt[v] = (uint8_t)cnt_new;
        io.Dcc[v] = (uint8_t)dcnt;
        const int counted = cnt_new < k ? dcnt : __popc(newm & ((1u << (k - 1)) - 1u));
        stage_group<G>(io, sh, v, deg, slot, dcnt, counted, kth);
    }
    __syncwarp();
    return dcnt;
}

// Write the results of head vertex v whose new sketch is the mask nw over the
// ordinals 0..63 (k bits) with gained bits delta (nonzero); the same outputs
// as finish_vertex.
template <int G>
__device__ __forceinline__ void finish_head(const Lock<G>& g, const HopIO& io, HopShared& sh, int32_t v, int64_t deg,
                                            uint64_t nw, uint64_t delta, int64_t slot) {
    const int k = io.k;
    const int dcnt = __popcll(delta);
    if (g.l < k) {
        io.S[(int64_t)v * k + g.l] = (uint32_t)nth_bit64(nw, g.l);
        uint32_t x = kNil;
        if (g.l < dcnt) {
            x = (uint32_t)nth_bit64(delta, g.l);
            io.stg_ent[slot * k + g.l] = x;
        }
        io.Dc[(int64_t)v * k + g.l] = x;
    }
    if (g.l < kUWords) io.DMc[dm_word(io.n, v, g.l)] = g.l == 0 ? delta : 0ULL;
    if (g.l == 0) {
        const int top = 63 - __clzll(nw);  // the k-th ordinal
        io.W[v] = nw;
        io.Fc[v] = (uint32_t)(__ffsll(delta) - 1);
        io.Hc[v] = delta;
        io.Dcc[v] = (uint8_t)dcnt;
        const int counted = dcnt - (int)((delta >> top) & 1ULL);
        stage_group<G>(io, sh, v, deg, slot, dcnt, counted, (uint32_t)top);
    }
}

template <int G>
__device__ __forceinline__ void ctr_init(const Lock<G>& g, HopShared& sh) {
    if (g.l == 0)
        for (int i = 0; i < kNCtr; ++i) sh.ctr[threadIdx.x / G][i] = 0;
    __syncwarp();
}

// End of a hop kernel (every thread calls): the groups' counters, one atomic
// per counter and block.  (An atomic per counter and group put 60 k adds on one
// line: 100 us of a 130 us hop on a graph with 61 k vertices.)
__device__ __forceinline__ void flush_counters(HopShared& sh, int groups, unsigned cand, Counters* ctr) {
    cand = __reduce_add_sync(kFull, cand);
    if (lane_id() == 0) sh.cand[threadIdx.x >> 5] = cand;
    __syncthreads();
    if (threadIdx.x < kNCtr) {
        unsigned long long x = 0;
        for (int i = 0; i < groups; ++i) x += sh.ctr[i][threadIdx.x];
        unsigned long long* to[kNCtr] = {&ctr->frontier, &ctr->merges, &ctr->merging, &ctr->delta_next,
                                         &ctr->new_entries};
#pragma unroll
        for (int c = 0; c < kNCtr; ++c)
            if (threadIdx.x == c && x) atomicAdd(to[c], x);
    } else if (threadIdx.x == 32) {
        unsigned long long x = 0;
        for (int w = 0; w < 8; ++w) x += sh.cand[w];
        if (x) atomicAdd(&ctr->cand_reads, x);
    }
}

// ------------------------------------------------------------------ hop kernels

// Non-hub vertices: S_h(v) = bottom-k(S_{h-1}(v) U union_{u in N(v)} D_{h-1}(u)),
// by the head merge (head vertices), the mask merge (other saturated
// sketches) or the list merge.  The groups of a warp take part in each merge
// that one of them needs.
template <int G>
__global__ void __launch_bounds__(256, 6) k_hop_vertices(const int32_t* __restrict__ list, int64_t n_list, HopIO io) {
    __shared__ HopShared sh;
    const Lock<G> g;
    uint32_t* sx = sh.x[threadIdx.x >> 5];
    const int k = io.k;
    const int64_t groups = ((int64_t)gridDim.x * blockDim.x) / G;
    unsigned cand = 0;
    ctr_init(g, sh);
    const int64_t first = ((int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) / G;  // the warp's first group
    // the next vertex's id and row are loaded while this one merges
    const int64_t at0 = first + g.shift / G;
    int32_t v_next = at0 < n_list ? list[at0] : 0;
    int64_t beg_next = at0 < n_list ? io.rowp[v_next] : 0, end_next = at0 < n_list ? io.rowp[v_next + 1] : 0;
    for (int64_t i0 = first; i0 < n_list; i0 += groups) {
        const int64_t i = i0 + g.shift / G;
        const bool on = i < n_list, more = i + groups < n_list;
        const int32_t v = v_next;
        const int64_t beg = beg_next, end = end_next;
        v_next = more ? list[i + groups] : 0;
        const uint64_t wv = on && io.hop > 1 ? io.W[v] : 0ULL;
        bool front = false;
        if (warp_any(wv != 0)) {
            // head vertices: the head merge
            const bool head = wv != 0;
            const uint64_t acc = lock_or64(g, gather_heads(g, io, beg, head ? end : beg, front, cand));
            if (head) {
                const uint64_t nw = lowest_k64(wv | acc, k);
                const uint64_t delta = nw & ~wv;
                if (delta != 0) finish_head(g, io, sh, v, end - beg, nw, delta, i);
                else if (g.l == 0) io.stg_grp[i].info = 0;  // unchanged: empty slot
            }
        }
        const bool rest = on && wv == 0;
        if (warp_any(rest)) {
            const uint32_t old = rest && g.l < k ? io.S[(int64_t)v * k + g.l] : kNil;
            Sketch<G> s;
            s.sk = old;
            s.tau_base = kNil;
            s.retau(g, k);
            const bool sat = rest && io.hop > 1 && s.tau < (uint32_t)kUW;
            if (warp_any(sat))  // saturated: mask merge
                merge_slices(
                    g, k, sat,
                    [&](int q, uint32_t(&w)[kSliceWords]) { gather_slice(g, io, beg, end, q, w, front, cand); }, s.sk);
            if (warp_any(rest && !sat)) {
                s.retau(g, k);
                gather_lists(g, io, beg, rest && !sat ? end : beg, s, front, cand, sx);
            }
            beg_next = more ? io.rowp[v_next] : 0;
            end_next = more ? io.rowp[v_next + 1] : 0;
            finish_vertex(g, io, sh, rest, v, end - beg, old, s.sk, i);
        } else {
            beg_next = more ? io.rowp[v_next] : 0;
            end_next = more ? io.rowp[v_next + 1] : 0;
        }
        if (g.ballot(front) != 0 && g.l == 0) sh.ctr[threadIdx.x / G][kCMerging] += 1u;
    }
    flush_counters(sh, 256 / G, cand, io.ctr);
}

// Hub segments: partial results of one segment, written per segment -- the
// OR of its neighbours' delta heads (head hubs), the slices of their delta
// masks up to the hub's k-th ordinal (other saturated hubs), or the bottom-k
// of its candidates below the hub's old k-th ordinal (list hubs).
template <int G>
__global__ void __launch_bounds__(256) k_hop_hub_segments(const int32_t* __restrict__ hubs,
                                                             const int64_t* __restrict__ hub_seg,
                                                             const int32_t* __restrict__ seg_hub, int64_t n_seg,
                                                             uint32_t* __restrict__ part, uint32_t* __restrict__ PM,
                                                             uint64_t* __restrict__ PH, uint8_t* __restrict__ seg_flag,
                                                             const uint32_t* __restrict__ hub_stamp,
                                                             uint32_t sparse_hop, HopIO io) {
    __shared__ HopShared sh;
    const Lock<G> g;
    uint32_t* sx = sh.x[threadIdx.x >> 5];
    const int k = io.k;
    const int64_t groups = ((int64_t)gridDim.x * blockDim.x) / G;
    unsigned cand = 0;
    ctr_init(g, sh);
    const int64_t first = ((int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) / G;
    for (int64_t i0 = first; i0 < n_seg; i0 += groups) {
        const int64_t sidx = i0 + g.shift / G;
        bool on = sidx < n_seg;
        const int32_t h = on ? seg_hub[sidx] : 0;
        const int32_t v = on ? hubs[h] : 0;
        if (on && sparse_hop && hub_stamp[v] != sparse_hop) {
            // sparse hop: no neighbour of this hub gained entries
            if (g.l == 0) seg_flag[sidx] = 0;
            on = false;
        }
        const int64_t e0 = on ? io.rowp[v] + (sidx - hub_seg[h]) * io.seg : 0;
        const int64_t e1 = on ? min(e0 + (int64_t)io.seg, io.rowp[v + 1]) : 0;
        const bool head = on && io.hop > 1 && io.W[v] != 0;
        bool front = false;
        if (warp_any(head)) {
            const uint64_t acc = lock_or64(g, gather_heads(g, io, e0, head ? e1 : e0, front, cand));
            if (head && g.l == 0) PH[sidx] = acc;
        }
        const bool rest = on && !head;
        if (warp_any(rest)) {
            const uint32_t kth_old = rest ? io.S[(int64_t)v * k + k - 1] : kNil;  // kNil: not full
            const bool sat = rest && io.hop > 1 && kth_old < (uint32_t)kUW;
            if (warp_any(sat)) {
                // saturated hub: partial masks of the segment, the slices up to
                // the one holding the hub's k-th ordinal (the merge stops there)
                const int top = sat ? (int)(kth_old >> 8) : -1;
                for (int q = 0; warp_any(q <= top); ++q) {
                    uint32_t w[kSliceWords];
#pragma unroll
                    for (int j = 0; j < kSliceWords; ++j) w[j] = 0u;
                    if (q <= top) gather_slice(g, io, e0, e1, q, w, front, cand);
                    const uint32_t r = slice_or(g, w);
                    if (q <= top && g.l < kSliceWords) PM[sidx * 2 * kUWords + q * kSliceWords + g.l] = r;
                }
            }
            if (warp_any(rest && !sat)) {
                Sketch<G> s;
                s.sk = kNil;
                s.tau_base = kth_old;
                s.tau = kth_old;
                gather_lists(g, io, e0, rest && !sat ? e1 : e0, s, front, cand, sx);
                if (rest && !sat && g.l < k) part[sidx * k + g.l] = s.sk;
            }
        }
        const bool any = g.ballot(front) != 0;
        if (on && g.l == 0) seg_flag[sidx] = any ? 1 : 0;
    }
    flush_counters(sh, 256 / G, cand, io.ctr);
}

// Hubs: merge the partial results of all segments into the hub's sketch.
template <int G>
__global__ void __launch_bounds__(256) k_hop_hubs(const int32_t* __restrict__ hubs, int64_t n_hubs,
                                                     const int64_t* __restrict__ hub_seg,
                                                     const uint32_t* __restrict__ part, const uint32_t* __restrict__ PM,
                                                     const uint64_t* __restrict__ PH,
                                                     const uint8_t* __restrict__ seg_flag,
                                                     const uint32_t* __restrict__ hub_stamp, uint32_t sparse_hop,
                                                     int64_t slot0, HopIO io) {
    __shared__ HopShared sh;
    const Lock<G> g;
    uint32_t* sx = sh.x[threadIdx.x >> 5];
    const int k = io.k;
    const int64_t groups = ((int64_t)gridDim.x * blockDim.x) / G;
    ctr_init(g, sh);
    const int64_t first = ((int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) / G;
    for (int64_t i0 = first; i0 < n_hubs; i0 += groups) {
        const int64_t h = i0 + g.shift / G;
        bool on = h < n_hubs;
        const int32_t v = on ? hubs[h] : 0;
        const int64_t slot = slot0 + h;
        if (on && sparse_hop && hub_stamp[v] != sparse_hop) {
            if (g.l == 0) io.stg_grp[slot].info = 0;  // unchanged: empty slot
            on = false;
        }
        const int64_t deg = on ? io.rowp[v + 1] - io.rowp[v] : 0;
        const int64_t s0 = on ? hub_seg[h] : 0, s1 = on ? hub_seg[h + 1] : 0;
        bool any = false;
        for (int64_t q = s0 + g.l; q < s1; q += G) any |= seg_flag[q] != 0;
        any = g.ballot(any) != 0;
        if (any && g.l == 0) sh.ctr[threadIdx.x / G][kCMerging] += 1u;
        const uint64_t wv = on && io.hop > 1 ? io.W[v] : 0ULL;
        int dc = 0;
        if (warp_any(wv != 0)) {
            uint64_t acc = 0;
            if (wv != 0)
                for (int64_t q = s0 + g.l; q < s1; q += G) acc |= PH[q];
            acc = lock_or64(g, acc);
            if (wv != 0) {
                const uint64_t nw = lowest_k64(wv | acc, k);
                const uint64_t delta = nw & ~wv;
                if (delta != 0) finish_head(g, io, sh, v, deg, nw, delta, slot);
                else if (g.l == 0) io.stg_grp[slot].info = 0;  // unchanged: empty slot
                dc = __popcll(delta);
            }
        }
        const bool rest = on && wv == 0;
        if (warp_any(rest)) {
            const uint32_t old = rest && g.l < k ? io.S[(int64_t)v * k + g.l] : kNil;
            Sketch<G> s;
            s.sk = old;
            s.tau_base = kNil;
            s.retau(g, k);
            const bool sat = rest && io.hop > 1 && s.tau < (uint32_t)kUW;
            if (warp_any(sat))  // saturated hub: OR of the segments' partial masks
                merge_slices(
                    g, k, sat,
                    [&](int q, uint32_t(&w)[kSliceWords]) {
                        for (int64_t x = s0 + g.l; x < s1; x += G) {
                            const uint4* p = reinterpret_cast<const uint4*>(PM + x * 2 * kUWords + q * kSliceWords);
                            const uint4 a = p[0], b = p[1];
                            w[0] |= a.x;
                            w[1] |= a.y;
                            w[2] |= a.z;
                            w[3] |= a.w;
                            w[4] |= b.x;
                            w[5] |= b.y;
                            w[6] |= b.z;
                            w[7] |= b.w;
                        }
                    },
                    s.sk);
            if (warp_any(rest && !sat)) {
                s.retau(g, k);
                const int64_t end = rest && !sat ? s1 : s0;
                for (int64_t q = s0; warp_any(q < end); q += 4) {
                    uint32_t x[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) x[j] = q + j < end && g.l < k ? part[(q + j) * k + g.l] : kNil;
#pragma unroll
                    for (int j = 0; j < 4; ++j) merge_list(g, k, x[j], s, sx);
                }
            }
            const int got = finish_vertex(g, io, sh, rest, v, deg, old, s.sk, slot);
            if (rest) dc = got;
        }
        if (dc && g.l == 0) {
            atomicAdd(&io.ctr->merges, (unsigned long long)deg);
            atomicAdd(&io.ctr->delta_next, (unsigned long long)(deg * dc));
        }
    }
    flush_counters(sh, 256 / G, 0u, io.ctr);
}

// Sparse hops: the non-hub part of N(frontier).  Warp per frontier vertex;
// each neighbour is appended once (stamp = hop); hubs in N(frontier) get
// stamp = hop too, and the hub kernels skip the others.
__global__ void k_expand(const int32_t* __restrict__ fr, int64_t n_fr, const int64_t* __restrict__ rowp,
                         const int32_t* __restrict__ cols, uint32_t* __restrict__ stamp, uint32_t hop,
                         int seg, int32_t* __restrict__ act, Counters* ctr) {
    const int lane = lane_id();
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = (((int64_t)blockIdx.x * blockDim.x) + threadIdx.x) >> 5; w < n_fr; w += warps) {
        const int32_t u = fr[w];
        const int64_t beg = rowp[u], end = rowp[u + 1];
        for (int64_t cb = beg; cb < end; cb += 32) {
            int64_t e = cb + lane;
            bool fresh = false;
            int32_t v = 0;
            if (e < end) {
                v = cols[e];
                if (rowp[v + 1] - rowp[v] <= seg)
                    fresh = atomicExch(&stamp[v], hop) != hop;
                else
                    stamp[v] = hop;  // a hub with a frontier neighbour: its segments run this hop
            }
            long long at = warp_append(fresh, &ctr->active);
            if (at >= 0) act[at] = v;
        }
    }
}

// Vertices of a work list that gained entries this hop (the next frontier).
__global__ void k_collect_frontier(const int32_t* __restrict__ list, int64_t n, const uint8_t* __restrict__ Dcc,
                                   int32_t* __restrict__ fr, unsigned long long* __restrict__ n_fr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
        int64_t i = base + lane_id();
        int32_t v = i < n ? list[i] : 0;
        bool in = i < n && Dcc[v] > 0;
        long long at = warp_append(in, n_fr);
        if (at >= 0) fr[at] = v;
    }
}

// ------------------------------------------------------------------ ADS compaction

// v's group at distance 0: the entry v alone, a ball of one vertex (k >= 2).
__global__ void k_ads_hop0(int64_t n, const int64_t* __restrict__ gofs, const int64_t* __restrict__ eofs,
                           uint32_t* __restrict__ ginfo, double* __restrict__ gwt, int32_t* __restrict__ eid) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        ginfo[gofs[v]] = pack_info(0, 1, 1);
        gwt[gofs[v]] = 1.0;
        eid[eofs[v]] = (int32_t)v;
    }
}

// Staged groups -> vertex-major ADS, a thread per slot: the group's words and
// its HIP weight.  (The weight's FP64 division runs on all lanes here; on the
// one lane per vertex of a hop kernel it kept the FP64 pipe 25-40 % busy.)
__global__ void k_ads_groups(const StgGroup* __restrict__ stg_grp, const uint32_t* __restrict__ stg_kth,
                             int64_t n_slots, int k, uint64_t seed, const int32_t* __restrict__ ord_rid,
                             const int64_t* __restrict__ gofs, uint32_t* __restrict__ ginfo,
                             double* __restrict__ gwt) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_slots; i += stride) {
        const StgGroup gr = stg_grp[i];
        if (gr.info == 0) continue;
        const uint32_t kth = stg_kth[i];
        const int64_t at = gofs[gr.v] + gr.gidx;
        ginfo[at] = gr.info;
        gwt[at] = kth == kNil ? 1.0 : hip_weight(k, k, vertex_rank(seed, (int64_t)__ldg(&ord_rid[kth])));
    }
}

// Their entries; vid = vertex of each ordinal, a local id in a union.  A warp
// takes 32 slots and copies their entries end to end, 32 per pass (a lane finds
// its slot among the running counts): most slots hold far fewer than k entries
// and many none, so a thread per entry slot was bound by instructions
// (R-MAT 24, 416 M entries: 3.1 ms).
__global__ void __launch_bounds__(256) k_ads_entries(const StgGroup* __restrict__ stg_grp, int64_t n_slots, int k,
                                                     const uint32_t* __restrict__ stg_ent,
                                                     const int64_t* __restrict__ eofs,
                                                     const int32_t* __restrict__ vid,
                                                     const int32_t* __restrict__ vbase, int32_t* __restrict__ eid) {
    const int lane = lane_id();
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t b = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; b < n_slots; b += warps * 32) {
        StgGroup gr;
        gr.info = 0;
        if (b + lane < n_slots) gr = stg_grp[b + lane];
        const int cnt = (int)((gr.info >> 16) & 0xff);  // 0 for an empty slot
        const int incl = warp_incl_scan(cnt);
        const int total = __shfl_sync(kFull, incl, 31);
        const int64_t dst = cnt ? eofs[gr.v] + gr.eidx : 0;
        const int32_t base = cnt && vbase ? vbase[gr.v] : 0;
        for (int p = 0; p < total; p += 32) {
            const int j = p + lane;
            int w = 0;  // the slots whose entries all come before the j-th
#pragma unroll
            for (int s = 16; s > 0; s >>= 1)
                if (__shfl_sync(kFull, incl, w + s - 1) <= j) w += s;
            const int off = j - __shfl_sync(kFull, incl - cnt, w);
            const int64_t to = __shfl_sync(kFull, dst, w);
            const int32_t add = __shfl_sync(kFull, base, w);
            if (j < total) eid[to + off] = __ldg(&vid[stg_ent[(b + w) * k + off]]) + add;
        }
    }
}

// ------------------------------------------------------------------ graph work lists

__global__ void k_flag_degree(const int64_t* __restrict__ rowp, int64_t n, int seg, int32_t* __restrict__ low,
                              int32_t* __restrict__ hub, int32_t* __restrict__ nseg, int32_t* __restrict__ small) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const int64_t d = rowp[v + 1] - rowp[v];
        low[v] = (d > 0 && d <= seg) ? 1 : 0;
        hub[v] = d > seg ? 1 : 0;
        nseg[v] = d > seg ? (int32_t)((d + seg - 1) / seg) : 0;
        small[v] = (d > 0 && d <= kSmallDeg) ? 1 : 0;
    }
}

// Split the non-hub vertices by degree (ids ascending in both lists).
__global__ void k_scatter_by_degree(const int32_t* __restrict__ low, const int32_t* __restrict__ small,
                                    const int64_t* __restrict__ small_pos, const int64_t* __restrict__ low_pos,
                                    int64_t n, int32_t* __restrict__ small_list, int32_t* __restrict__ mid_list) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        if (small[v]) small_list[small_pos[v]] = (int32_t)v;
        else if (low[v]) mid_list[low_pos[v] - small_pos[v]] = (int32_t)v;
    }
}

__global__ void k_scatter_lists(const int32_t* __restrict__ low, const int32_t* __restrict__ hub,
                                const int64_t* __restrict__ low_pos, const int64_t* __restrict__ hub_pos,
                                const int64_t* __restrict__ seg_pos, int64_t n, int32_t* __restrict__ low_list,
                                int32_t* __restrict__ hub_list, int64_t* __restrict__ hub_seg) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        if (low[v]) low_list[low_pos[v]] = (int32_t)v;
        if (hub[v]) {
            hub_list[hub_pos[v]] = (int32_t)v;
            hub_seg[hub_pos[v]] = seg_pos[v];
        }
    }
}

__global__ void k_seg_owner(const int64_t* __restrict__ hub_seg, int64_t n_hubs, int32_t* __restrict__ seg_hub) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t h = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; h < n_hubs; h += stride)
        for (int64_t s = hub_seg[h]; s < hub_seg[h + 1]; ++s) seg_hub[s] = (int32_t)h;
}

static int grid_for(int64_t items, int per_block) {
    int64_t b = (items + per_block - 1) / per_block;
    if (b < 1) b = 1;
    if (b > 152 * 32) b = 152 * 32;
    return (int)b;
}

// Last element of an exclusive scan plus the last input = the total.
static int scan_total(const int64_t* pos, const int32_t* flag, int64_t n, cudaStream_t st, int64_t* total) {
    int64_t p = 0;
    int32_t f = 0;
    FL_CUDA(cudaMemcpyAsync(&p, pos + n - 1, 8, cudaMemcpyDeviceToHost, st));
    FL_CUDA(cudaMemcpyAsync(&f, flag + n - 1, 4, cudaMemcpyDeviceToHost, st));
    FL_CUDA(cudaStreamSynchronize(st));
    *total = p + f;
    return FL_OK;
}

// Longest row that is not cut, and edges per segment.  On a small graph the
// longest row ends every hop (61 k vertices: hub segments 81 us in hop 1 at
// 2048, 14 at 256); on larger ones shorter segments only add partial results to
// merge (all hop kernels, 2^20 vertices, k = 32: 3.4 ms at 2048, 3.5 at 512, 3.9
// at 256; 2^24, k = 16: 33.6 at 2048, 35.6 at 512).
static int seg_of(int64_t nnz) { return nnz <= (4 << 20) ? 256 : kMaxSeg; }

// Static work lists of a graph: non-hub non-isolated vertices, hubs and the
// segment table of the hubs.
int build_work_lists(fl_graph* g) {
    g->seg = seg_of(g->nnz);
    const int64_t n = g->n;
    cudaStream_t st = g->stream;
    DBuf low, hub, nseg, low_pos, hub_pos, seg_pos, small, small_pos;
    int rc = FL_OK;
    do {
        if ((rc = dalloc(low, (size_t)n * 4)) || (rc = dalloc(hub, (size_t)n * 4)) ||
            (rc = dalloc(nseg, (size_t)n * 4)) || (rc = dalloc(low_pos, (size_t)n * 8)) ||
            (rc = dalloc(hub_pos, (size_t)n * 8)) || (rc = dalloc(seg_pos, (size_t)n * 8)) ||
            (rc = dalloc(small, (size_t)n * 4)) || (rc = dalloc(small_pos, (size_t)n * 8)))
            break;
        FL_LAUNCH(kProfOther, k_flag_degree<<<grid_for(n, 256), 256, 0, st>>>(
                                  g->rowp.as<int64_t>(), n, g->seg, low.as<int32_t>(), hub.as<int32_t>(), nseg.as<int32_t>(),
                                  small.as<int32_t>()));
        if ((rc = scan_exclusive_i32_to_i64(low.as<int32_t>(), low_pos.as<int64_t>(), n, st, g->scratch, kProfOther)) ||
            (rc = scan_exclusive_i32_to_i64(hub.as<int32_t>(), hub_pos.as<int64_t>(), n, st, g->scratch, kProfOther)) ||
            (rc = scan_exclusive_i32_to_i64(nseg.as<int32_t>(), seg_pos.as<int64_t>(), n, st, g->scratch, kProfOther)) ||
            (rc = scan_exclusive_i32_to_i64(small.as<int32_t>(), small_pos.as<int64_t>(), n, st, g->scratch,
                                            kProfOther)))
            break;
        if ((rc = scan_total(low_pos.as<int64_t>(), low.as<int32_t>(), n, st, &g->n_low)) ||
            (rc = scan_total(hub_pos.as<int64_t>(), hub.as<int32_t>(), n, st, &g->n_hubs)) ||
            (rc = scan_total(seg_pos.as<int64_t>(), nseg.as<int32_t>(), n, st, &g->n_seg)) ||
            (rc = scan_total(small_pos.as<int64_t>(), small.as<int32_t>(), n, st, &g->n_small)))
            break;
        g->n_mid = g->n_low - g->n_small;
        if ((rc = dalloc(g->small_list, (size_t)std::max<int64_t>(g->n_small, 1) * 4)) ||
            (rc = dalloc(g->mid_list, (size_t)std::max<int64_t>(g->n_mid, 1) * 4)))
            break;
        FL_LAUNCH(kProfOther, k_scatter_by_degree<<<grid_for(n, 256), 256, 0, st>>>(
                                  low.as<int32_t>(), small.as<int32_t>(), small_pos.as<int64_t>(),
                                  low_pos.as<int64_t>(), n, g->small_list.as<int32_t>(), g->mid_list.as<int32_t>()));
        if ((rc = dalloc(g->low_list, (size_t)std::max<int64_t>(g->n_low, 1) * 4)) ||
            (rc = dalloc(g->hub_list, (size_t)std::max<int64_t>(g->n_hubs, 1) * 4)) ||
            (rc = dalloc(g->hub_seg, (size_t)(g->n_hubs + 1) * 8)) ||
            (rc = dalloc(g->seg_hub, (size_t)std::max<int64_t>(g->n_seg, 1) * 4)))
            break;
        FL_LAUNCH(kProfOther, k_scatter_lists<<<grid_for(n, 256), 256, 0, st>>>(
                                  low.as<int32_t>(), hub.as<int32_t>(), low_pos.as<int64_t>(), hub_pos.as<int64_t>(),
                                  seg_pos.as<int64_t>(), n, g->low_list.as<int32_t>(), g->hub_list.as<int32_t>(),
                                  g->hub_seg.as<int64_t>()));
        cudaError_t e = cudaMemcpyAsync(g->hub_seg.as<int64_t>() + g->n_hubs, &g->n_seg, 8, cudaMemcpyHostToDevice, st);
        if (e) { rc = status_of(e, "work lists", __FILE__, __LINE__); break; }
        if (g->n_hubs > 0)
            FL_LAUNCH(kProfOther, k_seg_owner<<<grid_for(g->n_hubs, 256), 256, 0, st>>>(
                                      g->hub_seg.as<int64_t>(), g->n_hubs, g->seg_hub.as<int32_t>()));
        e = cudaStreamSynchronize(st);
        if (e) { rc = status_of(e, "work lists", __FILE__, __LINE__); break; }
    } while (0);
    dfree_after(st, {&low, &hub, &nseg, &low_pos, &hub_pos, &seg_pos, &small, &small_pos});
    return rc == FL_OK ? build_items(g) : rc;
}

// Census of a hop's work list (profiling): CSR entries of the listed
// vertices, and of those whose sketch is saturated (read by the mask merge).
// Runs before the hop kernels change the sketches.
__global__ void k_hop_census(const int32_t* __restrict__ list, int64_t n_list, const int64_t* __restrict__ rowp,
                             const uint32_t* __restrict__ S, int k, int hop, const uint32_t* __restrict__ stamp, uint32_t sparse_hop, Counters* ctr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long sc = 0, mk = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_list; i += stride) {
        const int32_t v = list[i];
        if (sparse_hop && stamp[v] != sparse_hop) continue;  // a hub the hop skips
        const unsigned long long d = (unsigned long long)(rowp[v + 1] - rowp[v]);
        sc += d;
        if (hop > 1 && S[(int64_t)v * k + k - 1] < (uint32_t)kUW) mk += d;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sc += __shfl_xor_sync(kFull, sc, o);
        mk += __shfl_xor_sync(kFull, mk, o);
    }
    if (lane_id() == 0) {
        if (sc) atomicAdd(&ctr->scanned, sc);
        if (mk) atomicAdd(&ctr->mask_scanned, mk);
    }
}

// ------------------------------------------------------------------ ordinals

// Few ranks: each one's ordinal is the number of ranks below its own.  A block
// counts for 64 ids, two per lane, over its share of the ranks (blockIdx.y of
// gridDim.y), computed into shared memory a tile at a time.  (Ranks are a
// bijection of the ids.)
__global__ void __launch_bounds__(256) k_count_ranks(int m, uint64_t seed, uint32_t* __restrict__ of_rid,
                                                     Counters* ctr) {
    constexpr int kTile = 512;
    __shared__ uint64_t key[kTile];
    __shared__ int below[64];
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const int i0 = blockIdx.x * 64 + lane, i1 = i0 + 32;
    const uint64_t r0 = vertex_rank(seed, i0), r1 = vertex_rank(seed, i1);
    const int t0 = (int)((int64_t)m * blockIdx.y / gridDim.y), t1 = (int)((int64_t)m * (blockIdx.y + 1) / gridDim.y);
    int c0 = 0, c1 = 0;
    if (threadIdx.x < 64) below[threadIdx.x] = 0;
    for (int t = t0; t < t1; t += kTile) {
        const int cnt = min(kTile, t1 - t);
        __syncthreads();
        for (int j = threadIdx.x; j < cnt; j += 256) key[j] = vertex_rank(seed, t + j);
        __syncthreads();
#pragma unroll 4
        for (int j = warp; j < cnt; j += 8) {
            const uint64_t x = key[j];
            c0 += x < r0;
            c1 += x < r1;
        }
    }
    atomicAdd(&below[lane], c0);
    atomicAdd(&below[lane + 32], c1);
    __syncthreads();
    const int i = blockIdx.x * 64 + threadIdx.x;
    if (threadIdx.x < 64 && i < m) {
        atomicAdd(&of_rid[i], (uint32_t)below[threadIdx.x]);
        if (blockIdx.y == 0 && vertex_rank(seed, i) == kEmpty) atomicOr(&ctr->error, 1ULL);
    }
}

__global__ void k_place_ranks(const uint32_t* __restrict__ of_rid, int m, int32_t* __restrict__ ord_rid) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m) ord_rid[of_rid[i]] = i;
}

__global__ void k_rank_pairs(int64_t m, uint64_t seed, uint64_t* __restrict__ key, uint32_t* __restrict__ val,
                             Counters* ctr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) {
        const uint64_t r = vertex_rank(seed, i);
        key[i] = r;
        val[i] = (uint32_t)i;
        if (r == kEmpty) atomicOr(&ctr->error, 1ULL);
    }
}

// Ranks sorted by their bits from `shift` up: every id to its place, the few
// runs that these bits leave equal in the order of the whole rank.
__global__ void k_rank_place(const uint64_t* __restrict__ key, const uint32_t* __restrict__ val, int64_t m, int shift,
                             int32_t* __restrict__ ord_rid) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) {
        const uint64_t r = key[i];
        int64_t at = i;
        for (int64_t j = i - 1; j >= 0 && (key[j] >> shift) == (r >> shift); --j) at -= key[j] > r;
        for (int64_t j = i + 1; j < m && (key[j] >> shift) == (r >> shift); ++j) at += key[j] < r;
        ord_rid[at] = (int32_t)val[i];
    }
}

// vid[o] = inv[rid], the vertex of ordinal o, and ord[vid[o]] = o (inv NULL: vid = rid)
__global__ void k_ord_scatter(const int32_t* __restrict__ ord_rid, int64_t m, const int32_t* __restrict__ inv,
                              int32_t* __restrict__ vid, uint32_t* __restrict__ ord) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < m; o += stride) {
        const int32_t v = inv ? inv[ord_rid[o]] : ord_rid[o];
        vid[o] = v;
        ord[v] = (uint32_t)o;
    }
}

__global__ void k_ord_gather(const uint32_t* __restrict__ of_rid, const int32_t* __restrict__ rid, int64_t n,
                             uint32_t* __restrict__ ord) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) ord[v] = of_rid[rid[v]];
}

// g->ord_rid, g->ord_vid and g->ord.  The rank ids of a union are its parts' local ids
// (below the largest part's size).  A reserved rank sets bit 0 of ctr->error,
// which the caller clears before.  tmp: scratch, 28 bytes per rank id.
int build_ordinals(fl_graph* g, DBuf& tmp) {
    const int64_t n = g->n, m = g->max_part > 0 ? g->max_part : n;
    cudaStream_t st = g->stream;
    Counters* ctr = g->ctr.as<Counters>();
    FL_TRY(dalloc(g->ord, (size_t)n * 4));
    FL_TRY(dalloc(g->ord_rid, (size_t)m * 4));
    FL_TRY(dalloc(g->ord_vid, (size_t)m * 4));
    FL_TRY(dalloc(tmp, (size_t)m * 28));
    int32_t* ord_rid = g->ord_rid.as<int32_t>();
    uint32_t* of_rid = reinterpret_cast<uint32_t*>(tmp.as<char>() + (size_t)m * 24);
    if (m <= kCountMax) {
        FL_CUDA(cudaMemsetAsync(of_rid, 0, (size_t)m * 4, st));
        FL_LAUNCH(kProfSketchOther, k_count_ranks<<<dim3((unsigned)((m + 63) / 64), count_shares(m)), 256, 0, st>>>(
                                        (int)m, g->seed, of_rid, ctr));
        FL_LAUNCH(kProfSketchOther, k_place_ranks<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(of_rid, (int)m,
                                                                                              ord_rid));
    } else {
        SortPairs<uint64_t> p;
        p.key[0] = tmp.as<uint64_t>();
        p.key[1] = p.key[0] + m;
        p.val[0] = reinterpret_cast<uint32_t*>(p.key[1] + m);
        p.val[1] = p.val[0] + m;
        int lg = 0, shift[kSortDigits];
        while ((1LL << lg) < m) ++lg;
        // equal leading lg + 16 bits: about m / 2^17 pairs
        const int nd = digit_windows(~0ULL, lg + 16, shift);
        FL_LAUNCH(kProfSketchOther, k_rank_pairs<<<grid_for(m, 256), 256, 0, st>>>(m, g->seed, p.key[0], p.val[0],
                                                                                 ctr));
        FL_TRY(sort_pairs(p, m, shift, nd, st, g->scratch, kProfSketchOther, &ctr->error));
        FL_LAUNCH(kProfSketchOther, k_rank_place<<<grid_for(m, 256), 256, 0, st>>>(p.key[p.cur], p.val[p.cur], m,
                                                                                 shift[0], ord_rid));
    }
    if (g->max_part > 0) {
        FL_LAUNCH(kProfSketchOther, k_ord_scatter<<<grid_for(m, 256), 256, 0, st>>>(ord_rid, m, nullptr,
                                                                                  g->ord_vid.as<int32_t>(), of_rid));
        FL_LAUNCH(kProfSketchOther, k_ord_gather<<<grid_for(n, 256), 256, 0, st>>>(of_rid, g->rid.as<int32_t>(), n,
                                                                                 g->ord.as<uint32_t>()));
    } else {
        FL_LAUNCH(kProfSketchOther, k_ord_scatter<<<grid_for(m, 256), 256, 0, st>>>(
                                        ord_rid, m, g->relabelled ? g->inv.as<int32_t>() : nullptr,
                                        g->ord_vid.as<int32_t>(), g->ord.as<uint32_t>()));
    }
    FL_CUDA(cudaGetLastError());
    return FL_OK;
}

// Start of a hop, in one pass: the previous hop's frontier as a bitmap (bit v =
// (Dp[v] > 0); Dp NULL at hop 1, where every vertex counts), this hop's
// outputs at "no new entries" for every vertex that will not change, and the
// counters at zero.
__global__ void k_hop_begin(const uint8_t* __restrict__ Dp, int64_t n, uint32_t* __restrict__ bm,
                            uint8_t* __restrict__ Dc, uint32_t* __restrict__ F, uint64_t* __restrict__ H,
                            Counters* ctr) {
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    if (tid < (int64_t)(sizeof(Counters) / 8)) reinterpret_cast<unsigned long long*>(ctr)[tid] = 0;
    for (int64_t base = tid & ~(int64_t)31; base < n; base += stride) {
        const int64_t v = base + lane_id();
        if (Dp) {
            const unsigned w = __ballot_sync(kFull, v < n && Dp[v] > 0);
            if (lane_id() == 0) bm[base >> 5] = w;
        }
        if (v < n) {
            Dc[v] = 0;
            F[v] = kNil;
            H[v] = 0;
        }
    }
}

// Ends of the ADS offsets; the totals also to the counters (aux0, aux3).
__global__ void k_ads_totals(const int32_t* __restrict__ vg, const int32_t* __restrict__ ve, int64_t n,
                             int64_t* __restrict__ gofs, int64_t* __restrict__ eofs, Counters* ctr) {
    gofs[n] = gofs[n - 1] + vg[n - 1];
    eofs[n] = eofs[n - 1] + ve[n - 1];
    ctr->aux0 = (unsigned long long)gofs[n];
    ctr->aux3 = (unsigned long long)eofs[n];
}

// ------------------------------------------------------------------ driver

template <int G>
static int launch_hop(fl_graph* g, int hop, const int32_t* list, int64_t n_list, int pin, int pout,
                      int64_t slot_base, bool sparse) {
    cudaStream_t st = g->stream;
    const int k = g->k;
    const int per_block = 256 / G;
    const uint32_t sparse_hop = sparse ? (uint32_t)hop : 0u;
    HopIO io;
    io.rowp = g->rowp.as<int64_t>();
    io.cols = g->cols.as<int32_t>();
    io.k = k;
    io.hop = hop;
    io.seg = g->seg;
    io.ord = g->ord.as<uint32_t>();
    io.S = g->S.as<uint32_t>();
    io.Scnt = g->Scnt.as<uint8_t>();
    io.Dp = g->D[pin].as<uint32_t>();
    io.Dc = g->D[pout].as<uint32_t>();
    io.Dcc = g->Dcnt[pout].as<uint8_t>();
    io.Fp = g->F[pin].as<uint32_t>();
    io.Fc = g->F[pout].as<uint32_t>();
    io.Hp = g->H[pin].as<uint64_t>();
    io.Hc = g->H[pout].as<uint64_t>();
    io.W = g->W.as<uint64_t>();
    io.bm = g->fbm.as<uint32_t>();
    io.DMp = g->DM[pin].as<uint64_t>();
    io.DMc = g->DM[pout].as<uint64_t>();
    io.n = g->n;
    io.vg = g->vg.as<int32_t>();
    io.ve = g->ve.as<int32_t>();
    io.stg_ent = g->stg_ent.as<uint32_t>() + slot_base * k;
    io.stg_kth = g->stg_kth.as<uint32_t>() + slot_base;
    io.stg_grp = g->stg_grp.as<StgGroup>() + slot_base;
    io.ctr = g->ctr.as<Counters>();
    if (n_list > 0)
        FL_LAUNCH(kProfSketchMerge, k_hop_vertices<G><<<grid_for(n_list, per_block), 256, 0, st>>>(list, n_list, io));
    if (g->n_hubs > 0) {
        FL_LAUNCH(kProfSketchMerge, k_hop_hub_segments<G><<<grid_for(g->n_seg, per_block), 256, 0, st>>>(
                                        g->hub_list.as<int32_t>(), g->hub_seg.as<int64_t>(), g->seg_hub.as<int32_t>(),
                                        g->n_seg, g->part.as<uint32_t>(), g->PM.as<uint32_t>(), g->PH.as<uint64_t>(),
                                        g->seg_flag.as<uint8_t>(), g->stamp.as<uint32_t>(), sparse_hop, io));
        FL_LAUNCH(kProfSketchMerge, k_hop_hubs<G><<<grid_for(g->n_hubs, per_block), 256, 0, st>>>(
                                        g->hub_list.as<int32_t>(), g->n_hubs, g->hub_seg.as<int64_t>(),
                                        g->part.as<uint32_t>(), g->PM.as<uint32_t>(), g->PH.as<uint64_t>(),
                                        g->seg_flag.as<uint8_t>(), g->stamp.as<uint32_t>(), sparse_hop, n_list, io));
    }
    FL_CUDA(cudaGetLastError());
    return FL_OK;
}

int build_sketches(fl_graph* g, int k, uint64_t seed) {
    const int64_t n = g->n;
    cudaStream_t st = g->stream;
    g->built = 0;
    ++g->generation;
    g->k = k;
    g->seed = seed;
    if (g->wts.p) {  // a weighted graph: levels in Dijkstra order (k_wsketch.cu)
        g->hop_scanned.clear();
        g->hop_mask.clear();
        g->hop_changed.clear();
        g->hop_ms.clear();
        for (auto* vec : {&g->hop_E, &g->hop_A, &g->hop_R, &g->hop_SD, &g->hop_new}) vec->clear();
        FL_TRY(build_sketches_weighted(g, k, seed));
        g->built = 1;
        return FL_OK;
    }
    if (!g->lists_ready) {
        FL_TRY(build_work_lists(g));
        g->lists_ready = 1;
    }
    const size_t nk = (size_t)n * k;
    FL_TRY(dalloc(g->S, nk * 4));
    FL_TRY(dalloc(g->Scnt, (size_t)n));
    for (int p = 0; p < 2; ++p) {
        FL_TRY(dalloc(g->D[p], nk * 4));
        FL_TRY(dalloc(g->Dcnt[p], (size_t)n));
        FL_TRY(dalloc(g->frontier[p], (size_t)n * 4));
    }
    FL_TRY(dalloc(g->stamp, (size_t)n * 4));
    FL_TRY(dalloc(g->vg, (size_t)n * 4));
    FL_TRY(dalloc(g->ve, (size_t)n * 4));
    FL_TRY(dalloc(g->part, (size_t)std::max<int64_t>(g->n_seg, 1) * k * 4));
    FL_TRY(dalloc(g->DM[0], (size_t)n * kUWords * 8));
    FL_TRY(dalloc(g->DM[1], (size_t)n * kUWords * 8));
    FL_TRY(dalloc(g->PM, (size_t)std::max<int64_t>(g->n_seg, 1) * kUWords * 8));
    FL_TRY(dalloc(g->PH, (size_t)std::max<int64_t>(g->n_seg, 1) * 8));
    FL_TRY(dalloc(g->seg_flag, (size_t)std::max<int64_t>(g->n_seg, 1)));
    for (int p = 0; p < 2; ++p) {
        FL_TRY(dalloc(g->F[p], (size_t)n * 4));
        FL_TRY(dalloc(g->H[p], (size_t)n * 8));
    }
    FL_TRY(dalloc(g->W, (size_t)n * 8));
    FL_TRY(dalloc(g->fbm, ((size_t)(n + 31) / 32 + 1) * 4));
    // staging: one slot per work item of each hop
    const int64_t per_dense = g->n_low + g->n_hubs;
    size_t slot_cap = (size_t)per_dense * 8 + 1024;
    if (g->stg_grp_cap < slot_cap || g->stg_k != k) {
        slot_cap = std::max(slot_cap, g->stg_grp_cap);
        FL_TRY(dalloc(g->stg_grp, slot_cap * sizeof(StgGroup)));
        FL_TRY(dalloc(g->stg_kth, slot_cap * 4));
        FL_TRY(dalloc(g->stg_ent, slot_cap * k * 4));
        g->stg_grp_cap = slot_cap;
        g->stg_k = k;
    }
    DBuf act;  // active list of sparse hops
    FL_TRY(dalloc(act, (size_t)n * 4));

    FL_CUDA(cudaMemsetAsync(g->S.p, 0xff, nk * 4, st));
    FL_CUDA(cudaMemsetAsync(g->W.p, 0, (size_t)n * 8, st));
    FL_CUDA(cudaMemsetAsync(g->stamp.p, 0, (size_t)n * 4, st));
    FL_CUDA(cudaMemsetAsync(g->ctr.p, 0, sizeof(Counters), st));
    {
        int rc0 = build_ordinals(g, g->DM[0]);  // the delta masks are written later
        if (rc0 != FL_OK) {
            dfree_after(st, {&act});
            return rc0;
        }
    }
    FL_LAUNCH(kProfSketchOther, k_rank_init<<<grid_for(n, 256), 256, 0, st>>>(
                                    n, k, g->ord.as<uint32_t>(), g->S.as<uint32_t>(), g->Scnt.as<uint8_t>(),
                                    g->vg.as<int32_t>(), g->ve.as<int32_t>()));
    FL_CUDA(cudaGetLastError());
    FL_TRY(read_counters(g));
    if (g->h_ctr->error) {
        dfree_after(st, {&act});
        if (g->h_ctr->error & kSortError) FL_FAIL(FL_ETIMEOUT, "ordinals: a sort's wait ran out");
        FL_FAIL(FL_EINVAL, "a vertex rank equals the reserved empty-slot value; choose another seed");
    }
    g->hop_scanned.clear();
    g->hop_mask.clear();
    g->hop_changed.clear();
    g->hop_ms.clear();
    for (auto* vec : {&g->hop_E, &g->hop_A, &g->hop_R, &g->hop_SD, &g->hop_new}) vec->clear();
    const bool time_hops = g->prof.on != 0;
    const bool census = g->prof.on >= 2;  // per-hop scanned / mask counts (extra kernels)
    if (time_hops && !g->hop_ev[0]) {
        FL_CUDA(cudaEventCreate(&g->hop_ev[0]));
        FL_CUDA(cudaEventCreate(&g->hop_ev[1]));
    }
    int64_t used_slots = 0;
    int64_t n_front = n;  // hop 0: every vertex gained its own rank
    bool fr_list_ready = false;
    // hop 1: every vertex gained its own rank at hop 0, so each CSR entry is
    // an edge-merge carrying one delta rank
    int64_t total_merges = 0, next_merges = g->nnz, next_delta = g->nnz;
    int hop = 1;
    int rc = FL_OK;
    for (;; ++hop) {
        if (hop > kMaxHops) { rc = FL_ETIMEOUT; set_error(rc, "more than 65535 hops"); break; }
        total_merges += next_merges;
        const int64_t hop_merges = next_merges, hop_delta = next_delta;
        const int pin = (hop - 1) & 1, pout = hop & 1;
        const int32_t* list;
        int64_t n_list;
        // dense hops run every non-isolated vertex; sparse hops expand the frontier
        const bool dense = !fr_list_ready;
        FL_LAUNCH(kProfSketchOther, k_hop_begin<<<grid_for(n, 256), 256, 0, st>>>(
                                        hop > 1 ? g->Dcnt[pin].as<uint8_t>() : nullptr, n, g->fbm.as<uint32_t>(),
                                        g->Dcnt[pout].as<uint8_t>(), g->F[pout].as<uint32_t>(),
                                        g->H[pout].as<uint64_t>(), g->ctr.as<Counters>()));
        if (dense) {
            list = g->low_list.as<int32_t>();
            n_list = g->n_low;
        } else {
            FL_LAUNCH(kProfSketchExpand, k_expand<<<grid_for(n_front, 8), 256, 0, st>>>(
                                             g->frontier[pin].as<int32_t>(), n_front, g->rowp.as<int64_t>(),
                                             g->cols.as<int32_t>(), g->stamp.as<uint32_t>(), (uint32_t)hop, g->seg,
                                             act.as<int32_t>(), g->ctr.as<Counters>()));
            FL_CUDA(cudaGetLastError());
            FL_TRY(read_counters(g));
            list = act.as<int32_t>();
            n_list = (int64_t)g->h_ctr->active;
        }
        const int64_t slots = n_list + g->n_hubs;
        if ((size_t)(used_slots + slots) > g->stg_grp_cap) {
            size_t cap = std::max<size_t>((size_t)(used_slots + slots), g->stg_grp_cap * 3 / 2);
            FL_TRY(dgrow(g->stg_grp, cap * sizeof(StgGroup), (size_t)used_slots * sizeof(StgGroup), st));
            FL_TRY(dgrow(g->stg_kth, cap * 4, (size_t)used_slots * 4, st));
            FL_TRY(dgrow(g->stg_ent, cap * k * 4, (size_t)used_slots * k * 4, st));
            g->stg_grp_cap = cap;
        }
        if (census) {
            if (n_list > 0)
                FL_LAUNCH(kProfSketchOther, k_hop_census<<<grid_for(n_list, 256), 256, 0, st>>>(
                                                list, n_list, g->rowp.as<int64_t>(), g->S.as<uint32_t>(), k, hop,
                                                nullptr, 0u, g->ctr.as<Counters>()));
            if (g->n_hubs > 0)
                FL_LAUNCH(kProfSketchOther, k_hop_census<<<grid_for(g->n_hubs, 256), 256, 0, st>>>(
                                                g->hub_list.as<int32_t>(), g->n_hubs, g->rowp.as<int64_t>(),
                                                g->S.as<uint32_t>(), k, hop, g->stamp.as<uint32_t>(), dense ? 0u : (uint32_t)hop,
                                                g->ctr.as<Counters>()));
        }
        if (time_hops) FL_CUDA(cudaEventRecord(g->hop_ev[0], st));
        if (k <= 16 && g->sched.hop_group != 32)
            FL_TRY(launch_hop<16>(g, hop, list, n_list, pin, pout, used_slots, !dense));
        else
            FL_TRY(launch_hop<32>(g, hop, list, n_list, pin, pout, used_slots, !dense));
        if (time_hops) FL_CUDA(cudaEventRecord(g->hop_ev[1], st));
        used_slots += slots;
        FL_TRY(read_counters(g));
        {
            float hop_ms = 0.f;
            if (time_hops) FL_CUDA(cudaEventElapsedTime(&hop_ms, g->hop_ev[0], g->hop_ev[1]));
            g->hop_scanned.push_back(census ? (int64_t)g->h_ctr->scanned : 0);
            g->hop_mask.push_back(census ? (int64_t)g->h_ctr->mask_scanned : 0);
            g->hop_changed.push_back((int64_t)g->h_ctr->frontier);
            g->hop_ms.push_back(hop_ms);
            g->hop_E.push_back(hop_merges);
            g->hop_A.push_back((int64_t)g->h_ctr->merging);
            g->hop_R.push_back((int64_t)g->h_ctr->cand_reads);
            g->hop_SD.push_back(hop_delta);
            g->hop_new.push_back((int64_t)g->h_ctr->new_entries);
        }
        n_front = (int64_t)g->h_ctr->frontier;
        next_merges = (int64_t)g->h_ctr->merges;
        next_delta = (int64_t)g->h_ctr->delta_next;
        // algorithmic bytes of this hop's merge: row offsets of each merging
        // vertex (8 B), frontier columns (4 B per edge-merge), delta words read
        // (8 B each, the size of a mask word; the list merge's are ordinals of
        // 4 B), own sketch read + write (ordinals: 8k B per merging vertex); the
        // ADS entries (12 B each) are added after the last hop
        {
            const double A = (double)g->h_ctr->merging, R = (double)g->h_ctr->cand_reads;
            g->prof.bytes[kProfSketchMerge] += 8.0 * A + 4.0 * (double)hop_merges + 8.0 * R + 8.0 * k * A;
        }
        if (n_front == 0) break;
        // a small frontier makes the next hop sparse: collect its list
        fr_list_ready = false;
        if (n_front * g->sched.sparse_div < g->n_low + g->n_hubs) {
            // (aux0 is zero since the hop began)
            if (n_list > 0)
                FL_LAUNCH(kProfSketchExpand, k_collect_frontier<<<grid_for(n_list, 256), 256, 0, st>>>(
                                                 list, n_list, g->Dcnt[pout].as<uint8_t>(),
                                                 g->frontier[pout].as<int32_t>(), &g->ctr.as<Counters>()->aux0));
            if (g->n_hubs > 0)
                FL_LAUNCH(kProfSketchExpand, k_collect_frontier<<<grid_for(g->n_hubs, 256), 256, 0, st>>>(
                                                 g->hub_list.as<int32_t>(), g->n_hubs, g->Dcnt[pout].as<uint8_t>(),
                                                 g->frontier[pout].as<int32_t>(), &g->ctr.as<Counters>()->aux0));
            FL_CUDA(cudaGetLastError());
            FL_TRY(read_counters(g));
            fr_list_ready = true;
        }
    }
    dfree_after(st, {&act});
    if (rc != FL_OK) return rc;
    g->hops = hop - 1;
    g->edge_merges = total_merges;

    // vertex-major ADS
    FL_TRY(dalloc(g->gofs, (size_t)(n + 1) * 8));
    FL_TRY(dalloc(g->eofs, (size_t)(n + 1) * 8));
    FL_TRY(scan_exclusive_i32_to_i64(g->vg.as<int32_t>(), g->gofs.as<int64_t>(), n, st, g->scratch));
    FL_TRY(scan_exclusive_i32_to_i64(g->ve.as<int32_t>(), g->eofs.as<int64_t>(), n, st, g->scratch));
    FL_LAUNCH(kProfSketchOther, k_ads_totals<<<1, 1, 0, st>>>(g->vg.as<int32_t>(), g->ve.as<int32_t>(), n,
                                                              g->gofs.as<int64_t>(), g->eofs.as<int64_t>(),
                                                              g->ctr.as<Counters>()));
    FL_TRY(read_counters(g));
    g->n_groups = (int64_t)g->h_ctr->aux0;
    g->n_entries = (int64_t)g->h_ctr->aux3;
    g->prof.bytes[kProfSketchMerge] += 12.0 * (double)(g->n_entries - n);
    FL_TRY(dalloc(g->ginfo, (size_t)std::max<int64_t>(g->n_groups, 1) * 4));
    FL_TRY(dalloc(g->gwt, (size_t)std::max<int64_t>(g->n_groups, 1) * 8));
    FL_TRY(dalloc(g->eid, (size_t)std::max<int64_t>(g->n_entries, 1) * 4));
    FL_LAUNCH(kProfSketchOther, k_ads_hop0<<<grid_for(n, 256), 256, 0, st>>>(
                                    n, g->gofs.as<int64_t>(), g->eofs.as<int64_t>(), g->ginfo.as<uint32_t>(),
                                    g->gwt.as<double>(), g->eid.as<int32_t>()));
    if (used_slots > 0) {
        FL_LAUNCH(kProfSketchOther, k_ads_groups<<<grid_for(used_slots, 256), 256, 0, st>>>(
                                        g->stg_grp.as<StgGroup>(), g->stg_kth.as<uint32_t>(), used_slots, k, seed,
                                        g->ord_rid.as<int32_t>(), g->gofs.as<int64_t>(), g->ginfo.as<uint32_t>(),
                                        g->gwt.as<double>()));
        FL_LAUNCH(kProfSketchOther, k_ads_entries<<<grid_for(used_slots, 256), 256, 0, st>>>(
                                        g->stg_grp.as<StgGroup>(), used_slots, k, g->stg_ent.as<uint32_t>(),
                                        g->eofs.as<int64_t>(), g->ord_vid.as<int32_t>(),
                                        g->max_part > 0 ? g->vbase.as<int32_t>() : nullptr, g->eid.as<int32_t>()));
    }
    FL_CUDA(cudaGetLastError());
    FL_TRY(compute_ecc_bound(g));  // synchronises
    g->built = 1;
    return FL_OK;
}

// ------------------------------------------------------------------ eccentricity bound
// The minimum ordinal of a component (S[v][0] at the fixed point) names a root
// for every vertex of it; a multi-source BFS from the roots gives d(v, root)
// and ecc(root), and ecc(v) <= d(v, root) + ecc(root).

__global__ void k_roots(const uint32_t* __restrict__ S, int k, const uint32_t* __restrict__ ord, int64_t n,
                        int32_t* __restrict__ roots, Counters* ctr) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
        int64_t v = base + lane_id();
        bool is_root = false;
        if (v < n) is_root = S[v * k] == ord[v];
        long long at = warp_append(is_root, &ctr->aux0);
        if (at >= 0) roots[at] = (int32_t)v;
    }
}

__global__ void k_ecc_max(const int32_t* __restrict__ label, const int32_t* __restrict__ dist, int64_t n,
                          int32_t* __restrict__ eccr) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride)
        if (dist[v] > 0 && eccr[label[v]] < dist[v]) atomicMax(&eccr[label[v]], dist[v]);
}

__global__ void k_ecc_ub(const int32_t* __restrict__ label, const int32_t* __restrict__ dist,
                         const int32_t* __restrict__ eccr, int64_t n, int32_t* __restrict__ ub) {
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride)
        ub[v] = dist[v] + eccr[label[v]];
}

int compute_ecc_bound(fl_graph* g) {
    const int64_t n = g->n;
    cudaStream_t st = g->stream;
    DBuf roots, label, dist, eccr, X, stampb, fr[2], frval;
    int rc = FL_OK;
    do {
        if ((rc = dalloc(roots, (size_t)n * 4))) break;
        if ((rc = dalloc(label, (size_t)n * 4))) break;
        if ((rc = dalloc(dist, (size_t)n * 4))) break;
        if ((rc = dalloc(eccr, (size_t)n * 4))) break;
        if ((rc = dalloc(g->ecc_ub, (size_t)n * 4))) break;
        cudaError_t e = cudaMemsetAsync(g->ctr.p, 0, sizeof(Counters), st);
        if (e == cudaSuccess) e = cudaMemsetAsync(eccr.p, 0, (size_t)n * 4, st);
        if (e != cudaSuccess) { rc = status_of(e, "ecc init", __FILE__, __LINE__); break; }
        FL_LAUNCH(kProfSketchOther, k_roots<<<grid_for(n, 256), 256, 0, st>>>(
                                        g->S.as<uint32_t>(), g->k, g->ord.as<uint32_t>(), n, roots.as<int32_t>(),
                                        g->ctr.as<Counters>()));
        if ((rc = read_counters(g))) break;
        int64_t n_roots = (int64_t)g->h_ctr->aux0;
        if ((rc = msbfs(g, roots.as<int32_t>(), n_roots, label.as<int32_t>(), dist.as<int32_t>(), X, stampb,
                        fr, frval, kProfSketchOther)))
            break;
        FL_LAUNCH(kProfSketchOther, k_ecc_max<<<grid_for(n, 256), 256, 0, st>>>(label.as<int32_t>(),
                                                                                dist.as<int32_t>(), n,
                                                                                eccr.as<int32_t>()));
        FL_LAUNCH(kProfSketchOther, k_ecc_ub<<<grid_for(n, 256), 256, 0, st>>>(
                                        label.as<int32_t>(), dist.as<int32_t>(), eccr.as<int32_t>(), n,
                                        g->ecc_ub.as<int32_t>()));
        e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) { rc = status_of(e, "ecc bound", __FILE__, __LINE__); break; }
    } while (0);
    dfree_after(st, {&roots, &label, &dist, &eccr, &X, &stampb, &fr[0], &fr[1], &frval});
    return rc;
}

}  // namespace fl

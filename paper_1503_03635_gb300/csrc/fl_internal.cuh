// fl_internal.cuh -- shared internals of libflgpu (handles, errors, warp primitives).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <initializer_list>
#include <vector>

#include "../../include/fl.h"

namespace fl {

// ----------------------------------------------------------------- errors

void set_error(int status, const std::string& msg);
int status_of(cudaError_t e, const char* what, const char* file, int line);

#define FL_CUDA(call)                                                              \
    do {                                                                           \
        cudaError_t e__ = (call);                                                  \
        if (e__ != cudaSuccess) return ::fl::status_of(e__, #call, __FILE__, __LINE__); \
    } while (0)

#define FL_TRY(expr)                 \
    do {                             \
        int s__ = (expr);            \
        if (s__ != FL_OK) return s__; \
    } while (0)

#define FL_FAIL(code, msg)               \
    do {                                 \
        ::fl::set_error((code), (msg));  \
        return (code);                   \
    } while (0)

// ----------------------------------------------------------------- device buffers

struct DBuf {
    void* p = nullptr;
    size_t bytes = 0;
    template <class T>
    T* as() const { return static_cast<T*>(p); }
};

int dalloc(DBuf& b, size_t bytes);            // free + allocate (no copy)
int dgrow(DBuf& b, size_t bytes, size_t keep, cudaStream_t st);  // grow keeping `keep` bytes
void dfree(DBuf& b);
void dfree_idle(DBuf& b);                     // to the idle-block cache (no pending work uses b)
// A call's temporaries: to the idle-block cache once `st` has finished with them.
void dfree_after(cudaStream_t st, std::initializer_list<DBuf*> bufs);

// ----------------------------------------------------------------- constants

constexpr uint64_t kGamma = 0x9e3779b97f4a7c15ULL;   // SplitMix64 increment
constexpr uint64_t kMul1 = 0xbf58476d1ce4e5b9ULL;
constexpr uint64_t kMul2 = 0x94d049bb133111ebULL;
constexpr uint64_t kEmpty = ~0ULL;                   // empty sketch slot

// Vertex ids.  Kernels work on internal ids.  A graph may relabel its
// vertices (by descending degree, so that the values of high-degree vertices,
// read by most edges, share cache sectors) or be a disjoint union of parts
// (batches).  The rank id of a vertex is the id that ranks, priorities and
// reported facility labels use: the original id of a relabelled graph, the
// part-local id in a union, else the id itself.
struct IdMap {
    const int32_t* rid = nullptr;    // rank id of each internal vertex (NULL: the id itself)
    const int32_t* inv = nullptr;    // relabelled graph: internal id of each original id
    const int32_t* vbase = nullptr;  // union: first internal id of each vertex's part
};

__device__ __forceinline__ int64_t rank_id(const IdMap& m, int64_t v) {
    return m.rid ? (int64_t)__ldg(&m.rid[v]) : v;
}

// SplitMix64 finaliser (each step is a bijection on 64 bits).
__host__ __device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z = (z ^ (z >> 30)) * kMul1;
    z = (z ^ (z >> 27)) * kMul2;
    return z ^ (z >> 31);
}
// r(v): SplitMix64 output v+1 from state `seed`.
__host__ __device__ __forceinline__ uint64_t vertex_rank(uint64_t seed, int64_t v) {
    return mix64(seed + (uint64_t)(v + 1) * kGamma);
}
// pi(f): SplitMix64 output f+1 from the state given by the first output for `seed`.
__host__ __device__ __forceinline__ uint64_t facility_priority(uint64_t seed, int64_t f) {
    uint64_t stream = mix64(seed + kGamma);
    return mix64(stream + (uint64_t)(f + 1) * kGamma);
}

// ----------------------------------------------------------------- warp primitives
// A "lane list" holds up to 32 uint64 values, one per lane, ascending by lane,
// padded with kEmpty.

constexpr unsigned kFull = 0xffffffffu;

// Vertices with more than fl_graph::seg neighbours are hubs; their edge lists
// are processed in segments of that many edges, one group of lanes per segment
// (seg_of in k_sketch.cu).
constexpr int kMaxSeg = 2048;
// Non-hub vertices with at most kSmallDeg neighbours are pulled by one thread each.
constexpr int kSmallDeg = 8;
// Graphs of at most kResidentEdges CSR entries (and vertices) run their MIS and
// BFS as resident kernels over work items of at most kItemEdges entries.  The
// kernels read every row each round, the host-driven rounds only what the
// frontier needs, so the lines lie where the reads outgrow the launches.  MIS
// with keys, resident against host-driven: Erdos-Renyi 0.08 M entries 0.57 /
// 3.55 ms, 0.8 M 1.28 / 5.91, 10 M 1.90 / 4.10; R-MAT 1.8 M 0.46 / 1.18, 7.6 M
// 1.05 / 1.40, 15.5 M 2.65 / 1.90.
//
// A round costs a step per item, and a vertex is an item however short its row:
// graphs of short rows are bounded by their items too (kResidentItems; resident
// against host-driven in ms, by million items).
//   MIS, balls of up to 64 hops: Erdos-Renyi 1.2 2.77 / 4.73,
//   1.5 12.9 / 14.1, 2.0 6.47 / 5.71; R-MAT 1.2 1.80 / 1.63, 2.0 3.34 / 2.30; square
//   grid, 40 to 48 hops, 1.3 16.8 / 19.9 and 19.4 / 20.9, 1.6 22.1 / 22.2.
//   MIS, larger balls, whose sweeps are mostly thin (kWideBallItems): grid, 70 to
//   120 hops, 0.7 20.8 / 28.4, 1.0 31.4 / 37.1, 1.1 21.9 / 19.9, 1.3 21.3 / 18.2, 1.6
//   32.4 / 23.4, 2.2 79.8 / 53.9.
//   BFS: R-MAT 1.0 0.30 / 0.53, 1.2 0.36 / 0.39, 2.0 0.58 / 0.64; Erdos-Renyi 1.0 0.38 /
//   0.47, 1.5 1.05 / 1.12, 2.0 0.86 / 0.82, 4.0 3.18 / 1.80; grid, 55 levels, 1.0 1.86 /
//   2.44, 1.4 2.51 / 2.78, 2.2 3.74 / 3.42; 6 levels 1.4 0.62 / 0.46.  Whole batches,
//   replicas of R-MAT 1.3 3.90 / 5.09, union of Erdos-Renyi graphs 1.3 16.7 / 21.4.
constexpr int64_t kResidentEdges = 10 << 20;
constexpr int64_t kResidentItems = 3 << 19;
constexpr int64_t kWideBallItems = 1 << 20;  // above: only balls of at most kNarrowBall hops
constexpr int kNarrowBall = 64;
constexpr int kItemEdges = 64;
// Pinned host block of a graph: its Counters mirror, then scratch of a call.
constexpr size_t kPinnedBytes = 16384;
// Width of the masks of the sketch hops (a sketch that holds only ordinals
// below kUW is a kUW-bit mask).
constexpr int kUW = 1024;
constexpr int kUSlices = kUW / 256;  // a mask is read and merged in 256-bit slices
constexpr int kUWords = kUW / 64;

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

__device__ __forceinline__ uint64_t umin64(uint64_t a, uint64_t b) { return a < b ? a : b; }

// HIP weight of a group whose ball holds cnt ranks with k-th smallest kth:
// 1 while the ball has fewer than k vertices, else 1 / Pr[rank < k-th] =
// 2^64 / kth (one IEEE division).
__device__ __forceinline__ double hip_weight(int cnt, int k, uint64_t kth) {
    return cnt < k ? 1.0 : __ddiv_rn(18446744073709551616.0, __ull2double_rn(kth));
}

// Position of the n-th (0-based) set bit of m (m must have > n set bits).
__device__ __forceinline__ int nth_set_bit(unsigned m, int n) {
    int pos = 0;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        unsigned low = m & ((1u << s) - 1u);
        int c = __popc(low);
        if (n >= c) {
            n -= c;
            m >>= s;
            pos += s;
        } else {
            m = low;
        }
    }
    return pos;
}

__device__ __forceinline__ int warp_incl_scan(int x) {
    const int lane = lane_id();
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
        int y = __shfl_up_sync(kFull, x, s);
        if (lane >= s) x += y;
    }
    return x;
}

// Warp-aggregated append: every lane with `pred` gets a distinct slot index
// from `counter` (one atomic per warp); lanes without it get -1.  All 32
// lanes must call it.
__device__ __forceinline__ long long warp_append(bool pred, unsigned long long* counter) {
    const int lane = lane_id();
    unsigned m = __ballot_sync(kFull, pred);
    if (!m) return -1;
    int leader = __ffs(m) - 1;
    unsigned long long base = 0;
    if (lane == leader) base = atomicAdd(counter, (unsigned long long)__popc(m));
    base = __shfl_sync(kFull, base, leader);
    return pred ? (long long)(base + __popc(m & ((1u << lane) - 1u))) : -1LL;
}

// Append with one global atomic per block and call: the block's warps take
// consecutive places.  Every thread of the block calls it the same number of
// times (a block-uniform loop); blockDim.x = 32 * W.  Which places a block
// gets depends on the order of the blocks' atomics, like warp_append.
template <int W>
struct BlockAppend {
    unsigned cnt[W];
    unsigned long long off[W];
};

template <int W>
__device__ __forceinline__ long long block_append(bool pred, unsigned long long* counter, BlockAppend<W>& sh) {
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const unsigned m = __ballot_sync(kFull, pred);
    if (lane == 0) sh.cnt[warp] = __popc(m);
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long total = 0;
        for (int w = 0; w < W; ++w) {
            sh.off[w] = total;
            total += sh.cnt[w];
        }
        const unsigned long long base = total ? atomicAdd(counter, total) : 0ULL;
        for (int w = 0; w < W; ++w) sh.off[w] += base;
    }
    __syncthreads();
    return pred ? (long long)(sh.off[warp] + __popc(m & ((1u << lane) - 1u))) : -1LL;
}

// Adds the threads' counts to *counter, one global atomic per block (a launch
// of thousands of warps that each add to the same word waits for the word, some
// 2 ns an add).  Every thread of the block calls it, once per launch.
__device__ __forceinline__ void block_count(unsigned x, unsigned long long* counter) {
    __shared__ unsigned s_part[32];
    x = __reduce_add_sync(kFull, x);
    if (lane_id() == 0) s_part[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x < 32) {
        const unsigned long long y = __reduce_add_sync(kFull, threadIdx.x < (blockDim.x >> 5) ? s_part[threadIdx.x] : 0u);
        if (threadIdx.x == 0 && y) atomicAdd(counter, y);
    }
}

// ----------------------------------------------------------------- groups in lockstep
// A group is G consecutive lanes (16 or 32) that work on one vertex.  The two
// half-warp groups of a warp run in lockstep: every lane of the warp executes
// every group operation, a group without work carries empty ranges and empty
// lists through it, and branches are taken by the whole warp.  (Groups that
// diverge are executed one after the other, which cost half the issue slots.)
// A G-lane list holds up to G ordinals, one per lane, ascending, kNil after.

constexpr uint32_t kNil = 0xffffffffu;  // empty sketch or list slot

template <int G>
struct Lock {
    int l;      // lane within the group
    int shift;  // position of the group's bits in a warp ballot
    __device__ __forceinline__ Lock() {
        const int lane = lane_id();
        l = lane & (G - 1);
        shift = lane & ~(G - 1);
    }
    __device__ __forceinline__ unsigned mine(unsigned b) const { return G == 32 ? b : (b >> shift) & 0xffffu; }
    __device__ __forceinline__ unsigned ballot(bool p) const { return mine(__ballot_sync(kFull, p)); }
    __device__ __forceinline__ unsigned below() const { return (1u << l) - 1u; }  // the lanes before this one
    template <class T>
    __device__ __forceinline__ T shfl(T x, int src) const { return __shfl_sync(kFull, x, src, G); }
    template <class T>
    __device__ __forceinline__ T shfl_xor(T x, int m) const { return __shfl_xor_sync(kFull, x, m, G); }
    template <class T>
    __device__ __forceinline__ T shfl_up(T x, int d) const { return __shfl_up_sync(kFull, x, d, G); }
};

__device__ __forceinline__ bool warp_any(bool p) { return __any_sync(kFull, p); }

template <int G>
__device__ __forceinline__ uint32_t lock_sort(const Lock<G>& g, uint32_t x) {
#pragma unroll
    for (int k = 2; k <= G; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const uint32_t y = g.shfl_xor(x, j);
            const bool up = (g.l & k) == 0 || k == G;
            const bool low = (g.l & j) == 0;
            x = low == up ? min(x, y) : max(x, y);
        }
    }
    return x;
}

// Entries of the list L below x (0..G) and whether x is one of them.
template <int G>
__device__ __forceinline__ int lock_find(const Lock<G>& g, uint32_t L, uint32_t x, bool& member) {
    int pos = 0;
#pragma unroll
    for (int s = G / 2; s > 0; s >>= 1)
        if (g.shfl(L, pos + s - 1) < x) pos += s;
    const uint32_t y = g.shfl(L, pos);
    member = y == x;
    return pos + (y < x ? 1 : 0);
}

template <int G>
__device__ __forceinline__ uint64_t lock_or64(const Lock<G>& g, uint64_t x) {
    unsigned lo = (unsigned)x, hi = (unsigned)(x >> 32);
    if (G == 32) {
        lo = __reduce_or_sync(kFull, lo);
        hi = __reduce_or_sync(kFull, hi);
    } else {
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) {
            lo |= g.shfl_xor(lo, o);
            hi |= g.shfl_xor(hi, o);
        }
    }
    return ((uint64_t)hi << 32) | lo;
}

// Running sketch of one group: list `sk` (k valid lanes) and the filter `tau`:
// its k-th ordinal (kNil while it is not full), at most `tau_base` (kNil for a
// vertex's own sketch, the vertex's old k-th ordinal for a hub partial).
template <int G>
struct Sketch {
    uint32_t sk, tau, tau_base;
    __device__ __forceinline__ void retau(const Lock<G>& g, int k) { tau = min(g.shfl(sk, k - 1), tau_base); }
};

// Insert one ordinal per group (x uniform over the group; groups without
// `want` keep their sketch).
template <int G>
__device__ __forceinline__ void insert_one(const Lock<G>& g, int k, uint32_t x, bool want, Sketch<G>& s) {
    const bool dup = g.ballot(s.sk == x) != 0;
    const int p = __popc(g.ballot(s.sk < x));
    const uint32_t up = g.shfl_up(s.sk, 1);
    if (want && !dup) {
        s.sk = g.l > p ? up : (g.l == p ? x : s.sk);
        if (g.l >= k) s.sk = kNil;
    }
    s.retau(g, k);
}

// Merge candidates, ascending over the lanes that have one (kNil: none; no
// repeats among them): each lane finds its place in the sketch by search,
// candidates already there drop out, and the others take the places
// (entries below) + (kept candidates before); the sketch's entries fill the
// places left.  Candidates pass through shared memory to their places.
template <int G>
__device__ __forceinline__ void merge_sorted(const Lock<G>& g, int k, uint32_t x, Sketch<G>& s, uint32_t* sx) {
    bool member;
    const int pos = lock_find(g, s.sk, x, member);
    const bool keep = x != kNil && !member;
    const unsigned km = __ballot_sync(kFull, keep);
    if (!km) return;
    const int dest = pos + __popc(g.mine(km) & g.below());
    const bool fits = keep && dest < G;
    const unsigned occ = g.mine(__reduce_or_sync(kFull, fits ? 1u << (dest + g.shift) : 0u));
    if (fits) sx[g.shift + dest] = x;
    __syncwarp();
    const uint32_t old = g.shfl(s.sk, g.l - __popc(occ & g.below()));
    const uint32_t nv = (occ >> g.l) & 1u ? sx[g.shift + g.l] : old;
    __syncwarp();
    s.sk = g.l < k ? nv : kNil;
    s.retau(g, k);
}

// Merge a sorted list: the entries below tau form a prefix, absorbed by one or
// two insertions or one merge.
template <int G>
__device__ __forceinline__ void merge_list(const Lock<G>& g, int k, uint32_t x, Sketch<G>& s, uint32_t* sx) {
    const bool in = x < s.tau;
    const unsigned b = __ballot_sync(kFull, in);
    if (!b) return;
    const int c = __popc(g.mine(b));
    if (!warp_any(c > 2)) {
        insert_one(g, k, g.shfl(x, 0), c > 0, s);
        if (warp_any(c > 1)) {
            const uint32_t x1 = g.shfl(x, 1);
            insert_one(g, k, x1, c > 1 && x1 < s.tau, s);
        }
    } else {
        merge_sorted(g, k, in ? x : kNil, s, sx);
    }
}

// Absorb one batch of candidates (one per lane, kNil = none; unsorted, may
// repeat or already be in the sketch): filter by tau, then insert one by one
// when few survive, else sort and merge.
template <int G>
__device__ __forceinline__ void absorb(const Lock<G>& g, int k, uint32_t x, Sketch<G>& s, uint32_t* sx) {
    unsigned m = g.ballot(x < s.tau);
    if (!warp_any(m != 0)) return;
    if (!warp_any(__popc(m) > 3)) {
        while (warp_any(m != 0)) {
            const uint32_t y = g.shfl(x, m ? __ffs(m) - 1 : 0);
            insert_one(g, k, y, m != 0 && y < s.tau, s);
            m &= m - 1;
        }
    } else {
        x = lock_sort(g, x < s.tau ? x : kNil);
        const uint32_t prev = g.shfl_up(x, 1);
        merge_sorted(g, k, g.l > 0 && prev == x ? kNil : x, s, sx);
    }
}

// ----------------------------------------------------------------- resident kernels
// A cooperative launch of blocks of kResThreads threads, at most one per SM,
// that separates its passes by grid barriers.

constexpr int kResThreads = 1024;
constexpr int kResWarps = kResThreads / 32;
constexpr unsigned kWaitLimit = 1u << 25;   // barrier polls; past the limit the kernel returns

struct GridBar {
    unsigned long long pass[8];       // per pass (mod 8): counts of its threads << 32 | blocks arrived
    unsigned err;                     // bit 0: a barrier wait ran out (other bits: the kernel's own)
    unsigned pad;
};

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// End of a pass: a grid barrier that adds up the threads' counts on the way
// (one word per pass holds both, so the last poll also brings the total).
// *total is the same on every thread; false when the wait ran out.  The word
// of two passes ahead is cleared here.
__device__ __forceinline__ bool end_pass(GridBar* c, unsigned& pass, unsigned mine, unsigned* total) {
    __shared__ unsigned s_sum[kResWarps];
    __shared__ unsigned long long s_word;
    mine = __reduce_add_sync(kFull, mine);
    if (lane_id() == 0) s_sum[threadIdx.x >> 5] = mine;
    __syncthreads();
    if (threadIdx.x < 32) {
        const unsigned x = __reduce_add_sync(kFull, s_sum[threadIdx.x]);
        if (threadIdx.x == 0) {
            if (blockIdx.x == 0) c->pass[(pass + 2) & 7] = 0;
            unsigned long long* word = &c->pass[pass & 7];
            __threadfence();
            atomicAdd(word, ((unsigned long long)x << 32) | 1ULL);
            unsigned long long w = 0;
            unsigned polls = 0;
            while ((unsigned)(w = ld_acquire(word)) < gridDim.x) {
                if (++polls > kWaitLimit) {
                    atomicOr(&c->err, 1u);
                    w = ~0ULL;
                    break;
                }
            }
            __threadfence();
            s_word = w;
        }
    }
    __syncthreads();
    const unsigned long long w = s_word;
    *total = (unsigned)(w >> 32);
    ++pass;
    return w != ~0ULL;
}

// ----------------------------------------------------------------- device counters

// Small block of device counters read back by the host between launches.
struct Counters {
    unsigned long long frontier;     // vertices appended to the next frontier
    unsigned long long active;       // vertices in the active list of a hop
    unsigned long long stg_entries;  // ADS staging entries used
    unsigned long long stg_groups;   // ADS staging groups used
    unsigned long long merges;       // edge-merges of the next hop (sum of deg of frontier)
    unsigned long long error;        // nonzero: a kernel detected a bad input
    unsigned long long aux0;         // general purpose
    unsigned long long cand_reads;   // merge: neighbour-delta ranks read (sum of |D_{h-1}(u)| over frontier edges)
    unsigned long long merging;      // merge: vertices with at least one frontier neighbour
    unsigned long long aux3;
    unsigned long long scanned;      // hop census: CSR entries read this hop
    unsigned long long mask_scanned; // hop census: of those, read by the mask merge
    unsigned long long delta_next;   // merge: sum of deg(u) * |D_h(u)| over changed u (delta ranks of the next hop's edge-merges)
    unsigned long long new_entries;  // merge: entries gained this hop (sum of |D_h(v)|)
    unsigned long long key_or;       // keys: OR of the candidates' radius words
    unsigned long long key_orn;      // keys: OR of their complements (a bit set in both varies)
    unsigned long long key_ties;     // keys: 1: a run of equal prefixes too long to order in place, 2: equal radii out of order
};

// ----------------------------------------------------------------- profiling
// Kernel classes for launch counts and CUDA-event timings.
enum ProfClass {
    kProfSketchMerge = 0,  // the hop kernels (k_hop_*), k_wbuild
    kProfSketchExpand = 1, // k_expand
    kProfSketchOther = 2,  // rank init, ADS compaction, scans, eccentricity bound
    kProfRadius = 3,
    kProfKeys = 4,         // candidates, radix sort, ordinals
    kProfMis = 5,          // greedy-MIS rounds
    kProfBfs = 6,          // assignment BFS
    kProfOther = 7,        // validation, exports, objective
    kProfExact = 8,        // exact ball sizes, their HIP estimates, exact-count radii
    kProfClasses = 9
};

struct Prof {
    int on = 0;
    int64_t launches[kProfClasses] = {};
    double ms[kProfClasses] = {};
    double bytes[kProfClasses] = {};
    std::vector<cudaEvent_t> ev;   // pool of (start, stop) pairs
    std::vector<int> cls;          // class of each recorded pair
    size_t used = 0;
};

// The profiler of the handle whose API call is running on this thread.
Prof* current_prof();
void set_current_prof(Prof* p, cudaStream_t st);
int prof_begin(int cls);           // counts the launch; records a start event when on
void prof_end(int slot);           // records the stop event
int prof_drain(Prof* p);           // after a stream sync: accumulate elapsed times

// Launch a kernel statement and account it to a class.
#define FL_LAUNCH(cls, ...)                      \
    do {                                         \
        int slot__ = ::fl::prof_begin(cls);      \
        __VA_ARGS__;                             \
        ::fl::prof_end(slot__);                  \
    } while (0)

// ----------------------------------------------------------------- schedules
// Launch and round-switch parameters of a graph: they change how fast the
// path runs, never what it computes.
struct Sched {
    int hop_group = 0;    // lanes per vertex in the sketch hop for k <= 16 (16 or 32; 0: 16)
    int sparse_div = 16;  // a hop runs sparse when frontier * sparse_div < listed vertices
    int dense_div = 8;    // a relaxation round pulls when frontier * dense_div >= listed vertices
    int edge_div = 16;    // ... or when frontier edges * edge_div >= nnz
    int graph_bfs = 0;    // 1: the assignment BFS runs as one CUDA graph (a device-side level loop)
    int level_cap = 0;    // BFS levels at most (0: n + 2); beyond it FL_ETIMEOUT
    // dense_div or edge_div set: the caller asks for rounds that these switch
    bool switches_rounds() const { return dense_div != 8 || edge_div != 16; }
};

// ----------------------------------------------------------------- graph BFS
// A level-synchronous BFS run as one CUDA graph (k_solve.cu): its
// instantiation, cached per graph handle (prefix views of a batch share it)
// and rebuilt when the buffers or sizes it was built for change.
struct GraphBfs {
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    const void* key[4] = {nullptr, nullptr, nullptr, nullptr};
    int64_t key_n[4] = {0, 0, 0, 0};
    DBuf state;  // level (uint32), vertices reached this level, error flag
};

// ----------------------------------------------------------------- handles

}  // namespace fl

struct fl_graph {
    int64_t n = 0, nnz = 0;
    cudaStream_t stream = nullptr;
    fl::DBuf rowp, cols;           // int64[n+1], int32[nnz]
    fl::DBuf wts;                  // int32[nnz]: edge lengths of a weighted graph, else empty
    fl::DBuf wrev;                 // uint32[nnz]: (weighted) the entry (v, u) paired with each entry (u, v)
    int max_w = 0;                 // largest edge length
    int64_t wlevels = 0;           // distance levels with active vertices in the last weighted build
    // static work lists: non-hub non-isolated vertices, hubs, hub segments
    int lists_ready = 0;
    fl::DBuf low_list, hub_list;   // int32[n_low], int32[n_hubs]
    // the non-hub vertices split by degree for the relaxation rounds: at most
    // kSmallDeg neighbours (a thread each), more (a group of lanes each)
    fl::DBuf small_list, mid_list; // int32[n_small], int32[n_mid]
    int64_t n_small = 0, n_mid = 0;
    int seg = fl::kMaxSeg;         // longest row that is not a hub's, and edges per hub segment
    fl::DBuf hub_seg;              // int64[n_hubs+1]: first segment of each hub
    fl::DBuf seg_hub;              // int32[n_seg]: hub of each segment
    int64_t n_low = 0, n_hubs = 0, n_seg = 0;
    fl::DBuf items;                // int4[n_items]: work items of the resident kernels
    int64_t n_items = 0;           // 0: the graph is too large for them (kResidentEdges, kResidentItems)
    fl::DBuf part;                 // uint32[n_seg*k]: partial bottom-k of each hub segment (scratch)
    // A graph that is a disjoint union of parts (batched instances): vertex v
    // of the part starting at vbase[v] has local id v - vbase[v], and ranks
    // and priorities are those of the local id, so every part is solved
    // exactly as it would be alone.  Empty for an ordinary graph.
    fl::DBuf vbase;                // int32[n] or empty
    fl::DBuf vpart;                // int32[n]: part of each vertex (with vbase)
    // relabelled graphs (see IdMap): rid = original id of each internal
    // vertex, inv = internal id of each original id; unions keep rid = local id
    fl::DBuf rid, inv;             // int32[n] or empty
    bool relabelled = false;
    int64_t n_parts = 0;           // 0: not a union
    int64_t max_part = 0;          // union: vertices of the largest part
    fl::DBuf ord;                  // uint32[n]: ordinal of each vertex's rank (unions: among the local ids)
    fl::DBuf ord_rid, ord_vid;     // int32: rank id and vertex (unions: local id) of each ordinal
    fl::DBuf DM[2];                // uint64[kUSlices][n][4]: hop delta masks, slice-major
    fl::DBuf PM;                   // uint64[n_seg*kUWords]: partial masks of hub segments (scratch)
    fl::DBuf seg_flag;             // uint8[n_seg]: the segment had a neighbour that gained entries (scratch)
    fl::DBuf PH;                   // uint64[n_seg]: OR of the segment's neighbours' delta heads (scratch)
    fl::DBuf F[2];                 // uint32[n]: smallest new ordinal of the hop (all ones: none)
    fl::DBuf H[2];                 // uint64[n]: delta bits over the ordinals 0..63
    fl::DBuf W;                    // uint64[n]: own sketch's mask over the ordinals 0..63 of head vertices, else 0
    fl::DBuf fbm;                  // uint32[n/32+1]: frontier bitmap of the previous hop
    // sketches
    int k = 0;
    uint64_t seed = 0;
    int built = 0;
    uint64_t generation = 0;       // bumped by every build
    fl::DBuf S, Scnt;              // uint32[n*k] ordinals, uint8[n]
    fl::DBuf D[2], Dcnt[2];        // hop deltas (ordinals), counts
    fl::DBuf frontier[2];          // int32[n]
    fl::DBuf stamp;                // uint32[n]
    fl::DBuf vg, ve;               // int32[n] per-vertex running group / entry counts
    fl::DBuf stg_ent, stg_kth;     // uint32 staging entries (k per slot), k-th ordinals (one per slot)
    fl::DBuf stg_grp;              // staging group records (one per slot)
    size_t stg_grp_cap = 0;        // slots
    int stg_k = 0;
    // ADS (vertex-major)
    fl::DBuf gofs, eofs;           // int64[n+1]
    fl::DBuf ginfo, gwt, eid;      // uint32[G], double[G], int32[E]
    int64_t hops = 0, edge_merges = 0, n_entries = 0, n_groups = 0;
    // per-vertex eccentricity upper bound (caps ball radii; balls unchanged)
    fl::DBuf ecc_ub;               // int32[n]
    // counters + scratch
    fl::DBuf ctr;                  // Counters
    fl::Counters* h_ctr = nullptr; // pinned host mirror
    fl::DBuf scratch;              // general scratch (scans, sorts)
    fl::DBuf relax_aux;            // bitmap, hub frontier tags/values, edge counter of the rounds
    fl::Prof prof;                 // launch counts and kernel timings
    fl::Sched sched;               // launch and round-switch schedule (fl_set_schedule, fl_autotune)
    fl::GraphBfs* gbfs = new fl::GraphBfs();  // the CUDA-graph BFS of this handle (shared by prefix views)
    // per-hop counters of the last build (index h-1)
    std::vector<int64_t> hop_scanned, hop_mask, hop_changed;
    std::vector<double> hop_ms;
    // per-hop terms of the algorithmic-bytes model of a hop: edge-merges E_h,
    // merging vertices A_h, neighbour-delta ranks the kernels read R_h, the
    // delta ranks of the edge-merges sum |D_{h-1}(u)| over E_h, new entries |D_h|
    std::vector<int64_t> hop_E, hop_A, hop_R, hop_SD, hop_new;
    cudaEvent_t hop_ev[2] = {nullptr, nullptr};
    // exact sizes and radii: source bits (visited, two frontiers), row-length
    // lists and sweep state, staged query inputs and outputs
    fl::DBuf xbits, xaux, xio;
};

namespace fl {
inline IdMap idmap_of(const fl_graph* g) {
    IdMap m;
    m.rid = g->rid.p ? g->rid.as<int32_t>() : nullptr;
    m.inv = g->relabelled ? g->inv.as<int32_t>() : nullptr;
    m.vbase = (!g->relabelled && g->vbase.p) ? g->vbase.as<int32_t>() : nullptr;
    return m;
}
}  // namespace fl

struct fl_solve {
    fl_graph* g = nullptr;
    uint64_t generation = 0;
    int have_radii = 0, have_open = 0, have_assign = 0;
    fl::DBuf cost, client;         // double[n], uint8[n]
    fl::DBuf radii;                // double[n]
    fl::DBuf ord, fac_by_ord, bcap, state, claimed;  // MIS state
    fl::DBuf reach;                // uint8[n]: 1 + slack of a vertex in the current cover (gather pruning)
    fl::DBuf kill;                 // uint8[n]: 1 + distance to a client claimed in the current round
    fl::DBuf rlist, rctl;          // resident kernels: item lists of the greedy rounds, control block and log
    std::vector<int64_t> mis_log;  // rows of 6: the rounds of the last MIS (fl_mis_log)
    fl::DBuf X, stamp, mval, fr[2], frval, touched, ulist, ubuck, bcount;
    fl::DBuf key_hi, key_lo, key_val, key_alt, obj_tmp;  // key sort and objective scratch
    fl::DBuf part_T;               // int32[n_parts]: largest ball radius of a part's undecided facilities
    fl::DBuf io;                   // per-vertex inputs/outputs in original order (relabelled graphs)
    fl::DBuf open;                 // uint8[n]
    fl::DBuf assign, dist;         // int32[n]
    int64_t n_cand = 0, n_open = 0, mis_rounds = 0;
    // opening phase with eps > 0: per-vertex iterations and scratch, the grid
    // tables, one iteration's selection inputs, statistics of the last run
    fl::DBuf eps, eps_tab, eps_ev, eps_out, eps_r, eps_c;
    double eps_gamma = -1.0, eps_alpha0 = 0.0;
    int64_t eps_iterations = 0, eps_events = 0, eps_groups = 0;
    int have_eps = 0;
};

namespace fl {

// Shares of the keys in a counting kernel of m keys (a block per 64 keys and
// share): about eight blocks of 256 threads per SM, at least 512 keys each.
inline unsigned count_shares(int64_t m) {
    const int64_t groups = (m + 63) / 64, want = (152 * 8 + groups - 1) / groups, most = (m + 511) / 512;
    return (unsigned)(want < most ? want : most);
}

// ----------------------------------------------------------------- kernel launchers
// (implemented in the .cu files; all run on g->stream)

int scan_exclusive_i64(const int64_t* in, int64_t* out, int64_t n, cudaStream_t st, DBuf& tmp,
                       int cls = kProfSketchOther);
int scan_exclusive_i32_to_i64(const int32_t* in, int64_t* out, int64_t n, cudaStream_t st, DBuf& tmp,
                              int cls = kProfSketchOther);
// Stable LSD radix sort of (key, payload) pairs (k_sort.cu).  The pairs are in
// buffer `cur` before and after; shift[0..nd) are the low bits of the 8-bit
// digits, least significant first.  A wait of the sort that runs out sets
// kSortError in *err (never on a working device).
constexpr int kSortDigits = 8;
constexpr unsigned long long kSortError = 1ULL << 16;
template <class K>
struct SortPairs {
    K* key[2];
    uint32_t* val[2];
    int cur = 0;
};
template <class K>
int sort_pairs(SortPairs<K>& p, int64_t n, const int* shift, int nd, cudaStream_t st, DBuf& tmp, int cls,
               unsigned long long* err);
// 8-bit digits that cover the set bits of `varying` (bits > 0: only that many
// from its highest one down); returns their number.  The keys agree below
// shift[0] only if every varying bit is covered.
int digit_windows(uint64_t varying, int bits, int* shift);

int validate_csr(fl_graph* g);
int build_work_lists(fl_graph* g);
int build_sketches(fl_graph* g, int k, uint64_t seed);
int build_ordinals(fl_graph* g, DBuf& tmp);
// weighted graphs (k_wsketch.cu): length check, and the build in Dijkstra order
int check_weights(fl_graph* g);
int pair_reverse_edges(fl_graph* g);
int build_sketches_weighted(fl_graph* g, int k, uint64_t seed);
int compute_ecc_bound(fl_graph* g);

int check_costs(fl_solve* s);
int compute_radii(fl_solve* s);
int sort_candidates(fl_solve* s, int64_t* m_out, const uint32_t** sorted, int64_t known = -1);
int open_facilities(fl_solve* s);
int open_facilities_queued(fl_solve* s, int64_t known, uint8_t* acc, int* outcome, bool* queued);
// the greedy MIS and the assignment by weighted distance (k_wsolve.cu)
int open_facilities_weighted(fl_solve* s);
int assign_weighted(fl_solve* s);
int msbfs(fl_graph* g, const int32_t* src_list, int64_t n_src, int32_t* label, int32_t* dist,
          DBuf& X, DBuf& stampb, DBuf* fr, DBuf& frval, int cls);
int msbfs_graph(fl_graph* g, const int32_t* src_list, int64_t n_src, int32_t* label, int32_t* dist, DBuf& X,
                DBuf& stampb, int cls);
void graph_bfs_release(GraphBfs* c);
// resident kernels of small graphs (k_resident.cu): graphs with work items whose
// schedule leaves the round switches alone (a pull has no push to switch to)
inline bool runs_resident(const fl_graph* g) { return g->n_items > 0 && !g->sched.switches_rounds(); }
int build_items(fl_graph* g);
int mis_resident(fl_solve* s, int64_t m, bool* done);
int mis_resident_queue(fl_solve* s, int64_t m, uint8_t* acc, int* outcome);
int msbfs_resident(fl_graph* g, const int32_t* src, int64_t n_src, int32_t* label, int32_t* dist, DBuf& ctl, DBuf& lists,
                   int cls);

// Per-vertex pruning of the rounds of a sweep (the MIS cover and gather
// sweeps).  A round that first gives v a value below the limit records
// reach[v] = reach_val; a round skips every v with need[v] <= round, and
// every v with only[v] == 0: it does not lower v's value, and a push does
// not offer v one.
struct Prune {
    uint8_t* reach = nullptr;
    const uint8_t* need = nullptr;
    const uint8_t* only = nullptr;
    uint32_t reach_val = 0, round = 0;
};

// State of a sequence of synchronous min-propagation rounds (k_relax.cu).
struct Relax {
    bool narrow = false;                            // 32-bit values (else 64-bit)
    void* X[2] = {nullptr, nullptr};                // value buffers; X[cur] is current
    int cur = 0;
    int32_t* fr[2] = {nullptr, nullptr};            // frontier lists; fr[fc] is current
    int fc = 0;
    void* frval = nullptr;                          // snapshot of frontier values
    uint32_t* stamp = nullptr;                      // frontier stamps / changed flags
    unsigned long long* cnt = nullptr;              // device: [0], [1] list sizes, [2] changed count
    unsigned long long* h_cnt = nullptr;            // pinned host word
    int64_t n_front = 0;                            // host copy of the frontier size
    bool list_valid = true;                         // fr[fc] lists the frontier
    uint32_t sv_prev = 0;                           // stamp of the current frontier
    unsigned long long limit = ~0ULL;               // values >= limit are ignored by pulls
    int dense_div = 8;                              // pull when frontier * dense_div >= vertices
    int edge_div = 16;                              // pull when frontier edges * edge_div >= nnz
    bool settle = false;                            // a value < limit is final (level-synchronous BFS)
    // set by relax_begin (graph-owned scratch)
    uint32_t* bm = nullptr;                         // frontier bitmap of a pull round (n bits)
    uint32_t* hub_tag = nullptr;                    // uint32[n_hubs]: round whose push frontier holds the hub
    void* hub_val = nullptr;                        // [n_hubs]: the hub's snapshotted value
    unsigned long long* ecnt = nullptr;             // device: frontier edge count
    int32_t* part_cnt = nullptr;                    // device int32[n_parts]: frontier vertices per part
    const int32_t* part_limit = nullptr;            // device int32[n_parts] or NULL: a part whose limit is
    int32_t part_round = 0;                         //   below part_round sits the pull rounds out
    Prune prune;                                    // per-vertex reach / need of the sweep
    bool last_dense = false;                        // the last round pulled
};
// Binds the graph-owned scratch of the rounds to r; call once per sweep
// family, after r.stamp values of earlier users may have been reused.
int relax_begin(fl_graph* g, Relax& r);
int relax_round(fl_graph* g, Relax& r, unsigned long long add, uint32_t sv, int cls);
int relax_prepare_list(fl_graph* g, Relax& r, int cls);
// One round of a bounded marking BFS over g (k_relax.cu): kr[v] = b + 1 for
// every unmarked v with need[v] > b (need may be NULL) and a neighbour whose
// kr is in [1, b]; *marked = the marks made (hubs may count more than once).
int mark_round(fl_graph* g, Relax& r, uint8_t* kr, const uint8_t* need, uint32_t b, int cls, int64_t* marked);
int relax_collect_set(fl_graph* g, const uint32_t* X, int32_t* out, unsigned long long* n_out, int cls);
int assign_clients(fl_solve* s);
// the opening phase with eps > 0 and the selection of Algorithm 6 (k_eps.cu)
int open_facilities_eps(fl_solve* s, double eps);
const int32_t* eps_iterations_of(const fl_solve* s, bool clients);
// exact neighbourhood sizes, their HIP estimates, exact-count radii (k_exact.cu)
int map_sources(fl_graph* g, const int32_t* in, int64_t n_src, int32_t* out);
int exact_ball_sizes(fl_graph* g, int64_t n_src, const int32_t* src, int64_t D, const uint8_t* pred, int64_t* out);
int hip_ball_estimates(fl_graph* g, int64_t n_src, const int32_t* src, int64_t D, const uint8_t* pred, double* out);
int exact_radii(fl_solve* s);
int objective(fl_solve* s, double* obj, int64_t* dist_sum, int64_t* n_unserved);

int read_counters(fl_graph* g);
// batches (k_batch.cu)
int batch_place_parts(fl_graph* U, const std::vector<int64_t>& voff, const std::vector<int64_t>& eoff);
int batch_check_parts(fl_graph* U);
int batch_replicate(const fl_graph* G, int64_t R, fl_graph* U);
int batch_replicate_ecc(const fl_graph* G, int64_t R, fl_graph* U);
int batch_objective(fl_solve* s, const int64_t* off_d, int n_inst, double* obj, long long* n_open,
                    long long* dist_sum, long long* unserved);
int compute_radii_multi(const fl_graph* src, fl_graph* g, int64_t R, const double* cost, const uint8_t* client,
                        double* radii);
int relax_reserve(fl_graph* g);
// vertex numbering by descending degree (k_relabel.cu)
int relabel_graph(fl_graph* g);
template <class T>
int permute_vertices(const fl_graph* g, const T* in, T* out, int64_t reps, bool to_internal, cudaStream_t st);
int sketch_ranks_original(const fl_graph* g, uint64_t* out);
int ads_original(fl_graph* g, int64_t* gofs_o, int64_t* eofs_o, uint32_t* ginfo_o, double* gwt_o, int32_t* eid_o);

}  // namespace fl

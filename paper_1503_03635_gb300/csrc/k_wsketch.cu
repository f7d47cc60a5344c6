// k_wsketch.cu -- sketches and ADS of a weighted graph (Section 3.3 after
// Algorithm 2; edge weights drawn uniformly in [1, 100] in Section 5).
//
// The paper's Algorithm 2 runs in BFS-order supersteps, so on a weighted
// graph a vertex can accept an entry that a closer arrival later pushes out
// of the bottom-k, and a CleanUp step removes such entries.  This build runs
// in Dijkstra order instead: level L of the loop settles every ADS entry at
// distance exactly L, so an accepted entry is final and nothing needs
// cleaning (both orders end at the ADS of the definition).  Lengths are
// positive integers, so the levels are the integers 0, 1, 2, ... up to the
// largest distance (at most 65535, the width of a group's distance field).
//
// Level L: v is active when a neighbour u gained entries at distance
// L - w(u, v); a ring of (largest length + 1) bitmaps holds the activations
// of the coming levels, and a second ring of bitmaps over the CSR entries
// marks which entries (v, u) of an active v deliver at that level (u posts
// to the entry of v's row paired with its own entry (u, v), so v reads only
// the neighbours that gained).  u posts to v only if one of the ranks it
// gained is below v's k-th rank and not in v's sketch: k-th ranks only fall
// and a rank that leaves a sketch never returns, so the others could not
// enter v's sketch at level L either.  (Most are already there: every
// neighbour of v that holds a rank would offer it again.)  An active v merges
// into its bottom-k sketch the entries of each posting neighbour u at distance
// L - w(u, v), found by an 8-way search in u's row, which is in distance order; the
// ranks that enter form v's group at distance L, with the HIP weight and
// counted prefix of the unweighted build (the sketch after the level, ties at
// one distance in ascending rank).  Entries appended at level L have distance
// L and are never read in the same level (every length is >= 1): a level reads
// the row counts as they were when it started and writes the new counts to a
// second array, which the next level's first pass copies back.
//
// The whole loop is one resident kernel, two grid barriers per level (collect
// the active vertices; merge and post) and a third where hubs were active (post
// theirs), in place of three launches and a look at the ring by the host.  A
// warp merges an active vertex; a hub (a row above kWHub entries) is merged by a
// block, each warp taking every 32nd part of its marks into a copy of the
// sketch.  Posts are dealt out 32 entries at a time: a hub's to the warps of
// the grid, those of other rows above kWLong entries to the warps of the block.
// With a warp per merge and a block per hub's posts, a level of 30 k active
// vertices waited some 100 us for the block that held the hub (merge 270 k
// cycles, average of the blocks 100 k; posts 230 k, average 49 k).
// Bound by the latency of the dependent loads of a merge and of a post (column,
// row, sketch).  R-MAT, 65 k vertices, lengths up to 100, k = 16, 313 levels:
// 115 ms of level kernels and some 15 ms of gaps as launches per level, 18.0 ms
// now (23.2 without the sharing of hubs; 36 with bisections in place of the
// 8-way search and the 8-wide sketch test, 29 with 64-bit ranks in place of
// their ordinals, both before it).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <vector>

#include "fl_internal.cuh"

namespace fl {

namespace {

int grid_for(int64_t items, int per_block) {
    int64_t b = (items + per_block - 1) / per_block;
    if (b < 1) b = 1;
    if (b > 152 * 32) b = 152 * 32;
    return (int)b;
}

struct WEnt {
    uint32_t ord;  // ordinal of the entry's vertex
    int32_t dist;
};

// One group of the log: vertex, its index among the vertex's groups, and the
// group's distance, entry count, counted prefix, first entry and the sketch's
// k-th ordinal, which gives the HIP weight.
struct WGroup {
    int32_t v, gidx;
    int32_t dist, cnt, counted, first;
    uint32_t kth;
};

struct WArgs {
    const int64_t* rowp;
    const int32_t* cols;
    const int32_t* wts;
    int k;
    int cap;                 // entries per vertex row
    const uint32_t* ord;     // n: ordinal of each vertex's rank
    uint32_t* S;             // n*k: sketches, ascending ordinals, kNil after
    uint8_t* Scnt;           // n
    WEnt* ent;               // n*cap
    int32_t* ecnt;           // n: entries at the start of the level (read)
    int32_t* ecnt_n;         // n: entries after the level (written by the active vertices)
    int32_t* gcnt;           // n: groups
    WGroup* glog;            // group log
    unsigned long long glog_cap;
    uint32_t* ring;          // R bitmaps of `words` words
    int64_t words;
    int R;
    const uint32_t* rev;     // nnz: the entry (v, u) paired with each entry (u, v)
    uint32_t* marks;         // R bitmaps of `mwords` words over the CSR entries
    int64_t mwords;
    unsigned* pend;          // R: nonzero when the slot has activations
    int32_t* act[2];         // active vertices of the even / odd steps (n each; hubs from the back)
    uint32_t* hub_gain;      // 32 per hub of the level: the ordinals it gained
    int32_t* hub_cnt;        // per hub of the level: their number
    int64_t n;
    struct WCtl* c;
};

// Control block of the build (device, zero at its start).
struct WCtl {
    GridBar bar;
    unsigned long long n_act[2];  // active vertices of the even / odd steps, hubs left out
    unsigned long long n_hub[2];  // active hubs
    unsigned long long glog_n;    // groups logged
    unsigned long long err;       // 1: a row overflowed; 2: a distance above 65535; 4: the group log overflowed
    long long last;               // the largest level that added groups
    long long levels;             // levels run
};

constexpr int kWLong = 32;    // longer rows are posted by the whole block (128: 22.9 ms for 21.9)
constexpr int kWQueue = 128;  // of them, queued per block and level
// Rows above are hubs.  2048: 18.4 ms for 18.0; 512 and 256, with a block per
// hub: 26 and up, a block's shared merge costs more than the warps' own.
constexpr int kWHub = 1024;

__device__ __forceinline__ WEnt load_ent(const WEnt* p) {
    const int2 x = __ldcg(reinterpret_cast<const int2*>(p));
    return WEnt{(uint32_t)x.x, x.y};
}

// Which of the gained ordinals (lane j < dcnt of the warp: the j-th) are in the
// sketch row of k, as a mask per lane (all 32 lanes call; a lane without a row
// passes NULL), and the row's k-th ordinal.  Eight are loaded at a time (as two
// 16-byte words where rows are aligned), so that a row costs one or two L2
// latencies instead of the five of a bisection.  The row may be rewritten
// meanwhile: every value read is of the old or the new sketch.
__device__ __forceinline__ unsigned held_ranks(const uint32_t* row, int k, uint32_t gained, int dcnt, uint32_t* kth) {
    unsigned held = 0;
    uint32_t last = kNil;
    for (int c = 0; c < k; c += 8) {
        uint32_t y[8];
        if ((k & 3) == 0) {
#pragma unroll
            for (int q = 0; q < 8; q += 4) {
                uint4 a = make_uint4(kNil, kNil, kNil, kNil);
                if (row && c + q < k) a = __ldcg(reinterpret_cast<const uint4*>(row + c + q));
                y[q] = a.x;
                y[q + 1] = a.y;
                y[q + 2] = a.z;
                y[q + 3] = a.w;
            }
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) y[q] = row && c + q < k ? __ldcg(&row[c + q]) : kNil;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (c + q == k - 1) last = y[q];
        for (int j = 0; j < dcnt; ++j) {
            const uint32_t x = __shfl_sync(kFull, gained, j);
            bool hit = false;
#pragma unroll
            for (int q = 0; q < 8; ++q) hit |= y[q] == x;
            if (hit) held |= 1u << j;
        }
    }
    *kth = last;
    return held;
}

// First entry of the row's `have` entries (in distance order) at distance x or
// more: eight parts per round, their bounds loaded together.
__device__ __forceinline__ int first_at(const WEnt* row, int have, int32_t x) {
    int lo = 0, hi = have;
    while (lo < hi) {
        const int part = (hi - lo + 7) >> 3;
        int below = 0;  // probes lo + part - 1, lo + 2 part - 1, ... below x (a prefix)
#pragma unroll
        for (int q = 1; q <= 7; ++q) {
            const int at = lo + q * part - 1;
            below += at < hi && load_ent(&row[at]).dist < x;
        }
        if (below < 7) hi = min(hi, lo + (below + 1) * part - 1);
        lo += below * part;
    }
    return lo;
}

// The ranks gained by v at level L (lane j < dcnt: the j-th, ascending) go to
// the entries e0 + first, + step, ... of its row (all 32 lanes call).
__device__ __forceinline__ void post_row(const WArgs& a, int64_t e0, int64_t e1, int first, int step, uint32_t gained,
                                         int dcnt, int64_t L) {
    for (int64_t b = e0 + first; b < e1; b += step) {
        const int64_t e = b + lane_id();
        const uint32_t* row = nullptr;
        int32_t u = 0;
        int64_t lv = 0;
        if (e < e1) {
            u = __ldg(&a.cols[e]);
            lv = L + __ldg(&a.wts[e]);
            if (lv > 65535) atomicOr(&a.c->err, 2ULL);
            else row = a.S + (int64_t)u * a.k;
        }
        uint32_t kth;
        const unsigned held = held_ranks(row, a.k, gained, dcnt, &kth);
        bool want = false;
        for (int j = 0; j < dcnt; ++j) {
            const uint32_t x = __shfl_sync(kFull, gained, j);
            want |= x < kth && !((held >> j) & 1u);
        }
        if (want && row) {
            const int slot = (int)((uint32_t)lv % (uint32_t)a.R);
            const uint32_t re = __ldg(&a.rev[e]);
            atomicOr(&a.marks[(int64_t)slot * a.mwords + (re >> 5)], 1u << (re & 31));
            uint32_t* word = &a.ring[(int64_t)slot * a.words + (u >> 5)];
            const uint32_t bit = 1u << (u & 31);
            if (!(__ldcg(word) & bit) && !(atomicOr(word, bit) & bit)) a.pend[slot] = 1u;
        }
    }
}

__global__ void __launch_bounds__(kResThreads, 1) k_wbuild(WArgs a) {
    __shared__ uint32_t s_gained[kWQueue][32];
    __shared__ uint32_t s_x[kResWarps][32];  // per warp: merged candidates by place
    __shared__ uint32_t s_part[kResWarps][32];  // per warp: its share of a hub's merge
    __shared__ int64_t s_e0[kWQueue], s_e1[kWQueue];
    __shared__ int s_cnt[kWQueue];
    __shared__ unsigned s_queued, s_next;
    WCtl* c = a.c;
    const Lock<32> g;
    uint32_t* sx = s_x[threadIdx.x >> 5];
    const int lane = lane_id(), k = a.k;
    const int64_t tid = (int64_t)blockIdx.x * kResThreads + threadIdx.x, threads = (int64_t)gridDim.x * kResThreads;
    // item i to warp i / gridDim of block i mod gridDim: neighbours in a list go to different blocks
    const int64_t item0 = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x, warps = threads >> 5;
    unsigned pass = 0, total = 0;
    if (threadIdx.x == 0) s_queued = 0;

    // the ranks gained at level L go to the row [e0, e1): now, or by the whole block
    auto post = [&](int64_t e0, int64_t e1, uint32_t gained, int dcnt, int64_t L) {
        if (e1 - e0 > kWLong) {
            unsigned at = 0;
            if (lane == 0) at = atomicAdd(&s_queued, 1u);
            at = __shfl_sync(kFull, at, 0);
            if (at < kWQueue) {
                s_gained[at][lane] = gained;
                if (lane == 0) {
                    s_e0[at] = e0;
                    s_e1[at] = e1;
                    s_cnt[at] = dcnt;
                }
                return;
            }
        }
        post_row(a, e0, e1, 0, 32, gained, dcnt, L);
    };
    // the queued rows, 32 entries at a time, dealt to the warps in turn
    auto post_queued = [&](int64_t L) {
        __syncthreads();
        const int queued = (int)min(s_queued, (unsigned)kWQueue);
        int dealt = 0;
        for (int q = 0; q < queued; ++q) {
            const int64_t e0 = s_e0[q], e1 = s_e1[q];
            const int first = (int)((threadIdx.x >> 5) - (unsigned)dealt) & (kResWarps - 1);
            post_row(a, e0, e1, 32 * first, kResThreads, s_gained[q][lane], s_cnt[q], L);
            dealt += (int)((e1 - e0 + 31) >> 5);
        }
        __syncthreads();
        if (threadIdx.x == 0) s_queued = 0;
    };

    // level 0: every vertex's own rank
    for (int64_t i = tid; i < a.n * k; i += threads) a.S[i] = i % k == 0 ? a.ord[i / k] : kNil;
    for (int64_t v = tid; v < a.n; v += threads) {
        a.ent[v * a.cap] = WEnt{a.ord[v], 0};
        a.Scnt[v] = 1;
        a.ecnt[v] = 1;
        a.gcnt[v] = 1;
        WGroup gr;
        gr.v = (int32_t)v;
        gr.gidx = 0;
        gr.dist = 0;
        gr.cnt = 1;
        gr.counted = 1;
        gr.first = 0;
        gr.kth = kNil;  // a ball of one vertex (k >= 2)
        a.glog[v] = gr;
    }
    if (tid == 0) c->glog_n = (unsigned long long)a.n;
    if (!end_pass(&c->bar, pass, 0, &total)) return;
    for (int64_t v = item0; v < a.n; v += warps)
        post(__ldg(&a.rowp[v]), __ldg(&a.rowp[v + 1]), lane == 0 ? a.ord[v] : kNil, 1, 0);
    post_queued(0);
    if (!end_pass(&c->bar, pass, 0, &total)) return;

    int64_t L = 0, n_prev = 0, hub_prev = 0;
    for (unsigned step = 0;; ++step) {
        // the next level with activations
        if (threadIdx.x == 0) s_next = ~0u;
        __syncthreads();
        for (int d = 1 + threadIdx.x; d <= a.R; d += kResThreads)
            if (__ldcg(&a.pend[(uint32_t)(L + d) % (uint32_t)a.R])) {
                atomicMin(&s_next, (unsigned)d);
                break;
            }
        __syncthreads();
        const int par = (int)(step & 1);
        // the level before: its new row counts become current
        for (int64_t i = tid; i < n_prev; i += threads) {
            const int32_t v = __ldcg(&a.act[par ^ 1][i < hub_prev ? a.n - 1 - i : i - hub_prev]);
            a.ecnt[v] = __ldcg(&a.ecnt_n[v]);
        }
        if (s_next == ~0u) break;
        L += s_next;
        const int slot = (int)((uint32_t)L % (uint32_t)a.R);
        unsigned mine = 0;
        uint32_t* bm = a.ring + (int64_t)slot * a.words;
        for (int64_t w = tid >> 5; w < a.words; w += warps) {
            const uint32_t word = __ldcg(&bm[w]);
            if (!word) continue;
            const bool in = (word >> lane) & 1u;
            const int64_t v = w * 32 + lane;
            const bool hub = in && __ldg(&a.rowp[v + 1]) - __ldg(&a.rowp[v]) > kWHub;
            const long long at = warp_append(in && !hub, &c->n_act[par]);
            if (in && !hub) a.act[par][at] = (int32_t)v;
            if (__any_sync(kFull, hub)) {
                const long long ah = warp_append(hub, &c->n_hub[par]);
                if (hub) a.act[par][a.n - 1 - ah] = (int32_t)v;
            }
            mine += in;
            if (lane == 0) bm[w] = 0u;
        }
        if (!end_pass(&c->bar, pass, mine, &total)) return;
        n_prev = (int64_t)total;
        hub_prev = (int64_t)__ldcg(&c->n_hub[par]);
        if (tid == 0) {
            c->n_act[par ^ 1] = 0;
            c->n_hub[par ^ 1] = 0;
            a.pend[slot] = 0;  // no post of this level targets its own slot
            ++c->levels;
        }
        // Items [0, hub_prev) are the hubs; up to one per block, a block merges
        // its hub before its other items.
        const int64_t by_block = hub_prev <= (int64_t)gridDim.x ? hub_prev : 0;
        int64_t i = blockIdx.x < by_block ? blockIdx.x : by_block + item0;
        for (int64_t next; i < n_prev; i = next) {
            const bool shared = i < by_block, hub = i < hub_prev;
            next = shared ? by_block + item0 : i + warps;
            const int32_t v = __ldcg(&a.act[par][hub ? a.n - 1 - i : i - hub_prev]);
            const uint32_t s_old = lane < k ? __ldcg(&a.S[(int64_t)v * k + lane]) : kNil;
            const int64_t e0 = __ldg(&a.rowp[v]), e1 = __ldg(&a.rowp[v + 1]);
            Sketch<32> s;
            s.sk = s_old;
            s.tau_base = kNil;
            s.retau(g, k);
            uint32_t* mk = a.marks + (int64_t)slot * a.mwords;
            const int64_t w1 = (e1 + 31) >> 5;
            // the row's marks, 32 words at once (four per warp where the block shares
            // the row): their set bits inside [e0, e1) are the delivering entries
            const int span = shared ? 4 : 32;
            for (int64_t wb = (e0 >> 5) + (shared ? 4 * (threadIdx.x >> 5) : 0); wb < w1;
                 wb += shared ? 4 * kResWarps : 32) {
                const int64_t wi = wb + lane;
                uint32_t bits = 0;
                if (lane < span && wi < w1) {
                    bits = __ldcg(&mk[wi]);
                    const int64_t first = wi << 5;
                    uint32_t mask = ~0u;
                    if (first < e0) mask &= ~0u << (int)(e0 - first);
                    if (e1 - first < 32) mask &= (1u << (int)(e1 - first)) - 1u;
                    bits &= mask;
                    if (bits) {  // read: the slot serves level L + R next
                        if (mask == ~0u) mk[wi] = 0u;
                        else atomicAnd(&mk[wi], ~bits);
                    }
                }
                const int mine_n = __popc(bits);
                const int incl = warp_incl_scan(mine_n);
                const int n_del = __shfl_sync(kFull, incl, 31);
                for (int cb = 0; cb < n_del; cb += 32) {
                    const int j = cb + lane;
                    // the word that holds the j-th set bit: the words whose bits all come before it
                    int wl = 0;
#pragma unroll
                    for (int st = 16; st > 0; st >>= 1)
                        if (__shfl_sync(kFull, incl, wl + st - 1) <= j) wl += st;
                    const uint32_t word = __shfl_sync(kFull, bits, wl);
                    const int before = __shfl_sync(kFull, incl - mine_n, wl);
                    const WEnt* row = nullptr;
                    int32_t at = 0, have = 0, x = 0;
                    if (j < n_del) {
                        const int64_t e = ((wb + wl) << 5) + nth_set_bit(word, j - before);
                        const int32_t u = __ldg(&a.cols[e]);
                        x = (int32_t)(L - __ldg(&a.wts[e]));
                        have = min(__ldcg(&a.ecnt[u]), a.cap);
                        row = a.ent + (int64_t)u * a.cap;
                        at = first_at(row, have, x);
                    }
                    // each lane offers its entry's candidates one per round
                    for (;;) {
                        uint32_t r = kNil;
                        if (at < have) {
                            const WEnt en = load_ent(&row[at]);
                            ++at;
                            if (en.dist == x) r = en.ord;
                            else at = have;
                        }
                        if (!__any_sync(kFull, r != kNil)) break;
                        absorb(g, k, r, s, sx);
                    }
                }
            }
            if (shared) {
                s_part[threadIdx.x >> 5][lane] = s.sk;
                __syncthreads();
                if (threadIdx.x >= 32) continue;
                for (int w = 1; w < kResWarps; ++w) merge_list(g, k, s_part[w][lane], s, sx);
            }
            // the entries gained at distance L: in the new sketch, not in the old
            // (every lane takes part in the membership shuffles)
            bool held;
            lock_find(g, s_old, s.sk, held);
            const bool fresh = s.sk != kNil && !held;
            const int cnt = __popc(__ballot_sync(kFull, s.sk != kNil));
            const uint32_t kth = __shfl_sync(kFull, s.sk, k - 1);
            const unsigned fm = __ballot_sync(kFull, fresh);
            const int32_t base = __ldcg(&a.ecnt[v]);
            const int dcnt = __popc(fm);
            if (!fm || base + dcnt > a.cap) {
                if (lane == 0) {
                    a.ecnt_n[v] = base;
                    if (fm) atomicOr(&c->err, 1ULL);
                    if (hub) a.hub_cnt[i] = 0;
                }
                continue;
            }
            const int counted = __popc(fm & (cnt < k ? kFull : ((1u << (k - 1)) - 1u)));
            if (fresh) {
                const int at = base + __popc(fm & ((1u << lane) - 1u));
                a.ent[(int64_t)v * a.cap + at] = WEnt{s.sk, (int32_t)L};
            }
            if (lane < k) a.S[(int64_t)v * k + lane] = s.sk;
            if (lane == 0) {
                a.ecnt_n[v] = base + dcnt;
                a.Scnt[v] = (uint8_t)cnt;
                c->last = L;
                const unsigned long long gi = atomicAdd(&c->glog_n, 1ULL);
                if (gi < a.glog_cap) {
                    WGroup gr;
                    gr.v = v;
                    gr.gidx = __ldcg(&a.gcnt[v]);
                    gr.dist = (int32_t)L;
                    gr.cnt = dcnt;
                    gr.counted = counted;
                    gr.first = base;
                    gr.kth = kth;
                    a.glog[gi] = gr;
                    a.gcnt[v] = gr.gidx + 1;
                } else {
                    atomicOr(&c->err, 4ULL);
                }
            }
            const uint32_t mine_g = __shfl_sync(kFull, s.sk, lane < dcnt ? nth_set_bit(fm, lane) : 0);
            if (hub) {
                a.hub_gain[i * 32 + lane] = lane < dcnt ? mine_g : kNil;
                if (lane == 0) a.hub_cnt[i] = dcnt;
            } else {
                post(e0, e1, lane < dcnt ? mine_g : kNil, dcnt, L);
            }
        }
        post_queued(L);
        if (!end_pass(&c->bar, pass, 0, &total)) return;
        if (hub_prev == 0) continue;
        // the hubs' rows, 32 entries at a time, dealt to the grid's warps in turn
        unsigned dealt = 0;  // mod the number of warps
        for (int64_t h0 = 0; h0 < hub_prev; h0 += 32) {
            int64_t e0 = 0, e1 = 0;
            int dcnt = 0;
            if (h0 + lane < hub_prev) {
                const int32_t v = __ldcg(&a.act[par][a.n - 1 - (h0 + lane)]);
                dcnt = __ldcg(&a.hub_cnt[h0 + lane]);
                e0 = __ldg(&a.rowp[v]);
                e1 = __ldg(&a.rowp[v + 1]);
            }
            for (unsigned m = __ballot_sync(kFull, dcnt > 0); m; m &= m - 1) {
                const int l = __ffs(m) - 1;
                const int64_t b0 = __shfl_sync(kFull, e0, l), b1 = __shfl_sync(kFull, e1, l);
                const unsigned chunks = (unsigned)((b1 - b0 + 31) >> 5);
                // the first of the row's chunks that is this warp's
                const unsigned turn = (unsigned)item0 + ((unsigned)item0 < dealt ? (unsigned)warps : 0u) - dealt;
                dealt += chunks;
                if (dealt >= (unsigned)warps) dealt %= (unsigned)warps;
                if (turn >= chunks) continue;
                post_row(a, b0 + 32 * (int64_t)turn, b1, 0, (int)(32 * warps), __ldcg(&a.hub_gain[(h0 + l) * 32 + lane]),
                         __shfl_sync(kFull, dcnt, l), L);
            }
        }
        if (!end_pass(&c->bar, pass, 0, &total)) return;
    }
}

// Vertex-major ADS from the group log and the rows.
__global__ void k_wgroups(const WGroup* __restrict__ glog, int64_t m, int k, uint64_t seed,
                          const int32_t* __restrict__ ord_rid, const int64_t* __restrict__ gofs,
                          uint32_t* __restrict__ ginfo, double* __restrict__ gwt) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) {
        const WGroup gr = glog[i];
        const int64_t at = gofs[gr.v] + gr.gidx;
        ginfo[at] = (uint32_t)gr.dist | ((uint32_t)gr.cnt << 16) | ((uint32_t)gr.counted << 24);
        gwt[at] = gr.kth == kNil ? 1.0 : hip_weight(k, k, vertex_rank(seed, (int64_t)ord_rid[gr.kth]));
    }
}

__global__ void k_wentries(const WEnt* __restrict__ ent, int cap, const int32_t* __restrict__ ecnt,
                           const int64_t* __restrict__ eofs, const int32_t* __restrict__ ord_rid, int64_t n,
                           int32_t* __restrict__ eid) {
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += warps)
        for (int j = lane_id(); j < ecnt[v]; j += 32) eid[eofs[v] + j] = ord_rid[ent[v * cap + j].ord];
}

__global__ void k_wmaxlen(const int32_t* __restrict__ w, int64_t nnz, unsigned long long* __restrict__ out,
                          unsigned long long* __restrict__ bad) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned mx = 0;
    bool neg = false;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz; e += stride) {
        const int32_t x = w[e];
        neg |= x < 1;
        mx = max(mx, (unsigned)max(x, 0));
    }
    mx = __reduce_max_sync(kFull, mx);
    if (lane_id() == 0) atomicMax(out, (unsigned long long)mx);
    if (__any_sync(kFull, neg) && lane_id() == 0) atomicOr(bad, 1ULL);
}

// Pairing keys of the CSR entries: (min(u, v), max(u, v)) and (length,
// direction), the entry index as payload (a warp per source vertex u).
__global__ void k_wrevkeys(const int64_t* __restrict__ rowp, const int32_t* __restrict__ cols,
                           const int32_t* __restrict__ wts, int64_t n, uint64_t* __restrict__ hi,
                           uint32_t* __restrict__ lo, uint32_t* __restrict__ val) {
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < n; u += warps) {
        for (int64_t e = rowp[u] + lane_id(); e < rowp[u + 1]; e += 32) {
            const int64_t v = cols[e];
            const uint64_t a = (uint64_t)(u < v ? u : v), b = (uint64_t)(u < v ? v : u);
            hi[e] = (a << 32) | b;
            lo[e] = ((uint32_t)wts[e] << 1) | (u > v ? 1u : 0u);
            val[e] = (uint32_t)e;
        }
    }
}

// out[i] = in[at[i]]
template <class T>
__global__ void k_wgather(const T* __restrict__ in, const uint32_t* __restrict__ at, int64_t m, T* __restrict__ out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) out[i] = in[at[i]];
}

// First index of the sorted keys at or above (h, l).
__device__ __forceinline__ int64_t key_lower_bound(const uint64_t* __restrict__ hi, const uint32_t* __restrict__ lo,
                                                   int64_t m, uint64_t h, uint32_t l) {
    int64_t a = 0, b = m;
    while (a < b) {
        const int64_t mid = (a + b) >> 1;
        const uint64_t x = hi[mid];
        if (x < h || (x == h && lo[mid] < l)) a = mid + 1;
        else b = mid;
    }
    return a;
}

// After the sort, the entries of one edge and length form a group whose
// first half runs min -> max and second half max -> min; the i-th of each
// half pair up (a self-loop pairs with itself).  A group whose halves differ
// means a length that is not the same in both directions (bad = 1).
__global__ void k_wpair(const uint64_t* __restrict__ hi, const uint32_t* __restrict__ lo,
                        const uint32_t* __restrict__ val, int64_t m, uint32_t* __restrict__ rev,
                        unsigned long long* __restrict__ bad) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) {
        const uint64_t h = hi[i];
        const uint32_t l = lo[i];
        if ((h >> 32) == (h & 0xffffffffULL)) {
            rev[val[i]] = val[i];
            continue;
        }
        const uint32_t l0 = l & ~1u;  // the group: keys (h, l0) and (h, l0 | 1)
        const int64_t g0 = key_lower_bound(hi, lo, m, h, l0);
        const int64_t g1 = key_lower_bound(hi, lo, m, h, l0 + 2);
        const int64_t half = (g1 - g0) >> 1;
        if (((g1 - g0) & 1) || half < 1 || lo[g0 + half - 1] != l0 || lo[g0 + half] != (l0 | 1u)) {
            atomicOr(bad, 1ULL);
            continue;
        }
        if (l & 1u) continue;  // the second half is written by its partners
        const int64_t j = i + half;
        rev[val[i]] = val[j];
        rev[val[j]] = val[i];
    }
}

}  // namespace

// For every CSR entry (u, v) of a weighted graph, an entry (v, u) of the same
// length, paired one to one (duplicates pair in order): the weighted build
// marks the paired entry of v's row when u gains entries.  FL_EINVAL when an
// edge's lengths differ between its two directions.
int pair_reverse_edges(fl_graph* g) {
    const int64_t n = g->n, nnz = g->nnz;
    cudaStream_t st = g->stream;
    if (nnz >= (1LL << 32)) FL_FAIL(FL_EINVAL, "a weighted graph holds fewer than 2^32 CSR entries");
    FL_TRY(dalloc(g->wrev, (size_t)std::max<int64_t>(nnz, 1) * 4));
    if (nnz == 0) return FL_OK;
    DBuf hi, lo, val, flag;
    int rc = FL_OK;
    do {
        if ((rc = dalloc(hi, (size_t)nnz * 16)) || (rc = dalloc(lo, (size_t)nnz * 8)) ||
            (rc = dalloc(val, (size_t)nnz * 8)) || (rc = dalloc(flag, 16)))
            break;
        cudaError_t e = cudaMemsetAsync(flag.p, 0, 16, st);
        if (e != cudaSuccess) { rc = status_of(e, "edge pairing", __FILE__, __LINE__); break; }
        SortPairs<uint64_t> sh;
        SortPairs<uint32_t> sl;
        for (int q = 0; q < 2; ++q) {
            sh.key[q] = hi.as<uint64_t>() + q * nnz;
            sl.key[q] = lo.as<uint32_t>() + q * nnz;
            sh.val[q] = sl.val[q] = val.as<uint32_t>() + q * nnz;
        }
        unsigned long long* bad = flag.as<unsigned long long>();
        const uint64_t* hi_of = sh.key[1];  // keys by entry
        FL_LAUNCH(kProfOther, k_wrevkeys<<<grid_for(n * 32, 256), 256, 0, st>>>(
                                  g->rowp.as<int64_t>(), g->cols.as<int32_t>(), g->wts.as<int32_t>(), n,
                                  sh.key[1], sl.key[0], sl.val[0]));
        // the bits that can vary: ids below n in both halves of hi, the
        // length and the direction bit in lo; lo's digits first, then hi's
        int nb = 1, wb = 1, shift[kSortDigits];
        while (nb < 31 && (1LL << nb) < n) ++nb;
        while (wb < 17 && (1 << wb) <= g->max_w) ++wb;
        if ((rc = sort_pairs(sl, nnz, shift, digit_windows((2ULL << wb) - 1, 0, shift), st, g->scratch, kProfOther,
                             bad)))
            break;
        sh.cur = 0;
        if (sl.cur == 1) {  // the payload goes with the first key buffer
            std::swap(sh.val[0], sh.val[1]);
        }
        FL_LAUNCH(kProfOther, k_wgather<<<grid_for(nnz, 256), 256, 0, st>>>(hi_of, sh.val[0], nnz, sh.key[0]));
        int nd = 0;
        for (int half = 0; half < 2; ++half)
            for (int b = 0; b < nb; b += 8) shift[nd++] = 32 * half + b;
        if ((rc = sort_pairs(sh, nnz, shift, nd, st, g->scratch, kProfOther, bad))) break;
        // lo in the sorted order, recomputed from the entries in a free buffer
        const uint32_t* perm = sh.val[sh.cur];
        uint32_t* lo_by_entry = sl.key[0];
        uint32_t* lo_sorted = sl.key[1];
        FL_LAUNCH(kProfOther, k_wrevkeys<<<grid_for(n * 32, 256), 256, 0, st>>>(
                                  g->rowp.as<int64_t>(), g->cols.as<int32_t>(), g->wts.as<int32_t>(), n,
                                  sh.key[sh.cur ^ 1], lo_by_entry, sh.val[sh.cur ^ 1]));
        FL_LAUNCH(kProfOther, k_wgather<<<grid_for(nnz, 256), 256, 0, st>>>(lo_by_entry, perm, nnz, lo_sorted));
        FL_LAUNCH(kProfOther, k_wpair<<<grid_for(nnz, 256), 256, 0, st>>>(sh.key[sh.cur], lo_sorted, perm, nnz,
                                                                          g->wrev.as<uint32_t>(), bad));
        unsigned long long h = 0;
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(&h, flag.p, 8, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) { rc = status_of(e, "edge pairing", __FILE__, __LINE__); break; }
        if (h & kSortError) {
            rc = FL_ETIMEOUT;
            set_error(rc, "edge pairing: a sort's wait ran out");
        } else if (h) {
            rc = FL_EINVAL;
            set_error(rc, "an edge's length must be the same in both directions");
        }
    } while (0);
    dfree_after(st, {&hi, &lo, &val, &flag});
    return rc;
}

int check_weights(fl_graph* g) {
    cudaStream_t st = g->stream;
    DBuf tmp;
    FL_TRY(dalloc(tmp, 16));
    unsigned long long* d = tmp.as<unsigned long long>();
    FL_CUDA(cudaMemsetAsync(d, 0, 16, st));
    if (g->nnz > 0)
        FL_LAUNCH(kProfOther, k_wmaxlen<<<grid_for(g->nnz, 256), 256, 0, st>>>(g->wts.as<int32_t>(), g->nnz, d, d + 1));
    unsigned long long h[2] = {0, 0};
    FL_CUDA(cudaMemcpyAsync(h, d, 16, cudaMemcpyDeviceToHost, st));
    FL_CUDA(cudaStreamSynchronize(st));
    dfree_after(st, {&tmp});
    if (h[1]) FL_FAIL(FL_EINVAL, "edge lengths must be positive integers");
    if (h[0] > 65535) FL_FAIL(FL_EINVAL, "edge lengths must be at most 65535");
    g->max_w = (int)h[0];
    return FL_OK;
}

int build_sketches_weighted(fl_graph* g, int k, uint64_t seed) {
    const int64_t n = g->n, nnz = g->nnz;
    cudaStream_t st = g->stream;
    const int R = g->max_w + 1;
    const int64_t words = (n + 31) / 32;
    // entries per vertex: about k (1 + ln(n / k)) expected; twice that plus a
    // margin, at most n; doubled and rebuilt on overflow
    const double expect = (double)k * (1.0 + std::log(std::max(1.0, (double)n / k)));
    int64_t cap = std::min<int64_t>(n, (int64_t)(2.0 * expect) + 64);
    const int64_t mwords = (nnz + 31) / 32;
    const int64_t hubs_max = nnz / kWHub + 1;
    DBuf ent, ecnt, ecnt_n, gcnt, glog, ring, pend, act, cnt, marks, hubs;
    int rc = FL_OK;
    FL_CUDA(cudaMemsetAsync(g->ctr.p, 0, sizeof(Counters), st));
    if ((rc = build_ordinals(g, ent)) || (rc = read_counters(g))) {
        dfree_after(st, {&ent});
        return rc;
    }
    if (g->h_ctr->error & kSortError) {
        dfree_after(st, {&ent});
        FL_FAIL(FL_ETIMEOUT, "ordinals: a sort's wait ran out");
    }
    for (;;) {
        const unsigned long long glog_cap = (unsigned long long)n * (unsigned long long)cap;
        if ((rc = dalloc(g->S, (size_t)n * k * 4)) || (rc = dalloc(g->Scnt, (size_t)n)) ||
            (rc = dalloc(ent, (size_t)n * cap * sizeof(WEnt))) || (rc = dalloc(ecnt, (size_t)n * 4)) ||
            (rc = dalloc(ecnt_n, (size_t)n * 4)) ||
            (rc = dalloc(gcnt, (size_t)n * 4)) ||
            (rc = dalloc(glog, (size_t)glog_cap * sizeof(WGroup))) ||
            (rc = dalloc(ring, (size_t)R * words * 4 + 16)) || (rc = dalloc(pend, (size_t)R * 4)) ||
            (rc = dalloc(act, (size_t)n * 8)) || (rc = dalloc(hubs, (size_t)hubs_max * 33 * 4)) || (rc = dalloc(cnt, sizeof(WCtl))) ||
            (rc = dalloc(marks, (size_t)R * mwords * 4 + 16)))
            break;
        WArgs a;
        a.rowp = g->rowp.as<int64_t>();
        a.cols = g->cols.as<int32_t>();
        a.wts = g->wts.as<int32_t>();
        a.k = k;
        a.cap = (int)cap;
        a.ord = g->ord.as<uint32_t>();
        a.S = g->S.as<uint32_t>();
        a.Scnt = g->Scnt.as<uint8_t>();
        a.ent = ent.as<WEnt>();
        a.ecnt = ecnt.as<int32_t>();
        a.ecnt_n = ecnt_n.as<int32_t>();
        a.gcnt = gcnt.as<int32_t>();
        a.glog = glog.as<WGroup>();
        a.glog_cap = glog_cap;
        a.ring = ring.as<uint32_t>();
        a.words = words;
        a.R = R;
        a.pend = pend.as<unsigned>();
        a.act[0] = act.as<int32_t>();
        a.act[1] = a.act[0] + n;
        a.hub_gain = hubs.as<uint32_t>();
        a.hub_cnt = hubs.as<int32_t>() + hubs_max * 32;
        a.n = n;
        a.c = cnt.as<WCtl>();
        a.rev = g->wrev.as<uint32_t>();
        a.marks = marks.as<uint32_t>();
        a.mwords = mwords;
        cudaError_t e = cudaMemsetAsync(ring.p, 0, (size_t)R * words * 4, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(marks.p, 0, (size_t)R * mwords * 4, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(pend.p, 0, (size_t)R * 4, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(cnt.p, 0, sizeof(WCtl), st);
        if (e != cudaSuccess) { rc = status_of(e, "weighted build", __FILE__, __LINE__); break; }
        int dev = 0, sms = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) {
            const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(sms, (n + 31) / 32));
            void* args[] = {&a};
            FL_LAUNCH(kProfSketchMerge, e = cudaLaunchCooperativeKernel((const void*)k_wbuild, dim3(blocks),
                                                                        dim3(kResThreads), args, 0, st));
        }
        WCtl hc{};
        if (e == cudaSuccess) e = cudaMemcpyAsync(&hc, cnt.p, sizeof(WCtl), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) { rc = status_of(e, "weighted build", __FILE__, __LINE__); break; }
        if (hc.bar.err) { rc = FL_ETIMEOUT; set_error(rc, "weighted build: a barrier wait ran out"); break; }
        if (hc.err & 2ULL) { rc = FL_EINVAL; set_error(rc, "a distance above 65535"); break; }
        if ((hc.err & 5ULL) && cap < n) {  // a row overflowed: twice the capacity
            cap = std::min<int64_t>(n, cap * 2);
            continue;
        }
        if (hc.err) { rc = FL_ECUDA; set_error(rc, "weighted build: inconsistent row capacity"); break; }
        // vertex-major ADS
        const int64_t m = (int64_t)hc.glog_n;
        if ((rc = dalloc(g->gofs, (size_t)(n + 1) * 8)) || (rc = dalloc(g->eofs, (size_t)(n + 1) * 8))) break;
        if ((rc = scan_exclusive_i32_to_i64(gcnt.as<int32_t>(), g->gofs.as<int64_t>(), n, st, g->scratch)) ||
            (rc = scan_exclusive_i32_to_i64(ecnt.as<int32_t>(), g->eofs.as<int64_t>(), n, st, g->scratch)))
            break;
        int64_t ne = 0;
        int64_t tail_g = 0, tail_e = 0;
        e = cudaMemcpyAsync(&tail_g, g->gofs.as<int64_t>() + n - 1, 8, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&tail_e, g->eofs.as<int64_t>() + n - 1, 8, cudaMemcpyDeviceToHost, st);
        int32_t lg = 0, le = 0;
        if (e == cudaSuccess) e = cudaMemcpyAsync(&lg, gcnt.as<int32_t>() + n - 1, 4, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&le, ecnt.as<int32_t>() + n - 1, 4, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) { rc = status_of(e, "weighted build", __FILE__, __LINE__); break; }
        g->n_groups = tail_g + lg;
        ne = tail_e + le;
        g->n_entries = ne;
        if (g->n_groups != m) { rc = FL_ECUDA; set_error(rc, "weighted build: group log and counts disagree"); break; }
        e = cudaMemcpyAsync(g->gofs.as<int64_t>() + n, &g->n_groups, 8, cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(g->eofs.as<int64_t>() + n, &g->n_entries, 8, cudaMemcpyHostToDevice, st);
        if (e != cudaSuccess) { rc = status_of(e, "weighted build", __FILE__, __LINE__); break; }
        if ((rc = dalloc(g->ginfo, (size_t)std::max<int64_t>(m, 1) * 4)) ||
            (rc = dalloc(g->gwt, (size_t)std::max<int64_t>(m, 1) * 8)) ||
            (rc = dalloc(g->eid, (size_t)std::max<int64_t>(ne, 1) * 4)))
            break;
        FL_LAUNCH(kProfSketchOther, k_wgroups<<<grid_for(m, 256), 256, 0, st>>>(
                                        glog.as<WGroup>(), m, k, seed, g->ord_rid.as<int32_t>(),
                                        g->gofs.as<int64_t>(), g->ginfo.as<uint32_t>(), g->gwt.as<double>()));
        FL_LAUNCH(kProfSketchOther, k_wentries<<<grid_for(n, 8), 256, 0, st>>>(
                                        ent.as<WEnt>(), (int)cap, ecnt.as<int32_t>(), g->eofs.as<int64_t>(),
                                        g->ord_rid.as<int32_t>(), n, g->eid.as<int32_t>()));
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) { rc = status_of(e, "weighted build", __FILE__, __LINE__); break; }
        g->hops = hc.last;
        g->edge_merges = 0;
        g->wlevels = hc.levels;
        break;
    }
    dfree_after(st, {&ent, &ecnt, &ecnt_n, &gcnt, &glog, &ring, &pend, &act, &cnt, &marks, &hubs});
    return rc;
}

}  // namespace fl

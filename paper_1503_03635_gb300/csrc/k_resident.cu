// k_resident.cu -- the greedy MIS and the multi-source BFS of a small graph,
// each as one resident kernel.
//
// A round of a sweep on a graph of up to some million CSR entries takes a few
// microseconds of device time, less than its launches and the host's look at
// the frontier (30-60 us a round).  Here the whole loop runs on the device: a
// cooperative launch of at most one block per SM, a grid barrier per round.
//
// Work items: every row is cut into items of at most kItemEdges entries (at
// least one item per vertex), eight lanes each, so that no warp carries a
// hub.  A round is a pull over the items (the BFS also pushes thin frontiers): X'[v] = min(X[v], min over the row
// of X[u]) with two value buffers.  A row of several items lowers X'[v] with
// atomicMin; X'[v] then still holds the value of two rounds ago, which is at
// least X[v] (values only fall within a sweep), so it needs no reset.
//
// Greedy rounds shrink: a vertex that no undecided facility's ball reached in
// one round's cover is in no later ball (the undecided facilities only get
// fewer), so each cover leaves the item list of the next round, and the
// gather and kill sweeps of the same round run on that list too (a shortest
// path from a client of a ball to its facility stays inside the ball).
//
// Barrier waits are bounded: past the limit the kernel sets an error flag and
// returns.
#include <algorithm>
#include <vector>

#include "fl_internal.cuh"

namespace fl {

namespace {

constexpr uint32_t kNone = 0xffffffffu;
constexpr uint64_t kDone = ~0ULL;           // fk of a vertex that is no undecided facility
constexpr int kMaxBall = 1023;              // larger ball radii take the host-driven rounds (kNarrowBall on large graphs)
constexpr int kRoundsPerLaunch = 32;        // greedy rounds (bounds the log)
constexpr int kFastRows = 128;              // log rows copied with the control block

// Control block of a launch (device).
struct Ctl {
    GridBar bar;                      // its err: 1: a barrier wait ran out; 2: a ball without clients; 4: the level cap
    unsigned deep;                    // 1: a ball radius above max_ball (nothing was done)
    unsigned n_list[2];               // items of the current / next greedy round
    unsigned tmax[2];                 // largest ball radius of the undecided, by round parity
    unsigned hist[2][kMaxBall + 1];   // undecided facilities by ball radius, by round parity
    long long rounds, n_u, n_open, log_n;
    long long done;                   // 1: the launch ran to its end
    unsigned long long bfs_n[4];      // BFS: lengths of the frontier lists (level mod 4)
};

struct ItemGraph {
    const int32_t* __restrict__ cols;
    int64_t n;
};

// Smallest x(u) over the item's entries, by eight lanes (all 32 lanes call).
template <class F>
__device__ __forceinline__ uint32_t item_min(const ItemGraph& g, int32_t beg, int32_t end, F x) {
    const int sub = lane_id() & 7;
    uint32_t m = kNone;
    for (int32_t e = beg + sub; e < end; e += 32) {
        int32_t u[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) u[j] = e + 8 * j < end ? __ldg(&g.cols[e + 8 * j]) : -1;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (u[j] >= 0) m = min(m, x(u[j]));
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) m = min(m, __shfl_xor_sync(kFull, m, o));
    return m;
}

// An item as stored: vertex, first and last + 1 entry, kFirst for the row's
// first item and kSingle for its only one.
constexpr int kFirst = 1, kSingle = 2;

__device__ __forceinline__ int4 load_item(const int4* list, int64_t i, int64_t n_list) {
    return i < n_list ? __ldcg(&list[i]) : make_int4(-1, 0, 0, 0);
}

// The item of a lane's group with its entries' columns in registers: when every
// item of a list has its own group of lanes, the passes over the list load
// them once (a pass was a chain of three dependent loads, item, column, value,
// and a barrier: 10^4 vertices 369 -> 353 us, 56 small selections on 65 k
// vertices 6 % of the whole call).
struct Held {
    bool on;             // the list has at most one item per group
    int4 it;
    int32_t u[kItemEdges / 8];
};

__device__ __forceinline__ void hold(Held& h, const ItemGraph& g, const int4* list, int64_t n, int64_t warp0,
                                     int64_t warps) {
    h.on = n <= warps * 4;
    if (!h.on) return;
    h.it = load_item(list, warp0 * 4 + (lane_id() >> 3), n);
#pragma unroll
    for (int j = 0; j < kItemEdges / 8; ++j) {
        const int32_t e = h.it.y + (lane_id() & 7) + 8 * j;
        h.u[j] = e < h.it.z ? __ldg(&g.cols[e]) : -1;
    }
}

// Calls body(item, min) for this warp's items of a list; min(want, x) is the
// smallest x(u) over the item's entries (kNone where want is false).
template <class B>
__device__ __forceinline__ void for_items(const Held& h, const ItemGraph& g, const int4* list, int64_t n,
                                          int64_t warp0, int64_t warps, B body) {
    if (h.on) {
        if (warp0 * 4 >= n) return;
        body(h.it, [&](bool want, auto x) {
            uint32_t m = kNone;
#pragma unroll
            for (int j = 0; j < kItemEdges / 8; ++j)
                if (want && h.u[j] >= 0) m = min(m, x(h.u[j]));
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) m = min(m, __shfl_xor_sync(kFull, m, o));
            return m;
        });
        return;
    }
    for (int64_t b = warp0 * 4; b < n; b += warps * 4) {
        const int4 it = load_item(list, b + (lane_id() >> 3), n);
        body(it, [&](bool want, auto x) { return item_min(g, it.y, want ? it.z : it.y, x); });
    }
}

struct MisArgs {
    ItemGraph g;
    const int4* items;      // every item
    int64_t n_items;
    uint32_t* X[2];         // cover values
    uint32_t* Y[2];         // gather values
    uint32_t* kr;           // kill marks: 1 + distance to a client claimed in this round
    unsigned long long* fk; // undecided facility: ball radius << 32 | ordinal, else kDone
    int4* list[2];
    const uint32_t* ord;      // read at the start only (kept in fk)
    const int32_t* fac_by_ord;
    const int32_t* bcap;
    uint8_t* state;         // in: 0 candidate, 3 other; out: 1 open, 2 closed
    const uint8_t* client;
    uint8_t* claimed;
    uint8_t* open;
    int32_t* open_list;
    Ctl* c;
    long long* log;         // rows of 6
    long long log_cap;
    long long m;            // candidates
    int max_ball;           // largest ball radius that the kernel takes
    int resume;             // 0: first launch; 1: goes on after kRoundsPerLaunch rounds
};

__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// One row of the log, by one thread that keeps the number of rows in a register
// (the grid waits for it at the next barrier: a counter in memory, and the
// buckets read one after the other, were 15 of a 39 us greedy round at 10^4
// vertices).
__device__ __forceinline__ void log_row(const MisArgs& a, long long at, long long rd, int kind, long long step,
                                        long long front, long long pulled, unsigned long long ns) {
    if (at >= a.log_cap) return;
    long long* r = a.log + at * 6;
    r[0] = rd;
    r[1] = kind;
    r[2] = step;
    r[3] = front;
    r[4] = pulled;
    r[5] = (long long)(ns / 1000);
}

__global__ void __launch_bounds__(kResThreads, 1) k_mis_resident(MisArgs a) {
    __shared__ unsigned s_hist[kMaxBall + 1];
    __shared__ unsigned s_t;
    Ctl* c = a.c;
    const int lane = lane_id();
    const int64_t warp0 = ((int64_t)blockIdx.x * kResThreads + threadIdx.x) >> 5;
    const int64_t warps = (int64_t)gridDim.x * kResWarps;
    const bool scribe = blockIdx.x == 0 && threadIdx.x == 0;
    const bool scribes = blockIdx.x == 0 && threadIdx.x < 32;  // the scribe's warp keeps the count
    long long log_n = 0;
    unsigned pass = 0, total = 0;

    // Undecided facilities by ball radius: block counts, then the grid's.
    auto hist_begin = [&]() {
        for (int i = threadIdx.x; i <= kMaxBall; i += kResThreads) s_hist[i] = 0;
        if (threadIdx.x == 0) s_t = 0;
        __syncthreads();
    };
    auto hist_add = [&](unsigned b) {
        const unsigned same = __match_any_sync(__activemask(), b);
        if (lane == __ffs(same) - 1) {
            atomicAdd(&s_hist[b], (unsigned)__popc(same));
            atomicMax(&s_t, b + 1);
        }
    };
    auto hist_end = [&](int parity) {
        __syncthreads();
        for (int i = threadIdx.x; i < (int)s_t; i += kResThreads)
            if (s_hist[i]) atomicAdd(&c->hist[parity][i], s_hist[i]);
        if (threadIdx.x == 0 && s_t) atomicMax(&c->tmax[parity], s_t - 1);
    };

    long long n_u = a.m, rounds = 0;
    int cl = 0;  // a.list[cl] is the current list (the first round: every item)
    bool whole = true;
    if (!a.resume) {
        unsigned deep = 0;
        hist_begin();
        for (int64_t b = warp0 * 32; b < a.g.n; b += warps * 32) {
            const int64_t v = b + lane;
            if (v >= a.g.n) continue;
            unsigned long long f = kDone;
            if (a.state[v] == 0) {
                const int32_t B = a.bcap[v];
                if (B > a.max_ball) {
                    deep = 1;
                } else {
                    f = ((unsigned long long)(uint32_t)B << 32) | a.ord[v];
                    hist_add((unsigned)B);
                }
            }
            a.fk[v] = f;
            a.claimed[v] = 0;
            a.X[0][v] = a.X[1][v] = kNone;
        }
        hist_end(1);
        if (!end_pass(&c->bar, pass, deep, &total)) return;
        if (total) {
            if (scribe) c->deep = 1;
            return;
        }
    } else {
        rounds = __ldcg(&c->rounds);
        n_u = __ldcg(&c->n_u);
        cl = (int)(rounds & 1);
        whole = false;
    }
    const long long stop_at = rounds + kRoundsPerLaunch;
    while (n_u > 0 && rounds < stop_at && rounds <= a.m) {
        ++rounds;
        const int par = (int)(rounds & 1);
        const int4* list = whole ? a.items : a.list[cl];
        int4* next = a.list[cl ^ 1];
        const int64_t n_list = whole ? a.n_items : (int64_t)__ldcg(&c->n_list[cl]);
        const int T = (int)__ldcg(&c->tmax[par]);
        const unsigned long long t_round = scribe ? now_ns() : 0;
        if (scribes)
            for (int b0 = 0; b0 <= T; b0 += 32) {
                const unsigned h = b0 + lane <= T ? __ldcg(&c->hist[par][b0 + lane]) : 0u;
                const unsigned some = __ballot_sync(kFull, h != 0);
                if (h) log_row(a, log_n + __popc(some & ((1u << lane) - 1u)), rounds, 2, b0 + lane, h, 0, 0);
                log_n += __popc(some);
            }
        total = __ldcg(&c->hist[par][T]);
        // ---- cover: facility f enters at time T - B_f, every wave stops at
        // time T.  The values of time 0 are read off fk.
        Held held;
        hold(held, a.g, list, n_list, warp0, warps);
        int x = 0;
        for (int t = 0; t < T; ++t) {
            const unsigned front = total;
            const unsigned long long t0 = scribe ? now_ns() : 0;
            unsigned changed = 0;
            const uint32_t* X = a.X[x];
            uint32_t* Xn = a.X[x ^ 1];
            for_items(held, a.g, list, n_list, warp0, warps, [&](const int4& it, auto low_of) {
                const bool work = it.x >= 0;
                const unsigned long long f = work ? __ldcg(&a.fk[it.x]) : kDone;
                uint32_t own, low;
                if (t == 0) {
                    auto start = [&](unsigned long long w) { return (int)(w >> 32) == T ? (uint32_t)w : kNone; };
                    own = start(f);
                    low = low_of(true, [&](int32_t u) { return start(__ldcg(&a.fk[u])); });
                } else {
                    own = work ? __ldcg(&X[it.x]) : 0u;
                    low = low_of(true, [&](int32_t u) { return __ldcg(&X[u]); });
                }
                if (work && (lane & 7) == 0) {
                    uint32_t nv = min(own, low);
                    if ((int)(f >> 32) == T - (t + 1)) nv = min(nv, (uint32_t)f);
                    if (it.w & kSingle) {
                        Xn[it.x] = nv;
                        changed += nv < own;
                    } else {
                        const uint32_t old = atomicMin(&Xn[it.x], nv);
                        changed += nv < own && old >= own;
                    }
                }
            });
            if (!end_pass(&c->bar, pass, changed, &total)) return;
            if (scribe && front) log_row(a, log_n, rounds, 0, t, front, 1, now_ns() - t0);
            log_n += front != 0;
            x ^= 1;
        }
        uint32_t* cover = a.X[x];
        // ---- gather seeds (0: claimed, else cover key + 1) and the items the
        // cover reached: the list of this round's other sweeps and of the next round
        unsigned seeds = 0;
        if (blockIdx.x == 0) {  // the other parity's buckets: filled after the next barriers
            for (int i = threadIdx.x; i <= kMaxBall; i += kResThreads) c->hist[par ^ 1][i] = 0;
            if (threadIdx.x == 0) c->tmax[par ^ 1] = 0;
        }
        for (int64_t b = warp0 * 32; b < n_list; b += warps * 32) {
            const int4 p = load_item(list, b + lane, n_list);
            uint32_t key = kNone;
            if (p.x >= 0) {
                if (T == 0) {
                    const unsigned long long f = __ldcg(&a.fk[p.x]);
                    key = (int)(f >> 32) == 0 ? (uint32_t)f : kNone;
                } else {
                    key = __ldcg(&cover[p.x]);
                }
            }
            if (p.w & kFirst) {
                const bool seed = key != kNone && a.client[p.x];
                a.Y[0][p.x] = seed ? (a.claimed[p.x] ? 0u : key + 1u) : kNone;
                a.Y[1][p.x] = kNone;
                a.kr[p.x] = 0;
                if (T == 0) cover[p.x] = key;
                seeds += seed;
            }
            const bool keep = key != kNone;
            const unsigned mk = __ballot_sync(kFull, keep);
            if (mk) {
                unsigned at = 0;
                if (lane == 0) at = atomicAdd(&c->n_list[cl ^ 1], (unsigned)__popc(mk));
                at = __shfl_sync(kFull, at, 0);
                if (keep) next[at + __popc(mk & ((1u << lane) - 1u))] = p;
            }
        }
        if (!end_pass(&c->bar, pass, seeds, &total)) return;
        const int64_t n_next = (int64_t)__ldcg(&c->n_list[cl ^ 1]);
        hold(held, a.g, next, n_next, warp0, warps);
        // ---- gather: after b rounds a facility of ball radius b holds the
        // smallest seed of its ball; it decides in the pass that follows (those
        // of radius T in the last pass of the round)
        auto decide = [&](int32_t v, unsigned long long f, uint32_t y) {
            if (y == 0 || y == (uint32_t)f + 1u) {
                a.state[v] = y == 0 ? 2 : 1;
                a.fk[v] = kDone;
                return true;
            }
            if (y == kNone) atomicOr(&c->bar.err, 2u);
            return false;
        };
        int y = 0;
        for (int b = 1; b <= T; ++b) {
            const unsigned front = total;
            const unsigned long long t0 = scribe ? now_ns() : 0;
            unsigned changed = 0;
            const uint32_t* Y = a.Y[y];
            uint32_t* Yn = a.Y[y ^ 1];
            for_items(held, a.g, next, n_next, warp0, warps, [&](const int4& it, auto low_of) {
                const bool work = it.x >= 0;
                const unsigned long long f = (it.w & kFirst) ? __ldcg(&a.fk[it.x]) : kDone;
                const uint32_t own = work ? __ldcg(&Y[it.x]) : 0u;
                const uint32_t low = low_of(true, [&](int32_t u) { return __ldcg(&Y[u]); });
                if (work && (lane & 7) == 0) {
                    if ((int)(f >> 32) == b - 1) decide(it.x, f, own);
                    const uint32_t nv = min(own, low);
                    if (it.w & kSingle) {
                        Yn[it.x] = nv;
                        changed += nv < own;
                    } else {
                        const uint32_t old = atomicMin(&Yn[it.x], nv);
                        changed += nv < own && old >= own;
                    }
                }
            });
            if (!end_pass(&c->bar, pass, changed, &total)) return;
            if (scribe && front) log_row(a, log_n, rounds, 1, b, front, 1, now_ns() - t0);
            log_n += front != 0;
            y ^= 1;
        }
        const uint32_t* ball = a.Y[y];
        // ---- claim the clients of this round's winners (a facility of radius T
        // wins when its ball's smallest seed is its own); they seed the kill sweep
        unsigned fresh = 0;
        if (scribe) c->n_list[cl] = 0;  // read at the round's start; the next round appends to it
        for (int64_t b = warp0 * 32; b < n_next; b += warps * 32) {
            const int4 p = load_item(next, b + lane, n_next);
            if (!(p.w & kFirst) || !a.client[p.x] || a.claimed[p.x]) continue;
            const uint32_t key = __ldcg(&cover[p.x]);
            const int32_t f = a.fac_by_ord[key];
            if (__ldcg(&a.state[f]) == 1 || ((int)(__ldcg(&a.fk[f]) >> 32) == T && __ldcg(&ball[f]) == key + 1u)) {
                a.claimed[p.x] = 1;
                a.kr[p.x] = 1;
                ++fresh;
            }
        }
        if (!end_pass(&c->bar, pass, fresh, &total)) return;
        // ---- kill: vertices within b of a newly claimed client after b rounds
        for (int b = 1; b <= T && total; ++b) {
            const unsigned long long t0 = scribe ? now_ns() : 0;
            unsigned marked = 0;
            for_items(held, a.g, next, n_next, warp0, warps, [&](const int4& it, auto low_of) {
                const bool open_v = it.x >= 0 && __ldcg(&a.kr[it.x]) == 0;
                const uint32_t low = low_of(open_v, [&](int32_t u) {
                    const uint32_t k = __ldcg(&a.kr[u]);
                    return k != 0 && k <= (uint32_t)b ? 0u : kNone;
                });
                if (open_v && (lane & 7) == 0 && low == 0) {
                    a.kr[it.x] = (uint32_t)b + 1;
                    ++marked;
                }
            });
            if (!end_pass(&c->bar, pass, marked, &total)) return;
            if (scribe) log_row(a, log_n, rounds, 4, b, total, 1, now_ns() - t0);
            ++log_n;
        }
        // ---- the facilities of radius T decide; an undecided facility with a
        // newly claimed client in its ball drops out; the others, and the
        // values of the next round's first cover, start the next round
        unsigned left = 0;
        hist_begin();
        for (int64_t b = warp0 * 32; b < n_next; b += warps * 32) {
            const int4 p = load_item(next, b + lane, n_next);
            if (!(p.w & kFirst)) continue;
            a.X[0][p.x] = a.X[1][p.x] = kNone;
            const unsigned long long f = __ldcg(&a.fk[p.x]);
            if (f == kDone) continue;
            if ((int)(f >> 32) == T && decide(p.x, f, __ldcg(&ball[p.x]))) continue;
            const uint32_t k = __ldcg(&a.kr[p.x]);
            if (k != 0 && k - 1 <= (uint32_t)(f >> 32)) {
                a.state[p.x] = 2;
                a.fk[p.x] = kDone;
                continue;
            }
            ++left;
            hist_add((unsigned)(f >> 32));
        }
        hist_end(par ^ 1);
        if (!end_pass(&c->bar, pass, left, &total)) return;
        if (scribe) log_row(a, log_n, rounds, 3, T, n_u, n_u - (long long)total, now_ns() - t_round);
        ++log_n;
        n_u = (long long)total;
        whole = false;
        cl ^= 1;
        if (__ldcg(&c->bar.err)) return;
    }
    if (n_u == 0) {  // the open set and its list
        for (int64_t b = warp0 * 32; b < a.g.n; b += warps * 32) {
            const int64_t v = b + lane;
            const bool o = v < a.g.n && __ldcg(&a.state[v]) == 1;
            if (v < a.g.n) a.open[v] = o ? 1 : 0;
            const unsigned mk = __ballot_sync(kFull, o);
            if (mk) {
                unsigned long long at = 0;
                if (lane == 0) at = atomicAdd(reinterpret_cast<unsigned long long*>(&c->n_open), (unsigned long long)__popc(mk));
                at = __shfl_sync(kFull, at, 0);
                if (o) a.open_list[at + __popc(mk & ((1u << lane) - 1u))] = (int32_t)v;
            }
        }
    }
    if (scribe) {
        c->rounds = rounds;
        c->n_u = n_u;
        c->log_n = min(log_n, a.log_cap);
        c->done = 1;
    }
}

struct BfsArgs {
    ItemGraph g;
    const int64_t* rowp;
    int64_t nnz;
    const int4* items;
    int64_t n_items;
    const int32_t* src;
    int64_t n_src;
    const int32_t* label_of;  // labels of the sources, or NULL (their ids)
    uint32_t* label;
    int32_t* dist;
    int32_t *list0, *list1;   // frontier lists (levels of even / odd number)
    Ctl* c;
    int64_t cap;              // levels at most
};

// With kPush, a level whose frontier's vertices and entries are less than
// 1 / kBfsPushDiv of the graph's items and entries is pushed; where the level
// before pulled, the frontier is listed first, a pass and a barrier more, for which
// a pull must take more than kBfsListSteps items per group of lanes.
constexpr int kBfsPushDiv = 128;
constexpr int kBfsPushSteps = 4;   // items per group of lanes above which the kernel with pushes runs
constexpr int kBfsListSteps = 16;
constexpr int kBfsLong = 64;       // longer rows are pushed by the block's warps in parts
constexpr int kBfsQueue = 256;     // of them, queued per block and level

// Level-synchronous BFS: level L gives every vertex without a distance the
// smallest label among its neighbours at distance L - 1.  In place: a
// distance written in this level is L and does not pass for L - 1.
//
// A pull reads every item and the rows of every vertex not reached.  On graphs of
// many levels, or with a few sources beside hubs, that is all rows for a handful
// of vertices, so thin frontiers push (div 64 costs more than it gives where many
// rows push to a few hubs).  One kernel of pulls alone | this one: grid of 490 k
// vertices, 460 levels 9.46 | 2.69 ms, 50 levels 1.27 | 1.08; Erdos-Renyi, 1 M vertices of
// degree 2, 31 levels 1.47 | 0.82; 50 hubs of 100 k entries, 3 levels 0.70 | 0.20.  A
// graph whose pulls are a few steps runs without: the code for pushes costs it 1 us a level.
template <bool kPush>
__global__ void __launch_bounds__(kResThreads, 1) k_bfs_resident(BfsArgs a) {
    __shared__ int32_t s_queue[kBfsQueue];
    __shared__ unsigned s_queued;
    Ctl* c = a.c;
    const int lane = lane_id(), sub = lane & 7;
    const int64_t tid = (int64_t)blockIdx.x * kResThreads + threadIdx.x, threads = (int64_t)gridDim.x * kResThreads;
    const int64_t group0 = (tid >> 5) * 4, groups = (threads >> 5) * 4;
    unsigned pass = 0, total = 0;
    if (kPush && threadIdx.x == 0) s_queued = 0;
    for (int64_t v = tid; v < a.g.n; v += threads) {
        a.label[v] = kNone;
        a.dist[v] = -1;
    }
    if (!end_pass(&c->bar, pass, 0, &total)) return;
    // total: with pushes the frontier's vertices and entries, else at least its vertices
    auto weight = [&](int64_t v) {
        return kPush ? 1u + (unsigned)(__ldg(&a.rowp[v + 1]) - __ldg(&a.rowp[v])) : 1u;
    };
    unsigned reached = 0;
    for (int64_t i = tid; i < a.n_src; i += threads) {
        const int32_t s = a.src[i];
        a.label[s] = (uint32_t)(a.label_of ? a.label_of[s] : s);
        a.dist[s] = 0;
        if (kPush) reached += weight(s);
    }
    if (!end_pass(&c->bar, pass, reached, &total)) return;
    if (!kPush) total = a.n_src > 0;
    bool listed = true;
    const int32_t* front = a.src;
    int64_t n_front = a.n_src;
    for (int64_t L = 1; total; ++L) {
        if (L > a.cap) {
            if (tid == 0) c->bar.err = 4;
            return;
        }
        int32_t* next = L & 1 ? a.list1 : a.list0;
        unsigned long long* n_next = &c->bfs_n[L & 3];
        if (kPush) {
            if (tid == 0) c->bfs_n[(L + 1) & 3] = 0;  // read last in level L - 2
            const bool thin = (int64_t)total * kBfsPushDiv < a.nnz + a.n_items;
            if (thin && !listed && a.n_items > kBfsListSteps * groups) {
                int32_t* mine = L & 1 ? a.list0 : a.list1;
                for (int64_t b = (tid >> 5) * 32; b < a.g.n; b += (threads >> 5) * 32) {
                    const int64_t v = b + lane;
                    const bool in = v < a.g.n && __ldcg(&a.dist[v]) == (int32_t)L - 1;
                    const long long at = warp_append(in, &c->bfs_n[(L - 1) & 3]);
                    if (at >= 0) mine[at] = (int32_t)v;
                }
                if (!end_pass(&c->bar, pass, 0, &total)) return;
                listed = true;
                front = mine;
                n_front = (int64_t)__ldcg(&c->bfs_n[(L - 1) & 3]);
            }
            listed = listed && thin;  // so is the next level's frontier, then
        }
        reached = 0;
        if (kPush && listed) {
            // label lab to the vertices of the entries e, e + step, ... below end, four at a time (all 32 lanes)
            auto offer = [&](int64_t e, int64_t end, int step, uint32_t lab) {
                int32_t u[4], d[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) u[j] = e + j * step < end ? __ldg(&a.g.cols[e + j * step]) : -1;
#pragma unroll
                for (int j = 0; j < 4; ++j) d[j] = u[j] >= 0 ? __ldcg(&a.dist[u[j]]) : 0;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (d[j] < 0) d[j] = atomicCAS(&a.dist[u[j]], -1, (int32_t)L);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const bool fresh = d[j] < 0;
                    if (u[j] >= 0 && (fresh || d[j] == (int32_t)L) && lab < __ldcg(&a.label[u[j]]))
                        atomicMin(&a.label[u[j]], lab);
                    const long long at = warp_append(fresh, n_next);
                    if (at >= 0) {
                        next[at] = u[j];
                        reached += weight(u[j]);
                    }
                }
            };
            for (int64_t b = group0; b < n_front; b += groups) {
                const int64_t i = b + (lane >> 3);
                const int32_t v = i < n_front ? __ldcg(&front[i]) : -1;
                int64_t e = v >= 0 ? __ldg(&a.rowp[v]) : 0;
                int64_t end = v >= 0 ? __ldg(&a.rowp[v + 1]) : 0;
                if (end - e > kBfsLong) {
                    unsigned at = kBfsQueue;
                    if (sub == 0) at = atomicAdd(&s_queued, 1u);
                    at = __shfl_sync(0xffu << (lane & 24), at, 0, 8);  // the row's eight lanes
                    if (at < kBfsQueue) {
                        if (sub == 0) s_queue[at] = v;
                        end = e;
                    }
                }
                const uint32_t lab = v >= 0 ? __ldcg(&a.label[v]) : kNone;
                for (; __any_sync(kFull, e < end); e += 32) offer(e + sub, end, 8, lab);
            }
            __syncthreads();
            const int queued = (int)min(s_queued, (unsigned)kBfsQueue);
            int dealt = 0;  // 128 entries at a time, dealt to the warps in turn
            for (int q = 0; q < queued; ++q) {
                const int32_t v = s_queue[q];
                const int64_t beg = __ldg(&a.rowp[v]), end = __ldg(&a.rowp[v + 1]);
                const int turn = ((int)(threadIdx.x >> 5) - dealt) & (kResWarps - 1);
                const uint32_t lab = __ldcg(&a.label[v]);
                for (int64_t e = beg + 128 * turn; e < end; e += 128 * kResWarps) offer(e + lane, end, 32, lab);
                dealt += (int)((end - beg + 127) >> 7);
            }
            __syncthreads();
            if (threadIdx.x == 0) s_queued = 0;
        } else {
            for (int64_t b = group0; b < a.n_items; b += groups) {
                const int4 it = b + (lane >> 3) < a.n_items ? __ldg(&a.items[b + (lane >> 3)]) : make_int4(-1, 0, 0, 0);
                const int32_t d = it.x >= 0 ? __ldcg(&a.dist[it.x]) : 0;
                const bool want = it.x >= 0 && (d < 0 || d == (int32_t)L);
                const uint32_t low = item_min(a.g, it.y, want ? it.z : it.y, [&](int32_t u) {
                    return __ldcg(&a.dist[u]) == (int32_t)L - 1 ? __ldcg(&a.label[u]) : kNone;
                });
                if (want && sub == 0 && low != kNone) {
                    if (it.w & kSingle) a.label[it.x] = low;
                    else atomicMin(&a.label[it.x], low);
                    if (!kPush) {
                        a.dist[it.x] = (int32_t)L;
                        ++reached;
                    } else if (it.w & kSingle) {
                        a.dist[it.x] = (int32_t)L;
                        reached += 1u + (unsigned)(it.z - it.y);
                    } else if (d < 0 && atomicCAS(&a.dist[it.x], -1, (int32_t)L) < 0) {
                        reached += weight(it.x);
                    }
                }
            }
        }
        if (!end_pass(&c->bar, pass, reached, &total)) return;
        if (kPush && listed) {
            front = next;
            n_front = (int64_t)__ldcg(n_next);
        }
    }
}

__global__ void k_item_counts(const int64_t* __restrict__ rowp, int64_t n, int32_t* __restrict__ cnt) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const int64_t d = rowp[v + 1] - rowp[v];
        cnt[v] = d <= kItemEdges ? 1 : (int32_t)((d + kItemEdges - 1) / kItemEdges);
    }
}

__global__ void k_item_fill(const int64_t* __restrict__ rowp, const int64_t* __restrict__ pos, int64_t n,
                            int4* __restrict__ items) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const int32_t e0 = (int32_t)rowp[v], e1 = (int32_t)rowp[v + 1];  // nnz <= kResidentEdges
        int64_t at = pos[v];
        for (int32_t e = e0; e == e0 || e < e1; e += kItemEdges)
            items[at++] = make_int4((int)v, e, min(e + kItemEdges, e1),
                                    (e == e0 ? kFirst : 0) | (e1 - e0 <= kItemEdges ? kSingle : 0));
    }
}

// Blocks of a resident launch: one per SM, fewer for few items (a barrier
// among few blocks is cheaper).
int resident_blocks(int64_t n_items, int* out) {
    int dev = 0, sms = 0;
    FL_CUDA(cudaGetDevice(&dev));
    FL_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int64_t want = (n_items * 8 + kResThreads - 1) / kResThreads;
    *out = (int)std::max<int64_t>(1, std::min<int64_t>(sms, want));
    return FL_OK;
}

}  // namespace

int build_items(fl_graph* g) {
    g->n_items = 0;
    if (g->nnz > kResidentEdges || g->n > kResidentEdges) return FL_OK;
    cudaStream_t st = g->stream;
    const int64_t n = g->n;
    DBuf cnt, pos;
    int rc = FL_OK;
    do {
        if ((rc = dalloc(cnt, (size_t)n * 4)) || (rc = dalloc(pos, (size_t)n * 8)) ||
            (rc = dalloc(g->items, (size_t)(n + g->nnz / kItemEdges + 1) * 16)))
            break;
        const unsigned grid = (unsigned)std::min<int64_t>((n + 255) / 256, 152 * 8);
        FL_LAUNCH(kProfOther, k_item_counts<<<grid, 256, 0, st>>>(g->rowp.as<int64_t>(), n, cnt.as<int32_t>()));
        if ((rc = scan_exclusive_i32_to_i64(cnt.as<int32_t>(), pos.as<int64_t>(), n, st, g->scratch, kProfOther)))
            break;
        FL_LAUNCH(kProfOther, k_item_fill<<<grid, 256, 0, st>>>(g->rowp.as<int64_t>(), pos.as<int64_t>(), n,
                                                                g->items.as<int4>()));
        int64_t p = 0;
        int32_t c = 0;
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(&p, pos.as<int64_t>() + n - 1, 8, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&c, cnt.as<int32_t>() + n - 1, 4, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) { rc = status_of(e, "work items", __FILE__, __LINE__); break; }
        if (p + c <= kResidentItems) g->n_items = p + c;
    } while (0);
    if (g->n_items == 0) dfree_after(st, {&g->items});
    dfree_after(st, {&cnt, &pos});
    return rc;
}

static ItemGraph item_graph(const fl_graph* g) {
    ItemGraph ig;
    ig.cols = g->cols.as<int32_t>();
    ig.n = g->n;
    return ig;
}

constexpr size_t kCtlBytes = (sizeof(Ctl) + 255) & ~(size_t)255;

// Arguments of the greedy MIS of the m sorted candidates (s->ord,
// s->fac_by_ord, s->bcap, s->state set), its scratch and a cleared control block.
static int mis_args(fl_solve* s, int64_t m, MisArgs* out, int* blocks) {
    fl_graph* g = s->g;
    const int64_t n = g->n;
    MisArgs& a = *out;
    FL_TRY(dalloc(s->X, (size_t)n * 16));
    FL_TRY(dalloc(s->frval, (size_t)n * 8 + 64));
    FL_TRY(dalloc(s->fr[0], (size_t)n * 4));
    FL_TRY(dalloc(s->claimed, (size_t)n));
    FL_TRY(dalloc(s->rlist, (size_t)g->n_items * 32));
    // a greedy round logs at most its buckets, three sweeps and a total
    const long long log_cap = (long long)kRoundsPerLaunch * (4LL * kMaxBall + 8);
    FL_TRY(dalloc(s->rctl, kCtlBytes + (size_t)log_cap * 48));
    a.g = item_graph(g);
    a.items = g->items.as<int4>();
    a.n_items = g->n_items;
    a.X[0] = s->X.as<uint32_t>();
    a.X[1] = a.X[0] + n;
    a.Y[0] = a.X[0] + 2 * n;
    a.Y[1] = a.X[0] + 3 * n;
    a.kr = s->fr[0].as<uint32_t>();
    a.fk = s->frval.as<unsigned long long>();
    a.list[0] = s->rlist.as<int4>();
    a.list[1] = a.list[0] + g->n_items;
    a.ord = s->ord.as<uint32_t>();
    a.fac_by_ord = s->fac_by_ord.as<int32_t>();
    a.bcap = s->bcap.as<int32_t>();
    a.state = s->state.as<uint8_t>();
    a.client = s->client.as<uint8_t>();
    a.claimed = s->claimed.as<uint8_t>();
    a.open = s->open.as<uint8_t>();
    a.open_list = s->ulist.as<int32_t>();
    a.c = s->rctl.as<Ctl>();
    a.log = reinterpret_cast<long long*>(s->rctl.as<char>() + kCtlBytes);
    a.log_cap = log_cap;
    a.m = m;
    a.max_ball = g->n_items > kWideBallItems ? kNarrowBall : kMaxBall;
    a.resume = 0;
    FL_TRY(resident_blocks(g->n_items, blocks));
    FL_CUDA(cudaMemsetAsync(s->rctl.p, 0, sizeof(Ctl), g->stream));
    return FL_OK;
}

static cudaError_t mis_launch(const MisArgs& a, int blocks, cudaStream_t st) {
    void* args[] = {const_cast<MisArgs*>(&a)};
    return cudaLaunchCooperativeKernel((const void*)k_mis_resident, dim3(blocks), dim3(kResThreads), args, 0, st);
}

// A finished selection's open set into acc; *outcome = 1 when it finished (in
// one launch, without an error), else 0 and acc is left alone.
__global__ void k_mis_take(const Ctl* __restrict__ c, const uint8_t* __restrict__ open, int64_t n,
                           uint8_t* __restrict__ acc, int* __restrict__ outcome) {
    const bool done = c->done != 0 && c->n_u == 0 && c->bar.err == 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid == 0) *outcome = done ? 1 : 0;
    if (!done) return;
    for (int64_t v = tid; v < n; v += stride)
        if (open[v]) acc[v] = 1;
}

// One launch of the greedy MIS and k_mis_take behind it, without a look by the host.
int mis_resident_queue(fl_solve* s, int64_t m, uint8_t* acc, int* outcome) {
    cudaStream_t st = s->g->stream;
    MisArgs a;
    int blocks = 0;
    FL_TRY(mis_args(s, m, &a, &blocks));
    cudaError_t le = cudaSuccess;
    FL_LAUNCH(kProfMis, le = mis_launch(a, blocks, st));
    FL_CUDA(le);
    FL_LAUNCH(kProfMis, k_mis_take<<<(unsigned)std::min<int64_t>((s->g->n + 255) / 256, 152 * 4), 256, 0, st>>>(
                            a.c, a.open, s->g->n, acc, outcome));
    FL_CUDA(cudaGetLastError());
    return FL_OK;
}

// The greedy MIS of the m sorted candidates and its open list.  *done = false:
// not for this kernel (a ball radius above max_ball); nothing but scratch was
// written.
int mis_resident(fl_solve* s, int64_t m, bool* done) {
    fl_graph* g = s->g;
    cudaStream_t st = g->stream;
    *done = false;
    MisArgs a;
    int blocks = 0;
    FL_TRY(mis_args(s, m, &a, &blocks));
    char* h = reinterpret_cast<char*>(g->h_ctr) + sizeof(Counters);  // pinned
    const size_t h_b = kCtlBytes + kFastRows * 48;
    static_assert(sizeof(Counters) + kCtlBytes + kFastRows * 48 <= kPinnedBytes, "pinned block");
    for (;;) {
        cudaError_t le = cudaSuccess;
        FL_LAUNCH(kProfMis, le = mis_launch(a, blocks, st));
        FL_CUDA(le);
        FL_CUDA(cudaMemcpyAsync(h, s->rctl.p, h_b, cudaMemcpyDeviceToHost, st));
        FL_CUDA(cudaStreamSynchronize(st));
        const Ctl* c = reinterpret_cast<const Ctl*>(h);
        if (c->deep) return FL_OK;
        if (c->bar.err & 1u) FL_FAIL(FL_ETIMEOUT, "greedy MIS: a barrier wait ran out");
        if (c->bar.err) FL_FAIL(FL_ECUDA, "greedy MIS: inconsistent gather state");
        const size_t at = s->mis_log.size(), rows = (size_t)c->log_n;
        s->mis_log.resize(at + rows * 6);
        if (rows <= (size_t)kFastRows) {
            std::copy_n(reinterpret_cast<const int64_t*>(h + kCtlBytes), rows * 6, s->mis_log.begin() + at);
        } else {
            FL_CUDA(cudaMemcpyAsync(s->mis_log.data() + at, a.log, rows * 48, cudaMemcpyDeviceToHost, st));
            FL_CUDA(cudaStreamSynchronize(st));
        }
        s->mis_rounds = c->rounds;
        if (c->n_u == 0) {
            s->n_open = c->n_open;
            break;
        }
        if (c->rounds > m) FL_FAIL(FL_ETIMEOUT, "greedy MIS did not converge");
        // barrier and pass counters start again; the round state stays
        a.resume = 1;
        FL_CUDA(cudaMemsetAsync(a.c->bar.pass, 0, sizeof(a.c->bar.pass), st));
        FL_CUDA(cudaMemsetAsync(&a.c->log_n, 0, 8, st));
    }
    *done = true;
    return FL_OK;
}

int msbfs_resident(fl_graph* g, const int32_t* src, int64_t n_src, int32_t* label, int32_t* dist, DBuf& ctl,
                   DBuf& lists, int cls) {
    cudaStream_t st = g->stream;
    FL_TRY(dalloc(ctl, sizeof(Ctl)));
    int blocks = 0;
    FL_TRY(resident_blocks(g->n_items, &blocks));
    const bool push = g->n_items > (int64_t)kBfsPushSteps * blocks * (kResThreads / 8);
    if (push) FL_TRY(dalloc(lists, (size_t)g->n * 8));
    BfsArgs a;
    a.g = item_graph(g);
    a.rowp = g->rowp.as<int64_t>();
    a.nnz = g->nnz;
    a.list0 = lists.as<int32_t>();
    a.list1 = a.list0 + g->n;
    a.items = g->items.as<int4>();
    a.n_items = g->n_items;
    a.src = src;
    a.n_src = n_src;
    a.label_of = g->rid.p ? g->rid.as<int32_t>() : nullptr;
    a.label = reinterpret_cast<uint32_t*>(label);
    a.dist = dist;
    a.c = ctl.as<Ctl>();
    a.cap = g->sched.level_cap > 0 ? g->sched.level_cap : g->n + 2;
    FL_CUDA(cudaMemsetAsync(ctl.p, 0, sizeof(Ctl), st));
    void* args[] = {&a};
    cudaError_t le = cudaSuccess;
    const void* kernel = push ? (const void*)k_bfs_resident<true> : (const void*)k_bfs_resident<false>;
    FL_LAUNCH(cls, le = cudaLaunchCooperativeKernel(kernel, dim3(blocks), dim3(kResThreads), args, 0, st));
    FL_CUDA(le);
    unsigned* h = reinterpret_cast<unsigned*>(g->h_ctr + 1);
    FL_CUDA(cudaMemcpyAsync(h, &a.c->bar.err, 4, cudaMemcpyDeviceToHost, st));
    FL_CUDA(cudaStreamSynchronize(st));
    const unsigned err = *h;
    if (err & 4u) FL_FAIL(FL_ETIMEOUT, "BFS reached its level cap");
    if (err) FL_FAIL(FL_ETIMEOUT, "BFS: a barrier wait ran out");
    return FL_OK;
}

}  // namespace fl

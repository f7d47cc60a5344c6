// k_wsolve.cu -- the greedy MIS (phase iii) and the assignment on a weighted
// graph: balls and nearest facilities by weighted distance (Section 3.1 with
// the edge lengths of Section 3.3).
//
// Ball(f) = the clients within distance B_f = floor(r_f) of f.  The MIS is
// the lexicographically-first one under the keys (r_f, pi_f), as on an
// unweighted graph, found in greedy rounds: in each round every client gets
// the smallest key among the undecided facilities whose ball holds it (the
// cover), a facility whose ball holds only clients carrying its own key
// joins S (the gather), its clients are claimed, and every undecided facility
// whose ball holds a newly claimed client drops out (the kill).  The round's
// smallest undecided key always joins, and a facility joins exactly when
// every facility before it in key order that shares a client with it has
// dropped out, so the rounds end at the sequential greedy's set.
//
// Each of the three steps is a sweep over integer time: a value leaving
// vertex u at time t reaches neighbour v at time t + w(u, v).  A ring of
// R = (largest length + 1) slots holds the arrivals of the coming times: slot
// t mod R keeps, per vertex, the smallest value arriving at time t, and the
// list of vertices that have one.  Step t drains its slot into the labels and
// a vertex whose label drops pushes it along its edges into later slots.
// A sweep is one resident kernel with one grid barrier per time that has
// arrivals; times without are passed over.  With three launches per time step
// a sweep was bound by them and by the largest hub, pushed by one warp: the 24
// sweeps (2819 times) of an R-MAT graph with 65 k vertices and lengths up to
// 100 took 45 ms, 12.3 ms now; bound by the barriers (4.5 us per time) and dependent
// loads.
//   cover:  facility f enters at time H - B_f with its key ordinal (H = the
//           largest B_f), so every wave ends at H and the label of v at H is
//           the smallest key whose ball holds v;
//   gather: each covered client enters at time 0 with its cover label, and f
//           reads its label at time B_f: the smallest cover label over its
//           ball (a deadline per vertex);
//   kill:   each newly claimed client enters at time 0, and f drops out when
//           anything has reached it by time B_f.
// The assignment is the same sweep with every open facility entering at
// time 0 with its id, where a vertex keeps its first arrival: the distance
// to the nearest open facility and, among those at that distance, the
// smallest id (the slot keeps the minimum of the values arriving together).
#include <algorithm>
#include <chrono>
#include <cstdio>
#include <vector>

#include "fl_internal.cuh"

namespace fl {

namespace {

constexpr uint32_t kNone = 0xffffffffu;
int grid_for(int64_t items, int per_block, int cap = 152 * 4) {
    int64_t b = (items + per_block - 1) / per_block;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return (int)b;
}

struct WSweep {
    const int64_t* rowp;
    const int32_t* cols;
    const int32_t* wts;
    int64_t n;
    int R;
    uint32_t* pend;             // R*n: smallest value arriving at each vertex at the slot's time (kNone: none)
    int32_t* plist;             // R*n: vertices with an arrival, per slot
    unsigned long long* pcnt;   // 2R: list lengths, of time t at t mod 2R
    uint32_t* lab;              // current label (kNone: none)
    const int32_t* dl;          // deadline: the label at this time is kept in dlab (or NULL)
    uint32_t* dlab;             // smallest arrival up to the deadline
    int32_t* dist;              // first-arrival mode: arrival time
    uint8_t* past;              // first-arrival mode: 1 where a push went past the horizon
    int32_t* ft;                // (cover) time of each vertex's first arrival, or NULL
    const int32_t* fts;         // (gather, kill) the cover's first arrivals: prune by slack, or NULL
    int first;                  // 1: a vertex keeps its first arrival; 0: the minimum
};

// One arrival of x at v at time t; true when v joins the step's frontier.
__device__ __forceinline__ bool arrive(const WSweep& a, int32_t v, uint32_t x, int64_t t) {
    if (a.dl && t <= (int64_t)__ldg(&a.dl[v]) && x < __ldcg(&a.dlab[v])) a.dlab[v] = x;
    const uint32_t old = __ldcg(&a.lab[v]);
    if (a.first) {
        if (old != kNone) return false;
        a.dist[v] = (int32_t)t;
    } else if (x >= old) {
        return false;
    }
    if (a.ft && old == kNone) a.ft[v] = (int32_t)t;
    a.lab[v] = x;
    return true;
}

// First index i in [0, m) with bs[i] >= b (m when none), bs non-decreasing.
// All 32 lanes call it and get the answer: each pass probes 32 evenly spaced
// positions of the remaining range at once (log32 m dependent loads).
__device__ int64_t warp_lower_bound(const int32_t* __restrict__ bs, int64_t m, int64_t b) {
    int64_t lo = 0, hi = m;  // the answer lies in [lo, hi]
    while (lo < hi) {
        const int64_t step = (hi - lo + 31) / 32;
        const int64_t p = lo + step * lane_id();
        const bool below = p < hi && (int64_t)bs[p] < b;
        const int c = __popc(__ballot_sync(kFull, below));  // the probes below b are a prefix
        if (c == 0) break;                                  // bs[lo] >= b
        const int64_t first_not = lo + step * c;
        lo += step * (c - 1) + 1;
        hi = first_not < hi ? first_not : hi;
    }
    return lo;
}

// Control block of a sweep (device, zero at its start).
struct WSweepCtl {
    GridBar bar;
    long long t_end, steps;  // last time that had arrivals, times run
};

// The cover's entering facilities (m = 0 for sweeps whose sources all enter
// at time 0): candidates in key order have non-decreasing B_f (bsort[i] = B of
// the i-th), a candidate's value is its ordinal.  Or the sources of time 0:
// every vertex with mask[v] (all when NULL) enters with val[v] (its id when
// val is NULL), unless that is kNone.
struct WEntry {
    const int32_t* fac_by_ord;
    const int32_t* bsort;
    const uint8_t* state;
    int64_t m;
    bool seeds;
    const uint32_t* val;
    const uint8_t* mask;
};

constexpr int kPLong = 32;    // longer rows are pushed by the whole block (512: 13.3 ms of sweeps for 12.7)
constexpr int kPQueue = 256;  // of them, queued per block and step

// x arrives at v at time t: into the ring.
__device__ __forceinline__ void send(const WSweep& a, int32_t v, uint32_t x, uint32_t t) {
    const int64_t slot = (int64_t)(t % (uint32_t)a.R) * a.n;
    if (atomicMin(&a.pend[slot + v], x) == kNone)
        a.plist[slot + (int64_t)atomicAdd(&a.pcnt[t % (2u * (uint32_t)a.R)], 1ULL)] = v;
}

// v's label x goes out along the entries e0 + first, + step, ... of its row.
// An arrival that cannot lower u's label is not sent: u's label already holds
// a value at most x from an arrival at or before t, and that arrival was also
// kept by u's deadline whenever this one would be.  (A label that drops in
// this same step does so by an arrival at t.)  The same holds for an arrival of
// time t that is still in the slot (now: the slot's values): the step drains
// and pushes at once, and an arrival sent past a label that is about to drop is
// one more time to run.  Star of 1000 vertices, lengths up to 5000, every vertex
// a source: assignment 1.4 to 2.8 ms without the look at the slot, 0.12 with it.
__device__ __forceinline__ void push_row(const WSweep& a, int64_t e0, int64_t e1, int first, int step, uint32_t x,
                                         int64_t t, int64_t H, const uint32_t* now) {
    for (int64_t e = e0 + first + lane_id(); e < e1; e += step) {
        const int32_t u = __ldg(&a.cols[e]);
        const uint32_t lu = __ldcg(&a.lab[u]);
        if (a.first ? lu != kNone : lu <= x) continue;
        const int64_t t2 = t + __ldg(&a.wts[e]);
        if (a.fts) {  // u relays nothing useful after its slack H - (first cover arrival)
            const int32_t fu = __ldg(&a.fts[u]);
            if (fu < 0 || t2 > H - (int64_t)fu) continue;
        }
        if (t2 > H) {
            if (a.first) a.past[u] = 1;
            continue;
        }
        const uint32_t pu = __ldcg(&now[u]);
        if (a.first ? pu != kNone : pu <= x) continue;
        send(a, u, x, (uint32_t)t2);
    }
}

// One sweep over times 0..H.
//
// A facility that enters at time te is sent to itself as an arrival of te as
// soon as te is less than R away.  The list length of time t is read by every
// block in step t and cleared in the next one, t': t' <= t + R - 1, so no
// send of step t' (to times up to t' + R - 1) uses the same of the 2R counters.
__global__ void __launch_bounds__(kResThreads, 1) k_wsweep(WSweep a, WEntry in, int64_t H, WSweepCtl* c) {
    __shared__ int64_t s_e0[kPQueue], s_e1[kPQueue];
    __shared__ uint32_t s_x[kPQueue];
    __shared__ unsigned s_queued, s_next;
    __shared__ long long s_first;
    const int lane = lane_id();
    const int64_t tid = (int64_t)blockIdx.x * kResThreads + threadIdx.x, threads = (int64_t)gridDim.x * kResThreads;
    // chunk i to warp i / gridDim of block i mod gridDim: neighbours in a list go to different blocks
    const int64_t item0 = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x, warps = threads >> 5;
    unsigned pass = 0, total = 0;
    if (threadIdx.x == 0) s_queued = 0;

    // the facilities with entry times below t + R that have not entered:
    // candidates [first, left); left = first
    int64_t left = in.m;
    auto enter = [&](int64_t t) {
        if (left == 0) return;
        if (threadIdx.x < 32) {
            const int64_t at = warp_lower_bound(in.bsort, left, H - t - a.R + 1);
            if (lane == 0) s_first = at;
        }
        __syncthreads();
        const int64_t first = s_first;
        __syncthreads();
        for (int64_t i = first + tid; i < left; i += threads) {
            const int32_t f = __ldg(&in.fac_by_ord[i]);
            if (__ldg(&in.state[f]) == 0) send(a, f, (uint32_t)i, (uint32_t)(H - (int64_t)__ldg(&in.bsort[i])));
        }
        left = first;
    };
    // the first time from t + from on, below t + R, that has arrivals (-1: none)
    auto next_time = [&](int64_t t, int from) -> int64_t {
        if (threadIdx.x == 0) s_next = ~0u;
        __syncthreads();
        for (int d = from + (int)threadIdx.x; d < a.R; d += kResThreads)
            if (__ldcg(&a.pcnt[(uint32_t)(t + d) % (2u * (uint32_t)a.R)])) {
                atomicMin(&s_next, (unsigned)d);
                break;
            }
        __syncthreads();
        const unsigned d = s_next;
        __syncthreads();
        return d == ~0u ? -1 : t + (int64_t)d;
    };

    if (in.seeds)
        for (int64_t v = tid; v < a.n; v += threads)
            if (!in.mask || in.mask[v]) {
                const uint32_t x = in.val ? in.val[v] : (uint32_t)v;
                if (x != kNone) send(a, (int32_t)v, x, 0u);
            }
    enter(0);
    if (!end_pass(&c->bar, pass, 0, &total)) return;
    int64_t t = next_time(0, 0), prev = -1, steps = 0;
    for (;;) {
        if (t < 0) {  // nothing in flight: the next entry, or the end
            if (left == 0) break;
            const int64_t te = H - (int64_t)__ldg(&in.bsort[left - 1]);
            if (tid == 0 && prev >= 0) a.pcnt[(uint32_t)prev % (2u * (uint32_t)a.R)] = 0;
            prev = -1;
            if (!end_pass(&c->bar, pass, 0, &total)) return;
            enter(te);
            if (!end_pass(&c->bar, pass, 0, &total)) return;
            t = next_time(te, 0);
            continue;
        }
        const int64_t slot = (int64_t)((uint32_t)t % (uint32_t)a.R) * a.n;
        const int64_t cnt = (int64_t)__ldcg(&a.pcnt[(uint32_t)t % (2u * (uint32_t)a.R)]);
        if (tid == 0 && prev >= 0) a.pcnt[(uint32_t)prev % (2u * (uint32_t)a.R)] = 0;
        // chunks of a few arrivals per warp, one lane each to drain them
        const int64_t per = min((int64_t)32, (cnt + warps - 1) / warps);
        for (int64_t i0 = item0 * per; i0 < cnt; i0 += warps * per) {
            const int64_t i = i0 + lane;
            bool join = false;
            int32_t v = 0;
            uint32_t x = kNone;
            if (lane < per && i < cnt) {
                v = __ldcg(&a.plist[slot + i]);
                x = __ldcg(&a.pend[slot + v]);
                join = arrive(a, v, x, t);
                a.pend[slot + v] = kNone;  // after the label: push_row looks at it and then at the slot
            }
            for (unsigned m = __ballot_sync(kFull, join); m; m &= m - 1) {
                const int l = __ffs(m) - 1;
                const int32_t u = __shfl_sync(kFull, v, l);
                const uint32_t y = __shfl_sync(kFull, x, l);
                const int64_t e0 = __ldg(&a.rowp[u]), e1 = __ldg(&a.rowp[u + 1]);
                if (e1 - e0 > kPLong) {
                    unsigned at = 0;
                    if (lane == 0) at = atomicAdd(&s_queued, 1u);
                    at = __shfl_sync(kFull, at, 0);
                    if (at < kPQueue) {
                        if (lane == 0) {
                            s_e0[at] = e0;
                            s_e1[at] = e1;
                            s_x[at] = y;
                        }
                        continue;
                    }
                }
                push_row(a, e0, e1, 0, 32, y, t, H, a.pend + slot);
            }
        }
        __syncthreads();
        const int queued = (int)min(s_queued, (unsigned)kPQueue);
        int dealt = 0;  // 32 entries at a time, dealt to the warps in turn
        for (int q = 0; q < queued; ++q) {
            const int64_t e0 = s_e0[q], e1 = s_e1[q];
            const int turn = (int)((threadIdx.x >> 5) - (unsigned)dealt) & (kResWarps - 1);
            push_row(a, e0, e1, 32 * turn, kResThreads, s_x[q], t, H, a.pend + slot);
            dealt += (int)((e1 - e0 + 31) >> 5);
        }
        __syncthreads();
        if (threadIdx.x == 0) s_queued = 0;
        enter(t);
        ++steps;
        if (!end_pass(&c->bar, pass, 0, &total)) return;
        prev = t;
        t = next_time(t, 1);
    }
    if (tid == 0) {
        if (prev >= 0) a.pcnt[(uint32_t)prev % (2u * (uint32_t)a.R)] = 0;
        c->t_end = prev < 0 ? 0 : prev;
        c->steps = steps;
    }
}

// Ordinals and ball radii of the sorted candidates: ord[f] = position in key
// order, B_f = floor(r_f) (at most 2^31 - 1).
__global__ void k_wordinals(const uint32_t* __restrict__ sorted_f, int64_t m, const double* __restrict__ r,
                            uint32_t* __restrict__ ord, int32_t* __restrict__ fac_by_ord, int32_t* __restrict__ bcap,
                            int32_t* __restrict__ bsort) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) {
        const int32_t f = (int32_t)sorted_f[i];
        ord[f] = (uint32_t)i;
        fac_by_ord[i] = f;
        const double fl = floor(r[f]);
        const int32_t b = fl >= 2147483647.0 ? 2147483647 : (int32_t)fl;
        bcap[f] = b;
        bsort[i] = b;
    }
}

// Undecided facilities: count, largest and smallest B_f.
__global__ void k_wundecided(const int32_t* __restrict__ fac_by_ord, const int32_t* __restrict__ bcap,
                             const uint8_t* __restrict__ state, int64_t m, unsigned long long* __restrict__ out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long c = 0, bmax = 0, bmin = ~0ULL;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < m; base += stride) {
        const int64_t i = base + lane_id();
        if (i < m) {
            const int32_t f = fac_by_ord[i];
            if (state[f] == 0) {
                const unsigned long long b = (unsigned long long)bcap[f];
                ++c;
                bmax = b > bmax ? b : bmax;
                bmin = b < bmin ? b : bmin;
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        c += __shfl_xor_sync(kFull, c, o);
        const unsigned long long x = __shfl_xor_sync(kFull, bmax, o), y = __shfl_xor_sync(kFull, bmin, o);
        bmax = x > bmax ? x : bmax;
        bmin = y < bmin ? y : bmin;
    }
    if (lane_id() == 0 && c) {
        atomicAdd(&out[0], c);
        atomicMax(&out[1], bmax);
        atomicMin(&out[2], bmin);
    }
}

// Gather decision: an undecided f whose ball's smallest cover label is its
// own ordinal (or whose ball holds no client) joins S.  A smaller label means
// an undecided facility before f shares a client with it; a larger one
// cannot happen (f's own wave labels every client of its ball).
__global__ void k_wdecide(const int32_t* __restrict__ fac_by_ord, int64_t m, const uint32_t* __restrict__ dlab,
                          uint8_t* __restrict__ state, unsigned long long* __restrict__ joined,
                          unsigned long long* __restrict__ err) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long c = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) {
        const int32_t f = fac_by_ord[i];
        if (state[f] != 0) continue;
        const uint32_t g = dlab[f];
        if (g == kNone || g == (uint32_t)i) {
            state[f] = 1;
            ++c;
        } else if (g > (uint32_t)i) {
            atomicOr(err, 1ULL);
        }
    }
    if (c) atomicAdd(joined, c);
}

// Claims: a covered client whose cover label belongs to a facility that
// joined S is claimed and seeds the kill sweep.
__global__ void k_wclaim(int64_t n, const uint8_t* __restrict__ client, const uint32_t* __restrict__ cover,
                         const int32_t* __restrict__ fac_by_ord, const uint8_t* __restrict__ state,
                         uint8_t* __restrict__ claimed, uint8_t* __restrict__ seed,
                         unsigned long long* __restrict__ n_new) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long c = 0;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        uint8_t sd = 0;
        const uint32_t o = cover[v];
        if (client[v] && o != kNone && state[fac_by_ord[o]] == 1) {
            claimed[v] = 1;
            sd = 1;
            ++c;
        }
        seed[v] = sd;
    }
    if (c) atomicAdd(n_new, c);
}

// Kill decision: an undecided facility reached by a newly claimed client
// within its ball radius drops out.
__global__ void k_wkill(const int32_t* __restrict__ fac_by_ord, int64_t m, const uint32_t* __restrict__ dlab,
                        uint8_t* __restrict__ state) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) {
        const int32_t f = fac_by_ord[i];
        if (state[f] == 0 && dlab[f] != kNone) state[f] = 2;
    }
}

__global__ void k_wopen(const uint8_t* __restrict__ state, int64_t n, uint8_t* __restrict__ open,
                        unsigned long long* __restrict__ n_open) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long c = 0;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const uint8_t o = state[v] == 1 ? 1 : 0;
        open[v] = o;
        c += o;
    }
    if (c) atomicAdd(n_open, c);
}

// A vertex that a push past the horizon would have reached but that no
// arrival settled lies farther than the horizon.
__global__ void k_wbeyond(int64_t n, const uint8_t* __restrict__ past, const uint32_t* __restrict__ lab,
                          unsigned long long* __restrict__ err) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride)
        if (past[v] && lab[v] == kNone) atomicOr(err, 2ULL);
}

// Device state of the sweeps of one call: the ring and counters.
struct WRing {
    DBuf pend, plist, cnt, ctl;
    int R = 0;
    int64_t n = 0;
    unsigned long long* c = nullptr;  // [0, 2R): list lengths; then kErr ... kOpen
    enum { kErr = 0, kUndecided = 1, kMaxB = 2, kMinB = 3, kJoined = 4, kClaimed = 5, kOpen = 6, kWords = 8 };
    int alloc(fl_graph* g) {
        R = g->max_w + 1;
        n = g->n;
        FL_TRY(dalloc(pend, (size_t)R * n * 4));
        FL_TRY(dalloc(plist, (size_t)R * n * 4));
        FL_TRY(dalloc(cnt, (size_t)(2 * R + kWords) * 8));
        FL_TRY(dalloc(ctl, sizeof(WSweepCtl)));
        c = cnt.as<unsigned long long>() + 2 * R;
        FL_CUDA(cudaMemsetAsync(pend.p, 0xff, (size_t)R * n * 4, g->stream));
        FL_CUDA(cudaMemsetAsync(cnt.p, 0, (size_t)(2 * R + kWords) * 8, g->stream));
        return FL_OK;
    }
    WSweep sweep(const fl_graph* g) const {
        WSweep a;
        a.rowp = g->rowp.as<int64_t>();
        a.cols = g->cols.as<int32_t>();
        a.wts = g->wts.as<int32_t>();
        a.n = n;
        a.R = R;
        a.pend = pend.as<uint32_t>();
        a.plist = plist.as<int32_t>();
        a.pcnt = cnt.as<unsigned long long>();
        a.lab = nullptr;
        a.dl = nullptr;
        a.dlab = nullptr;
        a.dist = nullptr;
        a.past = nullptr;
        a.ft = nullptr;
        a.fts = nullptr;
        a.first = 0;
        return a;
    }
    void release(cudaStream_t st) { dfree_after(st, {&pend, &plist, &cnt, &ctl}); }
};

// Runs one sweep (the ring is empty before and after).  *t_end = the last
// time that had arrivals, *steps = the times run.
int run_sweep(fl_graph* g, WRing& ring, WSweep a, int64_t H, WEntry in, int cls, int64_t* t_end, int64_t* steps) {
    cudaStream_t st = g->stream;
    int dev = 0, sms = 0;
    FL_CUDA(cudaGetDevice(&dev));
    FL_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(sms, (a.n + 31) / 32));
    WSweepCtl* c = ring.ctl.as<WSweepCtl>();
    FL_CUDA(cudaMemsetAsync(c, 0, sizeof(WSweepCtl), st));
    void* args[] = {&a, &in, &H, &c};
    cudaError_t le = cudaSuccess;
    FL_LAUNCH(cls, le = cudaLaunchCooperativeKernel((const void*)k_wsweep, dim3(blocks), dim3(kResThreads), args, 0,
                                                    st));
    FL_CUDA(le);
    WSweepCtl h{};
    FL_CUDA(cudaMemcpyAsync(&h, c, sizeof(WSweepCtl), cudaMemcpyDeviceToHost, st));
    FL_CUDA(cudaStreamSynchronize(st));
    if (h.bar.err) FL_FAIL(FL_ETIMEOUT, "weighted sweep: a barrier wait ran out");
    *t_end = h.t_end;
    *steps = h.steps;
    return FL_OK;
}

}  // namespace

int open_facilities_weighted(fl_solve* s) {
    fl_graph* g = s->g;
    const int64_t n = g->n;
    cudaStream_t st = g->stream;
    using clock = std::chrono::steady_clock;
    s->mis_log.clear();
    int64_t m = 0;
    const uint32_t* sorted = nullptr;
    FL_TRY(sort_candidates(s, &m, &sorted));
    FL_TRY(dalloc(s->ord, (size_t)n * 4));
    FL_TRY(dalloc(s->fac_by_ord, (size_t)std::max<int64_t>(m, 1) * 4));
    FL_TRY(dalloc(s->bcap, (size_t)n * 4));
    FL_TRY(dalloc(s->claimed, (size_t)n));
    FL_TRY(dalloc(s->kill, (size_t)n));
    FL_TRY(dalloc(s->open, (size_t)n));
    FL_TRY(dalloc(s->X, (size_t)n * 16));  // cover labels, sweep labels, deadline labels, first arrivals
    FL_TRY(dalloc(s->ubuck, (size_t)std::max<int64_t>(m, 1) * 4));
    uint32_t* cover = s->X.as<uint32_t>();
    uint32_t* lab = cover + n;
    uint32_t* dlab = cover + 2 * n;
    int32_t* ft = reinterpret_cast<int32_t*>(cover + 3 * n);
    int32_t* bsort = s->ubuck.as<int32_t>();
    int32_t* fac_by_ord = s->fac_by_ord.as<int32_t>();
    int32_t* bcap = s->bcap.as<int32_t>();
    uint8_t* state = s->state.as<uint8_t>();
    FL_CUDA(cudaMemsetAsync(s->bcap.p, 0xff, (size_t)n * 4, st));
    FL_CUDA(cudaMemsetAsync(s->claimed.p, 0, (size_t)n, st));
    if (m > 0)
        FL_LAUNCH(kProfKeys, k_wordinals<<<grid_for(m, 256), 256, 0, st>>>(sorted, m,
                                                                          s->radii.as<double>(), s->ord.as<uint32_t>(),
                                                                          fac_by_ord, bcap, bsort));
    FL_CUDA(cudaGetLastError());
    WRing ring;
    int rc = ring.alloc(g);
    unsigned long long* c = ring.c;
    int64_t rounds = 0;
    while (rc == FL_OK) {
        const auto round_t0 = clock::now();
        unsigned long long h[4] = {0, 0, 0, 0};
        cudaError_t e = cudaMemsetAsync(c + WRing::kUndecided, 0, 16, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(c + WRing::kMinB, 0xff, 8, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(c + WRing::kJoined, 0, 16, st);
        if (e != cudaSuccess) { rc = status_of(e, "weighted MIS", __FILE__, __LINE__); break; }
        if (m > 0)
            FL_LAUNCH(kProfMis, k_wundecided<<<grid_for(m, 256), 256, 0, st>>>(fac_by_ord, bcap, state, m,
                                                                               c + WRing::kUndecided));
        e = cudaMemcpyAsync(h, c, 32, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) { rc = status_of(e, "weighted MIS", __FILE__, __LINE__); break; }
        if (h[0]) { rc = FL_ECUDA; set_error(rc, "weighted MIS: a ball's smallest label is above its own key"); break; }
        const int64_t nu = (int64_t)h[WRing::kUndecided];
        if (nu == 0) break;
        if (++rounds > m + 1) { rc = FL_ETIMEOUT; set_error(rc, "weighted MIS did not converge"); break; }
        const int64_t H = (int64_t)h[WRing::kMaxB];
        auto timed = [&](int kind, int64_t t_end, int64_t steps, clock::time_point t0) {
            const double us = std::chrono::duration<double, std::micro>(clock::now() - t0).count();
            s->mis_log.insert(s->mis_log.end(), {rounds, (int64_t)kind, t_end, steps, 0, (int64_t)us});
        };
        int64_t t_end = 0, steps = 0;
        // cover
        auto t0 = clock::now();
        WSweep a = ring.sweep(g);
        a.lab = cover;
        a.ft = ft;
        e = cudaMemsetAsync(cover, 0xff, (size_t)n * 4, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(ft, 0xff, (size_t)n * 4, st);
        if (e != cudaSuccess) { rc = status_of(e, "weighted MIS", __FILE__, __LINE__); break; }
        // candidates of a larger B_f than any undecided one have been decided
        if ((rc = run_sweep(g, ring, a, H, WEntry{fac_by_ord, bsort, state, m, false, nullptr, nullptr}, kProfMis,
                            &t_end, &steps)))
            break;
        timed(0, t_end, steps, t0);
        // gather
        t0 = clock::now();
        a.lab = lab;
        a.dl = bcap;
        a.dlab = dlab;
        a.ft = nullptr;
        a.fts = ft;
        e = cudaMemsetAsync(lab, 0xff, (size_t)n * 8, st);  // lab and dlab
        if (e != cudaSuccess) { rc = status_of(e, "weighted MIS", __FILE__, __LINE__); break; }
        if ((rc = run_sweep(g, ring, a, H, WEntry{nullptr, nullptr, nullptr, 0, true, cover, s->client.as<uint8_t>()},
                            kProfMis, &t_end, &steps)))
            break;
        timed(1, t_end, steps, t0);
        if (m > 0)
            FL_LAUNCH(kProfMis, k_wdecide<<<grid_for(m, 256), 256, 0, st>>>(fac_by_ord, m, dlab, state,
                                                                            c + WRing::kJoined, c));
        FL_LAUNCH(kProfMis, k_wclaim<<<grid_for(n, 256), 256, 0, st>>>(n, s->client.as<uint8_t>(), cover, fac_by_ord,
                                                                       state, s->claimed.as<uint8_t>(),
                                                                       s->kill.as<uint8_t>(), c + WRing::kClaimed));
        e = cudaMemcpyAsync(h, c + WRing::kJoined, 16, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) { rc = status_of(e, "weighted MIS", __FILE__, __LINE__); break; }
        const int64_t joined = (int64_t)h[0], claimed = (int64_t)h[1];
        if (joined == 0) { rc = FL_ECUDA; set_error(rc, "weighted MIS: a round decided nothing"); break; }
        // kill
        if (nu > joined && claimed > 0) {
            t0 = clock::now();
            e = cudaMemsetAsync(lab, 0xff, (size_t)n * 8, st);
            if (e != cudaSuccess) { rc = status_of(e, "weighted MIS", __FILE__, __LINE__); break; }
            if ((rc = run_sweep(g, ring, a, H,
                                WEntry{nullptr, nullptr, nullptr, 0, true, nullptr, s->kill.as<uint8_t>()}, kProfMis,
                                &t_end, &steps)))
                break;
            timed(4, t_end, steps, t0);
            FL_LAUNCH(kProfMis, k_wkill<<<grid_for(m, 256), 256, 0, st>>>(fac_by_ord, m, dlab, state));
        }
        s->mis_log.insert(s->mis_log.end(),
                          {rounds, 3, H, nu, joined,
                           (int64_t)std::chrono::duration<double, std::micro>(clock::now() - round_t0).count()});
    }
    if (rc == FL_OK) {
        unsigned long long no = 0;
        cudaError_t e = cudaMemsetAsync(c + WRing::kOpen, 0, 8, st);
        if (e == cudaSuccess) {
            FL_LAUNCH(kProfMis, k_wopen<<<grid_for(n, 256), 256, 0, st>>>(state, n, s->open.as<uint8_t>(), c + WRing::kOpen));
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaMemcpyAsync(&no, c + WRing::kOpen, 8, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) rc = status_of(e, "weighted MIS", __FILE__, __LINE__);
        s->n_open = (int64_t)no;
        s->mis_rounds = rounds;
    }
    ring.release(st);
    return rc;
}

int assign_weighted(fl_solve* s) {
    fl_graph* g = s->g;
    const int64_t n = g->n;
    cudaStream_t st = g->stream;
    FL_TRY(dalloc(s->assign, (size_t)n * 4));
    FL_TRY(dalloc(s->dist, (size_t)n * 4));
    FL_TRY(dalloc(s->kill, (size_t)n));
    FL_CUDA(cudaMemsetAsync(s->assign.p, 0xff, (size_t)n * 4, st));
    FL_CUDA(cudaMemsetAsync(s->dist.p, 0xff, (size_t)n * 4, st));
    FL_CUDA(cudaMemsetAsync(s->kill.p, 0, (size_t)n, st));
    WRing ring;
    int rc = ring.alloc(g);
    if (rc == FL_OK) {
        WSweep a = ring.sweep(g);
        a.lab = s->assign.as<uint32_t>();  // facility id; kNone reads as -1
        a.dist = s->dist.as<int32_t>();
        a.past = s->kill.as<uint8_t>();
        a.first = 1;
        int64_t t_end = 0, steps = 0;
        rc = run_sweep(g, ring, a, 2147483647LL,
                       WEntry{nullptr, nullptr, nullptr, 0, true, nullptr, s->open.as<uint8_t>()}, kProfBfs, &t_end,
                       &steps);
        unsigned long long err = 0;
        if (rc == FL_OK) {
            FL_LAUNCH(kProfBfs, k_wbeyond<<<grid_for(n, 256), 256, 0, st>>>(n, s->kill.as<uint8_t>(), a.lab,
                                                                           ring.c));
            cudaError_t e = cudaMemcpyAsync(&err, ring.c, 8, cudaMemcpyDeviceToHost, st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
            if (e != cudaSuccess) rc = status_of(e, "weighted assignment", __FILE__, __LINE__);
        }
        if (rc == FL_OK && (err & 2ULL)) {
            rc = FL_EINVAL;
            set_error(rc, "weighted assignment: a distance above 2^31 - 1");
        }
    }
    ring.release(st);
    return rc;
}

}  // namespace fl

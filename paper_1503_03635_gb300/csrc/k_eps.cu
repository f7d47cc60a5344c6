// k_eps.cu -- the opening phase with eps > 0 (Section 4.1, Algorithm 3;
// Section 4.2, Algorithms 4 and 5 with Eq. 2/3) and the selection of
// Algorithm 6 (Section 4.3).
//
// The phase runs on a grid of radii alpha_j = alpha_{j-1} (1 + eps) from
// alpha_0 = gamma (1 + eps) / m^2, m = |F||C|, gamma = max over clients that
// reach a facility of min_f (c(f) + d(c, f)).  In iteration j every unopened
// facility whose q(f) reaches c(f) opens (alpha(f) = alpha_j), then every
// unfrozen client with an open facility within (1 + eps) alpha_j freezes
// (alpha(c) = alpha_j).  q(f) is what Eq. 2 (first iteration) and Eq. 3
// (later ones) add up to: per client c of f's ADS (HIP-weighted), with d_c
// the smallest grid value >= d(c, f),
//     [d_c <= alpha(c)] ((1 + eps) alpha(c) - d_c),
// alpha(c) the current radius for unfrozen clients, else the one at which c
// froze; it is summed in ADS order with one IEEE operation per step.
//
// Nothing changes between iterations without an opening or a freezing, so the
// GPU jumps from event to event: for fixed frozen clients q(f) is
// non-decreasing in j (each rounded step is monotone), so the first
// iteration at which f opens is found by binary search over the grid, and the
// first at which a client freezes by binary search over (1 + eps) alpha_j.
// The next event is the smallest of them; its openings and freezings are
// applied and the search repeats.  The result is the iteration-by-iteration
// loop's.  Freezing a client can only lower q_j(f), so the iteration found for
// a facility is a lower bound at every later event: a facility is looked at
// again only while its bound is not above the next event found so far, and
// most keep their bound.  Distances to the open set only fall, so an event
// spreads from the facilities it opened alone.  The whole event loop is one
// resident kernel, some seven grid barriers per event.  R-MAT, 65 k vertices,
// eps = 0.1, 58 events: a full search per facility, a BFS from every open
// facility, and four looks by the host per event took about 10 ms, the kernel
// takes 2.4.
//
// Selection: H joins a client c to an open facility f iff alpha(c) =
// alpha(f) and d(c, f) <= (1 + eps) alpha(c), so facilities opened in
// different iterations never share a client.  Each iteration's facilities
// are selected by the lexicographically-first MIS under pi, with balls of
// floor((1 + eps) alpha_j) hops over the clients frozen in that iteration:
// the MIS machinery of the epsilon -> 0 path, run once per iteration that
// opened two or more facilities.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
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

constexpr int64_t kMaxGrid = 1 << 22;      // the grid of radii, at most
constexpr int32_t kNever = 0x7fffffff;

__device__ __forceinline__ unsigned long long dbits(double x) { return (unsigned long long)__double_as_longlong(x); }
__device__ __forceinline__ double bitsd(unsigned long long x) { return __longlong_as_double((long long)x); }

// Facilities, clients and the largest finite opening cost.
__global__ void k_eps_counts(const double* __restrict__ cost, const uint8_t* __restrict__ client, int64_t n,
                             unsigned long long* __restrict__ out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long nf = 0, nc = 0, mx = 0;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const double c = cost[v];
        if (c < INFINITY) {
            ++nf;
            mx = max(mx, dbits(c));  // positive doubles order as their bits
        }
        nc += client[v] ? 1ULL : 0ULL;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        nf += __shfl_xor_sync(kFull, nf, o);
        nc += __shfl_xor_sync(kFull, nc, o);
        mx = max(mx, __shfl_xor_sync(kFull, mx, o));
    }
    if (lane_id() == 0) {
        if (nf) atomicAdd(&out[0], nf);
        if (nc) atomicAdd(&out[1], nc);
        if (mx) atomicMax(&out[2], mx);
    }
}

// gamma, step d: M[v] = the smallest cost of a facility within d hops of v
// (as bits: positive doubles order as their bits, +inf for none); a client's
// gamma_c = min over d of fl(M + d), which equals min over facilities of
// fl(c(f) + d(c, f)) because rounded addition is monotone in each operand.
//
// Mn starts as M where there are segments.  A warp per row, and per segment of a row
// above `seg` entries: the largest hub's warp was the whole round.  R-MAT, 65 k vertices: 62 us a round
// with a warp per row, 16 now; the solve on R-MAT scale 20, eps = 1, 16.4 -> 13.3 ms.
__global__ void __launch_bounds__(256) k_eps_min_pull(const int64_t* __restrict__ rowp,
                                                      const int32_t* __restrict__ cols, int64_t n,
                                                      const int32_t* __restrict__ seg_hub, int64_t n_seg,
                                                      const int64_t* __restrict__ hub_seg,
                                                      const int32_t* __restrict__ hub_list, int seg,
                                                      const unsigned long long* __restrict__ M,
                                                      unsigned long long* __restrict__ Mn,
                                                      unsigned long long* __restrict__ changed) {
    const int lane = lane_id();
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    bool ch = false;
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n_seg + n; i += warps) {
        const int32_t hub = i < n_seg ? seg_hub[i] : 0;
        const int64_t v = i < n_seg ? hub_list[hub] : i - n_seg;
        int64_t e0 = rowp[v], e1 = rowp[v + 1];
        if (i < n_seg) {
            e0 += (i - hub_seg[hub]) * seg;
            e1 = min(e1, e0 + seg);
        } else if (e1 - e0 > seg) {
            continue;
        }
        const unsigned long long own = M[v];
        unsigned long long m = own;
        for (int64_t e = e0 + lane; e < e1; e += 32) m = min(m, __ldg(&M[cols[e]]));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = min(m, __shfl_xor_sync(kFull, m, o));
        ch |= m < own;
        if (lane == 0) {
            if (i >= n_seg) Mn[v] = m;
            else if (m < own) atomicMin(&Mn[v], m);
        }
    }
    if (__syncthreads_or(ch) && threadIdx.x == 0) *changed = 1;
}

__global__ void k_eps_gamma_step(const unsigned long long* __restrict__ M, const uint8_t* __restrict__ client,
                                 int64_t n, double d, double* __restrict__ gam) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        if (!client[v]) continue;
        const double m = bitsd(M[v]);
        if (!(m < INFINITY)) continue;
        const double t = __dadd_rn(m, d);
        if (t < gam[v]) gam[v] = t;
    }
}

// gamma = max over clients with a facility in reach; their number.
__global__ void k_eps_gamma_max(const double* __restrict__ gam, const uint8_t* __restrict__ client, int64_t n,
                                unsigned long long* __restrict__ out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long mx = 0, cnt = 0;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        if (client[v] && gam[v] < INFINITY) {
            mx = max(mx, dbits(gam[v]));
            ++cnt;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mx = max(mx, __shfl_xor_sync(kFull, mx, o));
        cnt += __shfl_xor_sync(kFull, cnt, o);
    }
    if (lane_id() == 0) {
        if (mx) atomicMax(&out[0], mx);
        if (cnt) atomicAdd(&out[1], cnt);
    }
}

struct EpsADS {
    const int64_t* __restrict__ gofs;
    const int64_t* __restrict__ eofs;
    const uint32_t* __restrict__ ginfo;
    const double* __restrict__ gwt;
    const int32_t* __restrict__ eid;
};

// q_j(f) by the closed form (see the top of this file).  who[w]: -2 no client, -1
// an unfrozen one, else the iteration at which it froze (written by the kernel
// that calls this); reach[j] = (1 + eps) alpha_j.  The unfrozen clients of a
// group add the same term, which is worked out once: one FP64 operation per
// entry in place of four, on a pipe of some two lanes per SM.
__device__ double eps_q(const EpsADS& a, int64_t f, int32_t j, const double* __restrict__ grid,
                        const double* __restrict__ reach, const int32_t* __restrict__ shell, int32_t nshell,
                        const int32_t* who) {
    double q = 0.0;
    int64_t e = a.eofs[f];
    const double reach_j = __ldg(&reach[j]);
    for (int64_t gi = a.gofs[f]; gi < a.gofs[f + 1]; ++gi) {
        const uint32_t info = a.ginfo[gi];
        const int hop = (int)(info & 0xffffu), cnt = (int)((info >> 16) & 0xffu), counted = (int)(info >> 24);
        const double wt = a.gwt[gi];
        const int32_t sj = hop < nshell ? shell[hop] : kNever;
        // a client whose radius is below the group's shell adds nothing
        const double gs = sj != kNever ? __ldg(&grid[sj]) : 0.0;
        const double unfrozen = sj <= j ? __dmul_rn(wt, __dsub_rn(reach_j, gs)) : 0.0;
        for (int i = 0; i < counted; i += 4) {
            int32_t w[4];
#pragma unroll
            for (int l = 0; l < 4; ++l) w[l] = i + l < counted ? a.eid[e + i + l] : -1;
#pragma unroll
            for (int l = 0; l < 4; ++l) w[l] = w[l] >= 0 ? __ldcg(&who[w[l]]) : -2;
#pragma unroll
            for (int l = 0; l < 4; ++l) {
                if (w[l] == -1) {
                    if (sj <= j) q = __dadd_rn(q, unfrozen);
                } else if (w[l] >= 0 && sj <= w[l]) {
                    q = __dadd_rn(q, __dmul_rn(wt, __dsub_rn(__ldg(&reach[w[l]]), gs)));
                }
            }
        }
        e += cnt;
    }
    return q;
}

// Control block of the event loop (device, zero at its start).
struct EpsCtl {
    GridBar bar;                   // its err: 2: more events than iterations; 4: the level cap
    int32_t jmin[3];               // next event's iteration (event number mod 3)
    unsigned pad;
    unsigned long long cnt[4];     // frontier list lengths (number of the pass mod 4)
    long long events, jcur;
};

constexpr int kELong = 512;   // longer rows are spread by the whole block
constexpr int kEQueue = 128;  // of them, queued per block and level

struct EpsArgs {
    const int64_t* rowp;
    const int32_t* cols;
    int64_t n;
    const int32_t* fac;
    int64_t n_fac;
    const double* cost;
    const uint8_t* client;
    const double* gam;
    EpsADS ads;
    const double* grid;
    const double* reach;
    const int32_t* shell;
    int32_t nshell, J;
    int32_t* fac_iter;
    int32_t* cli_iter;
    int32_t* who;       // cli_iter for the clients, -2 for the others
    int32_t* nxt;       // lower bound on the iteration at which each facility opens
    uint32_t* dist;     // hops to the open set (all ones: none in reach)
    int32_t* list[2];
    int2* openings;     // (iteration, facilities opened) of each event
    long long unfrozen;
    int64_t cap;        // BFS levels at most (a search from every open facility would need one more than the largest distance)
    EpsCtl* c;
};

// The events: see the top of this file.
__global__ void __launch_bounds__(kResThreads, 1) k_eps_events(EpsArgs a) {
    __shared__ int32_t s_v[kEQueue];
    __shared__ unsigned s_queued;
    EpsCtl* c = a.c;
    const int lane = lane_id();
    const int64_t tid = (int64_t)blockIdx.x * kResThreads + threadIdx.x, threads = (int64_t)gridDim.x * kResThreads;
    const int64_t item0 = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x, warps = threads >> 5;
    unsigned pass = 0, total = 0, lists = 0;  // lists: frontier lists filled
    long long unopened = a.n_fac, unfrozen = a.unfrozen, events = 0;
    int32_t jcur = 0;
    if (threadIdx.x == 0) s_queued = 0;
    for (int64_t i = tid; i < a.n_fac; i += threads) a.nxt[a.fac[i]] = 1;
    for (int64_t v = tid; v < a.n; v += threads) a.who[v] = a.client[v] ? -1 : -2;
    if (tid < 3) c->jmin[tid] = kNever;
    if (!end_pass(&c->bar, pass, 0, &total)) return;

    auto q = [&](int32_t f, int32_t j) {
        return eps_q(a.ads, f, j, a.grid, a.reach, a.shell, a.nshell, a.who);
    };
    // u at distance L through a frontier vertex: into the list of the next level
    auto offer = [&](int64_t e, int64_t end, uint32_t L) {
        bool fresh = false;
        int32_t u = 0;
        if (e < end) {
            u = __ldg(&a.cols[e]);
            if (__ldcg(&a.dist[u]) > L) fresh = atomicMin(&a.dist[u], L) > L;
        }
        const long long at = warp_append(fresh, &c->cnt[lists & 3]);
        if (at >= 0) a.list[lists & 1][at] = u;
        return fresh;
    };
    while (unopened > 0 && unfrozen > 0) {
        int32_t* jmin = &c->jmin[events % 3];  // holds the next freezing
        if (tid == 0) c->jmin[(events + 1) % 3] = kNever;
        // ---- the next opening
        if (jcur < a.J)
            for (int64_t i = tid; i < a.n_fac; i += threads) {
                const int32_t f = a.fac[i];
                if (__ldcg(&a.fac_iter[f]) >= 0) continue;
                const int32_t lb = max(__ldcg(&a.nxt[f]), jcur + 1), top = min(a.J, __ldcg(jmin));
                if (lb > top) continue;
                const double cf = a.cost[f];
                int32_t res;
                if (q(f, lb) >= cf) {
                    res = lb;
                } else if (lb == top || !(q(f, top) >= cf)) {
                    a.nxt[f] = top < a.J ? top + 1 : kNever;  // a bound, above this event
                    continue;
                } else {
                    int32_t lo = lb + 1, hi = top;
                    while (lo < hi) {
                        const int32_t mid = lo + (hi - lo) / 2;
                        if (q(f, mid) >= cf) hi = mid;
                        else lo = mid + 1;
                    }
                    res = lo;
                }
                a.nxt[f] = res;
                atomicMin(jmin, res);
            }
        if (!end_pass(&c->bar, pass, 0, &total)) return;
        const int32_t js = __ldcg(jmin);
        if (js == kNever) {
            jcur = a.J;  // nothing changes any more up to the last radius of the grid
            break;
        }
        ++events;
        if (events > (long long)a.J + 1) {
            if (tid == 0) c->bar.err = 2;
            return;
        }
        // ---- its facilities open (a bound equal to js was confirmed above)
        unsigned opened = 0;
        if (tid == 0) c->cnt[(lists + 1) & 3] = 0;
        for (int64_t b = (tid >> 5) * 32; b < a.n_fac; b += warps * 32) {
            const int32_t f = b + lane < a.n_fac ? a.fac[b + lane] : -1;
            const bool now = f >= 0 && __ldcg(&a.fac_iter[f]) < 0 && __ldcg(&a.nxt[f]) == js;
            if (now) {
                a.fac_iter[f] = js;
                a.dist[f] = 0u;
                ++opened;
            }
            const long long at = warp_append(now, &c->cnt[lists & 3]);
            if (at >= 0) a.list[lists & 1][at] = f;
        }
        if (!end_pass(&c->bar, pass, opened, &total)) return;
        if (tid == 0) a.openings[events - 1] = make_int2(js, (int)total);
        unopened -= (long long)total;
        // ---- distances to the open set
        for (uint32_t L = 1; total; ++L) {
            const int32_t* list = a.list[lists & 1];
            const int64_t n_front = (int64_t)total;
            ++lists;
            if (tid == 0) c->cnt[(lists + 1) & 3] = 0;
            unsigned found = 0;
            for (int64_t i = item0; i < n_front; i += warps) {
                const int32_t v = __ldcg(&list[i]);
                const int64_t beg = __ldg(&a.rowp[v]), end = __ldg(&a.rowp[v + 1]);
                if (end - beg > kELong) {
                    unsigned at = 0;
                    if (lane == 0) at = atomicAdd(&s_queued, 1u);
                    at = __shfl_sync(kFull, at, 0);
                    if (at < kEQueue) {
                        if (lane == 0) s_v[at] = v;
                        continue;
                    }
                }
                for (int64_t e = beg; e < end; e += 32) found += offer(e + lane, end, L);
            }
            __syncthreads();
            const int queued = (int)min(s_queued, (unsigned)kEQueue);
            for (int x = 0; x < queued; ++x) {
                const int64_t end = __ldg(&a.rowp[s_v[x] + 1]);
                for (int64_t e = __ldg(&a.rowp[s_v[x]]) + (threadIdx.x & ~31); e < end; e += kResThreads)
                    found += offer(e + lane, end, L);
            }
            __syncthreads();
            if (threadIdx.x == 0) s_queued = 0;
            if (!end_pass(&c->bar, pass, found, &total)) return;
        }
        ++lists;
        // ---- its clients freeze; the next freezing of the others
        unsigned frozen = 0;
        int32_t next = kNever;
        const double reach_j = __ldg(&a.reach[js]);
        for (int64_t v = tid; v < a.n; v += threads) {
            const uint32_t du = __ldcg(&a.dist[v]);
            if ((int32_t)du < 0) continue;
            if ((int64_t)du >= a.cap) atomicOr(&c->bar.err, 4u);
            if (__ldcg(&a.who[v]) != -1 || !(a.gam[v] < INFINITY)) continue;
            const double d = (double)du;
            if (d <= reach_j) {
                a.cli_iter[v] = a.who[v] = js;
                ++frozen;
            } else if (js < a.J && __ldg(&a.reach[a.J]) >= d) {
                int32_t lo = js + 1, hi = min(a.J, next);
                if (!(__ldg(&a.reach[hi]) >= d)) continue;  // later than this thread's earliest
                while (lo < hi) {
                    const int32_t mid = lo + (hi - lo) / 2;
                    if (__ldg(&a.reach[mid]) >= d) hi = mid;
                    else lo = mid + 1;
                }
                next = lo;
            }
        }
        next = (int32_t)__reduce_min_sync(kFull, (unsigned)next);
        if (lane == 0 && next != kNever) atomicMin(&c->jmin[events % 3], next);
        if (!end_pass(&c->bar, pass, frozen, &total)) return;
        if (__ldcg(&c->bar.err)) return;
        unfrozen -= (long long)total;
        jcur = js;
    }
    if (tid == 0) {
        c->events = events;
        c->jcur = jcur;
    }
}

// The facility list (finite costs).
__global__ void k_eps_facilities(const double* __restrict__ cost, int64_t n, int32_t* __restrict__ fac,
                                 unsigned long long* __restrict__ cnt) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
        const int64_t v = base + lane_id();
        const bool in = v < n && cost[v] < INFINITY;
        const long long at = warp_append(in, cnt);
        if (at >= 0) fac[at] = (int32_t)v;
    }
}

// Inputs of one iteration's selection: radius (1 + eps) alpha_j for its
// facilities (+inf for the others), its frozen clients as the client mask;
// facilities alone in their iteration are selected directly.
__global__ void k_eps_group(const int32_t* __restrict__ fac_iter, const int32_t* __restrict__ cli_iter, int64_t n,
                            int32_t j, double r, double* __restrict__ radii, uint8_t* __restrict__ gclient) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        radii[v] = fac_iter[v] == j ? r : INFINITY;
        gclient[v] = cli_iter[v] == j ? 1 : 0;
    }
}

__global__ void k_eps_or(const uint8_t* __restrict__ open, int64_t n, uint8_t* __restrict__ acc) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride)
        if (open[v]) acc[v] = 1;
}

__global__ void k_eps_single(const int32_t* __restrict__ fac_iter, int64_t n, const uint8_t* __restrict__ multi,
                             uint8_t* __restrict__ acc) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride)
        if (fac_iter[v] >= 0 && !multi[fac_iter[v]]) acc[v] = 1;
}

// Final open set and its list (for the assignment).
__global__ void k_eps_finish(const uint8_t* __restrict__ acc, int64_t n, uint8_t* __restrict__ open,
                             int32_t* __restrict__ list, unsigned long long* __restrict__ cnt) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
        const int64_t v = base + lane_id();
        const bool o = v < n && acc[v] != 0;
        if (v < n) open[v] = o ? 1 : 0;
        const long long at = warp_append(o, cnt);
        if (at >= 0) list[at] = (int32_t)v;
    }
}

__global__ void k_eps_fill(double* __restrict__ a, int64_t n, double x) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) a[v] = x;
}

int read_u64(const unsigned long long* d, unsigned long long* h, int cnt, cudaStream_t st) {
    FL_CUDA(cudaMemcpyAsync(h, d, (size_t)cnt * 8, cudaMemcpyDeviceToHost, st));
    FL_CUDA(cudaStreamSynchronize(st));
    return FL_OK;
}

}  // namespace

int open_facilities_eps(fl_solve* s, double eps) {
    fl_graph* g = s->g;
    const int64_t n = g->n;
    cudaStream_t st = g->stream;
    const double onepe = 1.0 + eps;
    const double* cost = s->cost.as<double>();
    const uint8_t* client = s->client.as<uint8_t>();
    // scratch: fac_iter, cli_iter, nxt, facility list, dist, two frontier lists
    // (int32); gamma (double); M[2] (uint64); selected (uint8); counters
    DBuf& E = s->eps;
    const size_t i32n = (size_t)n * 4;
    const size_t off_gam = ((i32n * 7 + 255) / 256) * 256;  // 8-byte values start aligned
    const size_t off_M = off_gam + (size_t)n * 8, off_acc = off_M + (size_t)n * 16;
    const size_t off_ctr = ((off_acc + (size_t)n + 255) / 256) * 256;
    FL_TRY(dalloc(E, off_ctr + 256));
    char* base = E.as<char>();
    int32_t* fac_iter = reinterpret_cast<int32_t*>(base);
    int32_t* cli_iter = fac_iter + n;
    int32_t* nxt = cli_iter + n;
    int32_t* fac = nxt + n;
    int32_t* dist = fac + n;
    int32_t* list[2] = {dist + n, dist + 2 * n};  // frontier lists
    double* gam = reinterpret_cast<double*>(base + off_gam);
    unsigned long long* M[2] = {reinterpret_cast<unsigned long long*>(base + off_M),
                                reinterpret_cast<unsigned long long*>(base + off_M) + n};
    uint8_t* acc = reinterpret_cast<uint8_t*>(base + off_acc);
    unsigned long long* ctr = reinterpret_cast<unsigned long long*>(base + off_ctr);
    FL_CUDA(cudaMemsetAsync(fac_iter, 0xff, i32n * 2, st));
    FL_CUDA(cudaMemsetAsync(dist, 0xff, i32n, st));
    FL_CUDA(cudaMemsetAsync(acc, 0, (size_t)n, st));
    FL_CUDA(cudaMemsetAsync(ctr, 0, 256, st));
    s->eps_gamma = -1.0;
    s->eps_alpha0 = 0.0;
    s->eps_iterations = 0;
    s->eps_events = 0;
    s->eps_groups = 0;
    unsigned long long h[4] = {0, 0, 0, 0};

    // the selected set -> s->open and its list -> s->ulist (for the assignment)
    auto finish = [&]() -> int {
        FL_TRY(dalloc(s->open, (size_t)n));
        FL_TRY(dalloc(s->ulist, (size_t)n * 8));
        FL_CUDA(cudaMemsetAsync(&ctr[8], 0, 8, st));
        FL_LAUNCH(kProfMis, k_eps_finish<<<grid_for(n, 256), 256, 0, st>>>(acc, n, s->open.as<uint8_t>(),
                                                                             s->ulist.as<int32_t>(), &ctr[8]));
        unsigned long long no = 0;
        FL_TRY(read_u64(&ctr[8], &no, 1, st));
        s->n_open = (int64_t)no;
        return FL_OK;
    };

    // |F|, |C|, the largest finite cost
    FL_LAUNCH(kProfMis, k_eps_counts<<<grid_for(n, 256), 256, 0, st>>>(cost, client, n, ctr));
    FL_TRY(read_u64(ctr, h, 3, st));
    const int64_t nF = (int64_t)h[0], nC = (int64_t)h[1];
    double max_cost = 0.0;
    std::memcpy(&max_cost, &h[2], 8);
    if (nF == 0 || nC == 0) return finish();

    // gamma: rounds of min-propagation of the costs
    if (!g->lists_ready) {
        FL_TRY(build_work_lists(g));
        g->lists_ready = 1;
    }
    FL_LAUNCH(kProfMis, k_eps_fill<<<grid_for(n, 256), 256, 0, st>>>(gam, n, INFINITY));
    FL_CUDA(cudaMemcpyAsync(M[0], cost, (size_t)n * 8, cudaMemcpyDeviceToDevice, st));
    FL_LAUNCH(kProfMis, k_eps_gamma_step<<<grid_for(n, 256), 256, 0, st>>>(M[0], client, n, 0.0, gam));
    int cur = 0;
    for (int64_t d = 1;; ++d) {
        if (d > n + 1) FL_FAIL(FL_ETIMEOUT, "epsilon phase: cost propagation did not settle");
        FL_CUDA(cudaMemsetAsync(&ctr[3], 0, 8, st));
        if (g->n_seg > 0)
            FL_CUDA(cudaMemcpyAsync(M[cur ^ 1], M[cur], (size_t)n * 8, cudaMemcpyDeviceToDevice, st));
        FL_LAUNCH(kProfMis, k_eps_min_pull<<<std::min(grid_for(n + g->n_seg, 8), 152 * 8), 256, 0, st>>>(
                                g->rowp.as<int64_t>(), g->cols.as<int32_t>(), n, g->seg_hub.as<int32_t>(), g->n_seg,
                                g->hub_seg.as<int64_t>(), g->hub_list.as<int32_t>(), g->seg, M[cur], M[cur ^ 1],
                                &ctr[3]));
        FL_LAUNCH(kProfMis, k_eps_gamma_step<<<grid_for(n, 256), 256, 0, st>>>(M[cur ^ 1], client, n, (double)d,
                                                                                 gam));
        cur ^= 1;
        FL_TRY(read_u64(&ctr[3], h, 1, st));
        if (h[0] == 0) break;
    }
    FL_CUDA(cudaMemsetAsync(&ctr[4], 0, 16, st));
    FL_LAUNCH(kProfMis, k_eps_gamma_max<<<grid_for(n, 256), 256, 0, st>>>(gam, client, n, &ctr[4]));
    FL_TRY(read_u64(&ctr[4], h, 2, st));
    if (h[1] == 0) return finish();  // no client reaches a facility
    double gamma = 0.0;
    std::memcpy(&gamma, &h[0], 8);
    const int64_t unfrozen = (int64_t)h[1];
    s->eps_gamma = gamma;

    // the grid of radii, (1 + eps) alpha_j, and the shell of every hop distance
    const double m = (double)nF * (double)nC;
    const double alpha0 = (gamma * onepe) / (m * m);
    s->eps_alpha0 = alpha0;
    const double bound = 2.0 * (max_cost + (double)n + 1.0);
    std::vector<double> grid(1, alpha0);
    while (grid.back() < bound) {
        if ((int64_t)grid.size() >= kMaxGrid) FL_FAIL(FL_EINVAL, "eps too small: the grid of radii exceeds 2^22 values");
        grid.push_back(grid.back() * onepe);
    }
    const int32_t J = (int32_t)grid.size() - 1;
    std::vector<double> reach(grid.size());
    for (size_t j = 0; j < grid.size(); ++j) reach[j] = onepe * grid[j];
    const int32_t nshell = (int32_t)g->hops + 1;
    std::vector<int32_t> shell(nshell);
    for (int32_t hop = 0; hop < nshell; ++hop)
        shell[hop] = (int32_t)(std::lower_bound(grid.begin(), grid.end(), (double)hop) - grid.begin());
    FL_TRY(dalloc(s->eps_tab, grid.size() * 17 + (size_t)nshell * 4 + 64));
    double* grid_d = s->eps_tab.as<double>();
    double* reach_d = grid_d + grid.size();
    int32_t* shell_d = reinterpret_cast<int32_t*>(reach_d + grid.size());
    uint8_t* multi_d = reinterpret_cast<uint8_t*>(shell_d + nshell);
    FL_CUDA(cudaMemcpyAsync(grid_d, grid.data(), grid.size() * 8, cudaMemcpyHostToDevice, st));
    FL_CUDA(cudaMemcpyAsync(reach_d, reach.data(), reach.size() * 8, cudaMemcpyHostToDevice, st));
    FL_CUDA(cudaMemcpyAsync(shell_d, shell.data(), (size_t)nshell * 4, cudaMemcpyHostToDevice, st));

    // the facilities
    FL_CUDA(cudaMemsetAsync(&ctr[6], 0, 8, st));
    FL_LAUNCH(kProfMis, k_eps_facilities<<<grid_for(n, 256), 256, 0, st>>>(cost, n, fac, &ctr[6]));
    EpsADS ads;
    ads.gofs = g->gofs.as<int64_t>();
    ads.eofs = g->eofs.as<int64_t>();
    ads.ginfo = g->ginfo.as<uint32_t>();
    ads.gwt = g->gwt.as<double>();
    ads.eid = g->eid.as<int32_t>();

    // events: the next iteration at which a facility opens or a client freezes
    std::vector<std::pair<int32_t, int64_t>> openings;  // (iteration, facilities opened)
    {
        EpsArgs a;
        a.rowp = g->rowp.as<int64_t>();
        a.cols = g->cols.as<int32_t>();
        a.n = n;
        a.fac = fac;
        a.n_fac = nF;
        a.cost = cost;
        a.client = client;
        a.gam = gam;
        a.ads = ads;
        a.grid = grid_d;
        a.reach = reach_d;
        a.shell = shell_d;
        a.nshell = nshell;
        a.J = J;
        a.fac_iter = fac_iter;
        a.cli_iter = cli_iter;
        a.who = reinterpret_cast<int32_t*>(M[0]);  // the costs have been spread
        a.nxt = nxt;
        a.dist = reinterpret_cast<uint32_t*>(dist);
        a.list[0] = list[0];
        a.list[1] = list[1];
        a.unfrozen = unfrozen;
        a.cap = g->sched.level_cap > 0 ? g->sched.level_cap : n + 2;
        const size_t ctl_b = (sizeof(EpsCtl) + 255) & ~(size_t)255;
        FL_TRY(dalloc(s->eps_ev, ctl_b + ((size_t)J + 2) * sizeof(int2)));
        a.c = s->eps_ev.as<EpsCtl>();
        a.openings = reinterpret_cast<int2*>(s->eps_ev.as<char>() + ctl_b);
        FL_CUDA(cudaMemsetAsync(a.c, 0, sizeof(EpsCtl), st));
        int dev = 0, sms = 0;
        FL_CUDA(cudaGetDevice(&dev));
        FL_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(sms, n / 64));
        void* args[] = {&a};
        cudaError_t le = cudaSuccess;
        FL_LAUNCH(kProfMis, le = cudaLaunchCooperativeKernel((const void*)k_eps_events, dim3(blocks),
                                                             dim3(kResThreads), args, 0, st));
        FL_CUDA(le);
        EpsCtl hc{};
        FL_CUDA(cudaMemcpyAsync(&hc, a.c, sizeof(EpsCtl), cudaMemcpyDeviceToHost, st));
        FL_CUDA(cudaStreamSynchronize(st));
        if (hc.bar.err & 2u) FL_FAIL(FL_ETIMEOUT, "epsilon phase: more events than iterations");
        if (hc.bar.err & 4u) FL_FAIL(FL_ETIMEOUT, "BFS reached its level cap");
        if (hc.bar.err) FL_FAIL(FL_ETIMEOUT, "epsilon phase: a barrier wait ran out");
        std::vector<int2> ev((size_t)hc.events);
        if (hc.events > 0) {
            FL_CUDA(cudaMemcpyAsync(ev.data(), a.openings, ev.size() * sizeof(int2), cudaMemcpyDeviceToHost, st));
            FL_CUDA(cudaStreamSynchronize(st));
        }
        for (const int2& o : ev)
            if (o.y > 0) openings.push_back({o.x, (int64_t)o.y});
        s->eps_events = hc.events;
        s->eps_iterations = hc.jcur;
    }

    // selection: one lexicographically-first MIS per iteration that opened
    // two or more facilities; the others' facilities are selected directly
    std::vector<uint8_t> multi(grid.size(), 0);
    for (const auto& o : openings)
        if (o.second >= 2) multi[o.first] = 1;
    FL_CUDA(cudaMemcpyAsync(multi_d, multi.data(), multi.size(), cudaMemcpyHostToDevice, st));
    FL_LAUNCH(kProfMis, k_eps_single<<<grid_for(n, 256), 256, 0, st>>>(fac_iter, n, multi_d, acc));
    FL_TRY(dalloc(s->eps_r, (size_t)n * 8));
    FL_TRY(dalloc(s->eps_c, (size_t)n));
    // All groups but the last are queued one behind the other (on graphs whose
    // selection is one launch), those that one launch did not finish run again
    // with the host's help; the last one runs like a plain selection and leaves
    // its log and counts.
    std::vector<size_t> groups;
    for (size_t i = 0; i < openings.size(); ++i)
        if (openings[i].second >= 2) groups.push_back(i);
    s->eps_groups = (int64_t)groups.size();
    FL_TRY(dalloc(s->eps_out, groups.size() * 4 + 16));
    int* outcome = s->eps_out.as<int>();
    auto select = [&](size_t i, bool queue, bool* queued) -> int {
        const auto& o = openings[groups[i]];
        FL_LAUNCH(kProfMis, k_eps_group<<<grid_for(n, 256), 256, 0, st>>>(fac_iter, cli_iter, n, o.first,
                                                                            reach[o.first], s->eps_r.as<double>(),
                                                                            s->eps_c.as<uint8_t>()));
        std::swap(s->radii, s->eps_r);
        std::swap(s->client, s->eps_c);
        *queued = false;
        int rc = queue ? open_facilities_queued(s, o.second, acc, outcome + i, queued) : FL_OK;
        if (rc == FL_OK && !*queued) rc = open_facilities(s);
        std::swap(s->radii, s->eps_r);
        std::swap(s->client, s->eps_c);
        FL_TRY(rc);
        if (!*queued)
            FL_LAUNCH(kProfMis, k_eps_or<<<grid_for(n, 256), 256, 0, st>>>(s->open.as<uint8_t>(), n, acc));
        return FL_OK;
    };
    std::vector<size_t> waiting;
    for (size_t i = 0; i < groups.size(); ++i) {
        const bool last = i + 1 == groups.size();
        if (last && !waiting.empty()) {
            std::vector<int> got(groups.size());
            FL_CUDA(cudaMemcpyAsync(got.data(), outcome, (i + 1) * 4, cudaMemcpyDeviceToHost, st));
            FL_CUDA(cudaStreamSynchronize(st));
            bool unused;
            for (size_t w : waiting)
                if (got[w] != 1) FL_TRY(select(w, false, &unused));
        }
        bool queued = false;
        FL_TRY(select(i, !last, &queued));
        if (queued) waiting.push_back(i);
    }
    FL_CUDA(cudaGetLastError());
    return finish();
}

// The iteration at which each vertex opened (as a facility) and froze (as a
// client) in the last epsilon phase of s (-1: never), internal numbering.
const int32_t* eps_iterations_of(const fl_solve* s, bool clients) {
    const int32_t* fi = s->eps.as<int32_t>();
    return clients ? fi + s->g->n : fi;
}

}  // namespace fl

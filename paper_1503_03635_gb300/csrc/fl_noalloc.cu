// fl_noalloc.cu -- nearest-open-facility assignment that allocates nothing.
//
// Some callers cannot let a library call cudaMalloc: applications that have
// reserved the whole device for their own memory pool (an allocation from
// elsewhere would fail or fragment it), and latency-critical loops for which
// an allocation's implicit device synchronisation is not acceptable.  For
// them this file offers the assignment step with its scratch memory (BFS
// values, two frontier lists, three frontier bitmaps, counters) in one
// file-scope device array of fixed size.  The caller passes the graph, the open set and the outputs.
//
// Every GPU that loads the library holds the array until the process exits.
// All calls share it and it keeps the last call's contents: each call clears
// what must start at zero.  Calls that overlap on the GPU (from several
// streams or threads) race on the array and give undefined results.
#include <algorithm>
#include <cstdio>
#include <mutex>

#include "fl_internal.cuh"

namespace fl {

// k_util.cu
__global__ void k_validate_csr(const int64_t* __restrict__ rowp, const int32_t* __restrict__ cols, int64_t n,
                               int64_t nnz, Counters* ctr);

namespace {

constexpr int64_t kMaxN = 1 << 20;  // largest graph the fixed scratch serves
constexpr int kMaxDevices = 64;

// Control block of the search (zero at its start).
struct NoallocCtl {
    GridBar bar;
    unsigned long long cnt[4];    // level L: vertices in its frontier list (L mod 4)
    unsigned long long edges[4];  // level L: CSR entries of its frontier's rows
    unsigned long long done;      // 1: the outputs are written
};

// X (8 B) + two frontier lists (4 B each) per vertex, three frontier bitmaps,
// then the control block and a Counters block (adjacent: one memset).
constexpr size_t kOffX = 0;
constexpr size_t kOffList = kOffX + 8 * kMaxN;
constexpr size_t kOffBm = kOffList + 8 * kMaxN;
constexpr size_t kOffCtl = kOffBm + 3 * (kMaxN / 8);
constexpr size_t kOffCtr = kOffCtl + 256;
constexpr size_t kScratchBytes = kOffCtr + 256;
static_assert(sizeof(Counters) <= 256, "the Counters block must fit its 256-byte slot of the scratch");
static_assert(sizeof(NoallocCtl) <= 256, "the control block must fit its 256-byte slot of the scratch");

static __device__ __align__(256) unsigned char noalloc_scratch[kScratchBytes];

std::mutex g_setup_mutex;
unsigned char* g_scratch_on[kMaxDevices] = {};

// Device address of the scratch array on the current device (looked up once
// per device, with that device current).
int scratch_address(unsigned char** out) {
    int dev = 0;
    FL_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) FL_FAIL(FL_EINVAL, "device index out of range");
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (!g_scratch_on[dev]) {
        void* p = nullptr;
        FL_CUDA(cudaGetSymbolAddress(&p, noalloc_scratch));
        g_scratch_on[dev] = static_cast<unsigned char*>(p);
    }
    *out = g_scratch_on[dev];
    return FL_OK;
}

// One cooperative launch runs the whole search: values, levels, outputs.
//
// X[v] = distance << 32 | label (~0: not reached).  Level L gives every vertex
// without a distance the smallest label among its neighbours at L - 1, by
// atomicMin; the lane that finds ~0 there appends the vertex to the next
// frontier list and sets its bit in the next frontier bitmap.
//   push (the frontier's rows hold less than 1/kPushDiv of the entries): a
//     warp per frontier row; rows above kLongRow entries are queued and taken
//     by the whole block, so that no warp walks a hub alone;
//   pull: every warp streams its equal share of the CSR entries, 32 rows at a
//     time (windows without an unreached row are passed over); the owner of an
//     entry is found among the window's 32 row ends, the neighbour's bit in a
//     copy of the frontier bitmap in shared memory, and entries of one row are
//     reduced in the warp before the atomic.
// What bounds it: the entries of unreached rows, read once per level from L2,
// and about 40 instructions per 32 entries; then a grid barrier per level.
// Before, a warp walked each frontier row alone, two launches and a look by
// the host per level: R-MAT, 500 k vertices, 16 M draws, 1 % open 2.62 ms per
// call (1.67 ms of it one launch that waits for the largest hub), now 0.35 ms;
// 167 k vertices 0.75 -> 0.20 ms, Erdos-Renyi, 12 k vertices 0.29 -> 0.12 ms.
constexpr int kPushDiv = 64;
constexpr int kLongRow = 512;
constexpr int kQueue = 256;   // long rows queued per block and level

struct NoallocArgs {
    const int64_t* rowp;
    const int32_t* cols;
    int64_t n, nnz;
    const uint8_t* open;
    unsigned long long* X;
    int32_t* list[2];
    uint32_t* bm[3];               // frontier bitmap of level L: bm[L % 3]
    NoallocCtl* c;
    const Counters* check;         // error != 0: the CSR did not pass, nothing is done
    int32_t* assign;
    int32_t* dist;
};

__global__ void __launch_bounds__(kResThreads, 1) k_noalloc_bfs(NoallocArgs a) {
    extern __shared__ uint32_t s_bm[];
    __shared__ int32_t s_queue[kQueue];
    __shared__ unsigned s_queued;
    __shared__ unsigned long long s_edges;
    if (a.check->error) return;
    NoallocCtl* c = a.c;
    const int lane = lane_id();
    const int64_t tid = (int64_t)blockIdx.x * kResThreads + threadIdx.x, threads = (int64_t)gridDim.x * kResThreads;
    const int64_t warp = tid >> 5, warps = threads >> 5;
    const int64_t words = (a.n + 31) >> 5;
    unsigned pass = 0, total = 0;

    // this warp's share of the entries, and the row that holds its first one
    const int64_t share = (a.nnz + warps - 1) / warps;
    const int64_t e0 = min(warp * share, a.nnz), e1 = min(e0 + share, a.nnz);
    int64_t row0 = 0;  // largest row with rowp[row] <= e0
    if (e0 < e1) {
        int64_t lo = 0, hi = a.n;  // rowp[lo] <= e0 < rowp[hi]
        while (hi - lo > 1) {
            const int64_t step = (hi - lo + 31) / 32;
            const int64_t p = lo + step * (lane + 1);
            const unsigned at_most = __ballot_sync(kFull, p < hi && a.rowp[p] <= e0);
            const int k = __popc(at_most);
            hi = min(hi, lo + step * (k + 1));
            lo += step * k;
        }
        row0 = lo;
    }

    // a vertex reached at this level: into the next frontier, its entries counted
    auto reach = [&](bool fresh, int32_t v, int64_t L, unsigned long long& edges, unsigned& found) {
        const long long at = warp_append(fresh, &c->cnt[L & 3]);
        if (!fresh) return;
        if (at < kMaxN) a.list[L & 1][at] = v;
        atomicOr(&a.bm[L % 3][v >> 5], 1u << (v & 31));
        edges += (unsigned long long)(a.rowp[v + 1] - a.rowp[v]);
        ++found;
    };
    // end of a level: the frontier's entries into c->edges, then the barrier
    auto end_level = [&](int64_t L, unsigned long long edges, unsigned found) -> bool {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) edges += __shfl_xor_sync(kFull, edges, o);
        if (lane == 0 && edges) atomicAdd(&s_edges, edges);
        __syncthreads();
        if (threadIdx.x == 0) {
            if (s_edges) atomicAdd(&c->edges[L & 3], s_edges);
            s_edges = 0;
            s_queued = 0;
        }
        return end_pass(&c->bar, pass, found, &total);
    };

    if (threadIdx.x == 0) s_edges = s_queued = 0;
    __syncthreads();
    {
        unsigned long long edges = 0;
        unsigned found = 0;
        for (int64_t b = warp * 32; b < a.n; b += warps * 32) {
            const int64_t v = b + lane;
            const bool src = v < a.n && a.open[v] != 0;
            if (v < a.n) a.X[v] = src ? (unsigned long long)v : ~0ULL;
            const unsigned m = __ballot_sync(kFull, src);
            if (lane == 0) {
                a.bm[0][b >> 5] = m;
                a.bm[1][b >> 5] = 0;
                a.bm[2][b >> 5] = 0;
            }
            const long long at = warp_append(src, &c->cnt[0]);
            if (src) {
                if (at < kMaxN) a.list[0][at] = (int32_t)v;
                edges += (unsigned long long)(a.rowp[v + 1] - a.rowp[v]);
                ++found;
            }
        }
        if (!end_level(0, edges, found)) return;
    }
    for (int64_t L = 1; total; ++L) {
        const int64_t n_front = min((int64_t)total, a.n);
        const unsigned long long fe = __ldcg(&c->edges[(L - 1) & 3]);
        unsigned long long edges = 0;
        unsigned found = 0;
        // the next level's counters, and the bitmap that held the frontier of L - 2
        if (tid == 0) {
            c->cnt[(L + 1) & 3] = 0;
            c->edges[(L + 1) & 3] = 0;
        }
        for (int64_t w = tid; w < words; w += threads) a.bm[(L + 1) % 3][w] = 0;
        const unsigned long long level = (unsigned long long)L << 32;
        if (fe * kPushDiv < (unsigned long long)a.nnz) {
            const int32_t* list = a.list[(L - 1) & 1];
            auto offer = [&](int64_t e, int64_t end, unsigned long long val) {
                bool fresh = false;
                int32_t u = 0;
                if (e < end) {
                    u = __ldg(&a.cols[e]);
                    const unsigned long long x = __ldcg(&a.X[u]);
                    if (val < x) fresh = atomicMin(&a.X[u], val) == ~0ULL;
                }
                reach(fresh, u, L, edges, found);
            };
            for (int64_t i = warp; i < n_front; i += warps) {
                const int32_t v = __ldcg(&list[i]);
                if ((uint32_t)v >= (uint64_t)a.n) continue;  // only in a race of overlapping calls
                const int64_t beg = a.rowp[v], end = a.rowp[v + 1];
                if (end - beg > kLongRow) {
                    unsigned at = 0;
                    if (lane == 0) at = atomicAdd(&s_queued, 1u);
                    at = __shfl_sync(kFull, at, 0);
                    if (at < kQueue) {
                        if (lane == 0) s_queue[at] = v;
                        continue;
                    }
                }
                const unsigned long long val = level | (uint32_t)__ldcg(&a.X[v]);
                for (int64_t e = beg; e < end; e += 32) offer(e + lane, end, val);
            }
            __syncthreads();
            const int queued = (int)min(s_queued, (unsigned)kQueue);
            for (int q = 0; q < queued; ++q) {
                const int32_t v = s_queue[q];
                const int64_t end = a.rowp[v + 1];
                const unsigned long long val = level | (uint32_t)__ldcg(&a.X[v]);
                for (int64_t e = a.rowp[v] + (threadIdx.x & ~31); e < end; e += kResThreads) offer(e + lane, end, val);
            }
        } else {
            for (int64_t w = threadIdx.x; w < words; w += kResThreads) s_bm[w] = __ldcg(&a.bm[(L - 1) % 3][w]);
            __syncthreads();
            int64_t e = e0;
            for (int64_t r = row0; e < e1; r += 32) {
                // 32 rows: their ends, and which of them have no distance of an earlier level
                const int64_t v = min(r + lane, a.n - 1);
                const int64_t end_v = a.rowp[v + 1];
                const unsigned long long x = __ldcg(&a.X[v]);
                const unsigned want = __ballot_sync(kFull, r + lane < a.n && x >= level);
                const int64_t w_end = min(__shfl_sync(kFull, end_v, 31), e1);
                if (want == 0) {
                    e = max(e, w_end);
                    continue;
                }
                const int rel_end = (int)(min(end_v, e1) - e0);  // a share holds fewer than 2^31 entries
                for (; e < w_end; e += 128) {
                    int own[4];
                    int32_t u[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int64_t at = e + 32 * j + lane;
                        const int rel = (int)(at - e0);
                        int o = 0;  // rows of the window that end at or before the entry
#pragma unroll
                        for (int s = 16; s > 0; s >>= 1)
                            if (__shfl_sync(kFull, rel_end, o + s - 1) <= rel) o += s;
                        own[j] = o;
                        u[j] = at < w_end && ((want >> o) & 1u) ? __ldg(&a.cols[at]) : -1;
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const bool hit = u[j] >= 0 && ((s_bm[u[j] >> 5] >> (u[j] & 31)) & 1u);
                        if (!__any_sync(kFull, hit)) continue;
                        // the smallest label of each run of entries of one row, on the run's last lane
                        uint32_t lab = hit ? (uint32_t)__ldcg(&a.X[u[j]]) : ~0u;
#pragma unroll
                        for (int s = 1; s < 32; s <<= 1) {
                            const uint32_t y = __shfl_up_sync(kFull, lab, s);
                            const int yo = __shfl_up_sync(kFull, own[j], s);
                            if (lane >= s && yo == own[j]) lab = min(lab, y);
                        }
                        const int next = __shfl_down_sync(kFull, own[j], 1);
                        const bool last = lane == 31 || next != own[j];
                        bool fresh = false;
                        if (last && lab != ~0u) fresh = atomicMin(&a.X[r + own[j]], level | lab) == ~0ULL;
                        reach(fresh, (int32_t)(r + own[j]), L, edges, found);
                    }
                }
                e = w_end;
            }
        }
        if (!end_level(L, edges, found)) return;
    }
    for (int64_t v = tid; v < a.n; v += threads) {
        const unsigned long long x = __ldcg(&a.X[v]);
        if (a.assign) a.assign[v] = x == ~0ULL ? -1 : (int32_t)(x & 0xffffffffULL);
        if (a.dist) a.dist[v] = x == ~0ULL ? -1 : (int32_t)(x >> 32);
    }
    if (tid == 0) c->done = 1;
}

int grid_for(int64_t items, int per_block) {
    int64_t b = (items + per_block - 1) / per_block;
    if (b < 1) b = 1;
    if (b > 152 * 32) b = 152 * 32;
    return (int)b;
}

}  // namespace
}  // namespace fl

using namespace fl;

extern "C" int fl_assign_nearest_noalloc(int64_t n, const int64_t* row_off, const int32_t* cols, int64_t nnz,
                                         const uint8_t* open, int32_t* assign_out, int32_t* dist_out,
                                         void* stream) {
    if (n < 1 || n > kMaxN) {
        char buf[160];
        std::snprintf(buf, sizeof(buf), "n = %lld outside [1, %lld], the size of the fixed scratch", (long long)n,
                      (long long)kMaxN);
        FL_FAIL(FL_EINVAL, buf);
    }
    if (nnz < 0 || !row_off || (nnz > 0 && !cols) || !open || (!assign_out && !dist_out))
        FL_FAIL(FL_EINVAL, "bad arguments");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned char* base = nullptr;
    FL_TRY(scratch_address(&base));
    NoallocArgs a;
    a.rowp = row_off;
    a.cols = cols;
    a.n = n;
    a.nnz = nnz;
    a.open = open;
    a.X = reinterpret_cast<unsigned long long*>(base + kOffX);
    a.list[0] = reinterpret_cast<int32_t*>(base + kOffList);
    a.list[1] = a.list[0] + kMaxN;
    for (int i = 0; i < 3; ++i) a.bm[i] = reinterpret_cast<uint32_t*>(base + kOffBm) + i * (kMaxN / 32);
    a.c = reinterpret_cast<NoallocCtl*>(base + kOffCtl);
    Counters* ctr = reinterpret_cast<Counters*>(base + kOffCtr);
    a.check = ctr;
    a.assign = assign_out;
    a.dist = dist_out;

    // the CSR is checked on the device; the search reads the verdict before
    // anything else and leaves a graph that failed alone
    FL_CUDA(cudaMemsetAsync(a.c, 0, 512, st));
    k_validate_csr<<<grid_for(n + nnz, 256), 256, 0, st>>>(row_off, cols, n, nnz, ctr);
    FL_CUDA(cudaGetLastError());
    int dev = 0, sms = 0;
    FL_CUDA(cudaGetDevice(&dev));
    FL_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(sms, (n + nnz) / (4 * kResThreads)));
    const size_t smem = (size_t)((n + 31) / 32) * 4;
    FL_CUDA(cudaFuncSetAttribute((const void*)k_noalloc_bfs, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(kMaxN / 8)));
    void* args[] = {&a};
    FL_CUDA(cudaLaunchCooperativeKernel((const void*)k_noalloc_bfs, dim3(blocks), dim3(kResThreads), args, smem, st));
    struct {
        NoallocCtl c;
        char pad[256 - sizeof(NoallocCtl)];
        Counters ctr;
    } out;
    FL_CUDA(cudaMemcpyAsync(&out, a.c, sizeof(out), cudaMemcpyDeviceToHost, st));
    FL_CUDA(cudaStreamSynchronize(st));
    if (out.ctr.error) FL_FAIL(FL_EINVAL, "invalid CSR (offsets must be monotone from 0 to nnz, ids in [0, n))");
    if (!out.c.done) FL_FAIL(FL_ETIMEOUT, "BFS: a barrier wait ran out");
    return FL_OK;
}

// k_sort.cu -- stable least-significant-digit radix sort of (key, payload)
// pairs, 8-bit digits, one kernel per digit.
//
// One histogram kernel counts every digit of the sort at once.  A digit's
// kernel then reads each pair once and writes it once: a block takes the next
// tile of kTile pairs, ranks them by digit within its warps (lanes with equal
// digits find each other with match_any), publishes the tile's 256 counts,
// adds up the counts of the tiles before it by looking back through their
// published words (decoupled look-back, Merrill and Garland 2016; the
// one-pass digit of Adinets and Merrill 2022), stages the pairs in shared
// memory in digit order and writes runs of equal digits contiguously.  Tiles
// are handed out by a counter, so every tile that a block waits for is already
// running; the wait is bounded all the same and reports through *err.
//
// What bounds it: for the sizes of the solves (10^5..10^7 pairs of 12 B, in
// L2) the latency of a tile, about 10 us per digit; the 4-bit, three-kernel
// passes over 20-byte triples that this replaces took 25-40 us per 8 bits.
#include "fl_internal.cuh"

namespace fl {

namespace {

constexpr int kThreads = 256;
constexpr int kItems = 12;
constexpr int kTile = kThreads * kItems;
constexpr int kBins = 256;
constexpr unsigned long long kAgg = 1ULL << 62, kPrefix = 2ULL << 62, kCount = (1ULL << 62) - 1;
constexpr unsigned kSpinLimit = 1u << 24;

struct Shifts {
    int s[kSortDigits];
};

template <class K>
__device__ __forceinline__ int digit_of(K key, int shift) {
    return (int)((key >> shift) & (K)(kBins - 1));
}

template <class K>
__global__ void __launch_bounds__(kThreads) k_sort_hist(const K* __restrict__ key, int64_t n, Shifts sh, int nd,
                                                        unsigned long long* __restrict__ hist) {
    __shared__ unsigned h[kSortDigits][kBins];
    for (int i = threadIdx.x; i < nd * kBins; i += kThreads) h[i / kBins][i % kBins] = 0;
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const K k = key[i];
        for (int d = 0; d < nd; ++d) atomicAdd(&h[d][digit_of(k, sh.s[d])], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nd * kBins; i += kThreads) {
        const unsigned c = h[i / kBins][i % kBins];
        if (c) atomicAdd(&hist[i], (unsigned long long)c);
    }
}

// Exclusive scan of one value per thread (kThreads threads); every thread calls.
template <class T>
__device__ __forceinline__ T block_scan(T x, T* warp_tot) {
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    T incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    T before = 0;
    for (int w = 0; w < warp; ++w) before += warp_tot[w];
    __syncthreads();
    return before + incl - x;
}

template <class K>
__global__ void __launch_bounds__(kThreads) k_sort_digit(const K* __restrict__ kin, const uint32_t* __restrict__ vin,
                                                         K* __restrict__ kout, uint32_t* __restrict__ vout, int64_t n,
                                                         int shift, const unsigned long long* __restrict__ hist,
                                                         volatile unsigned long long* status,
                                                         unsigned long long* __restrict__ next_tile,
                                                         unsigned long long* __restrict__ err) {
    __shared__ K skey[kTile];
    __shared__ uint32_t sval[kTile];
    __shared__ unsigned whist[kThreads / 32][kBins];
    __shared__ long long s_off[kBins];
    __shared__ unsigned long long wt[kThreads / 32];
    __shared__ long long s_tile;
    const int lane = lane_id(), warp = threadIdx.x >> 5, t = threadIdx.x;
    if (t == 0) s_tile = (long long)atomicAdd(next_tile, 1ULL);
    for (int w = 0; w < kThreads / 32; ++w) whist[w][t] = 0;
    __syncthreads();
    const int64_t tile = s_tile, base = tile * kTile;
    const int count = n - base < kTile ? (int)(n - base) : kTile;
    // the warp's kItems x 32 consecutive pairs, 32 at a time
    K key[kItems];
    uint32_t val[kItems];
    unsigned rank[kItems];
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
        const int at = (warp * kItems + i) * 32 + lane;
        key[i] = at < count ? kin[base + at] : (K)0;
        val[i] = at < count ? vin[base + at] : 0u;
    }
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
        const int at = (warp * kItems + i) * 32 + lane;
        const int d = at < count ? digit_of(key[i], shift) : kBins;
        const unsigned same = __match_any_sync(kFull, d);
        const int lead = __ffs(same) - 1;
        unsigned old = 0;
        if (lane == lead && d < kBins) {
            old = whist[warp][d];
            whist[warp][d] = old + __popc(same);
        }
        rank[i] = __shfl_sync(kFull, old, lead) + __popc(same & ((1u << lane) - 1u));
        __syncwarp();
    }
    __syncthreads();
    // thread t owns digit t: the warps' counts become offsets within the tile
    unsigned sum = 0;
    for (int w = 0; w < kThreads / 32; ++w) {
        const unsigned c = whist[w][t];
        whist[w][t] = sum;
        sum += c;
    }
    volatile unsigned long long* mine = status + tile * kBins + t;
    *mine = (tile == 0 ? kPrefix : kAgg) | sum;
    const unsigned long long in_tile = block_scan<unsigned long long>(sum, wt);
    const unsigned long long first = block_scan<unsigned long long>(hist[t], wt);
    unsigned long long before = 0;
    for (int64_t p = tile - 1; p >= 0; --p) {
        unsigned long long w = 0;
        unsigned spins = 0;
        while ((w = status[p * kBins + t]) == 0) {
            if (++spins > kSpinLimit) {
                atomicOr(err, kSortError);
                w = kPrefix;
                break;
            }
        }
        before += w & kCount;
        if (w & kPrefix) break;
    }
    if (tile > 0) *mine = kPrefix | (before + sum);
    for (int w = 0; w < kThreads / 32; ++w) whist[w][t] += (unsigned)in_tile;
    s_off[t] = (long long)(first + before) - (long long)in_tile;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
        const int at = (warp * kItems + i) * 32 + lane;
        if (at < count) {
            const unsigned pos = whist[warp][digit_of(key[i], shift)] + rank[i];
            skey[pos] = key[i];
            sval[pos] = val[i];
        }
    }
    __syncthreads();
    for (int j = t; j < count; j += kThreads) {
        const K k = skey[j];
        const long long to = s_off[digit_of(k, shift)] + j;
        if (to >= 0 && to < n) {  // always, unless a wait above ran out
            kout[to] = k;
            vout[to] = sval[j];
        }
    }
}

}  // namespace

template <class K>
int sort_pairs(SortPairs<K>& p, int64_t n, const int* shift, int nd, cudaStream_t st, DBuf& tmp, int cls,
               unsigned long long* err) {
    if (n <= 1 || nd == 0) return FL_OK;
    if (nd > kSortDigits) FL_FAIL(FL_EINVAL, "radix sort: too many digits");
    const int64_t tiles = (n + kTile - 1) / kTile;
    // histograms, tile counters, status words of every digit
    const size_t hist_b = (size_t)nd * kBins * 8, next_b = 256, status_b = (size_t)tiles * kBins * 8;
    FL_TRY(dalloc(tmp, hist_b + next_b + status_b * nd));
    unsigned long long* hist = tmp.as<unsigned long long>();
    unsigned long long* next = hist + (size_t)nd * kBins;
    unsigned long long* status = next + next_b / 8;
    FL_CUDA(cudaMemsetAsync(tmp.p, 0, hist_b + next_b + status_b * nd, st));
    Shifts sh;
    for (int d = 0; d < kSortDigits; ++d) sh.s[d] = d < nd ? shift[d] : 0;
    int64_t hb = (n + 4 * kThreads - 1) / (4 * kThreads);
    if (hb > 152 * 4) hb = 152 * 4;
    FL_LAUNCH(cls, k_sort_hist<K><<<(unsigned)hb, kThreads, 0, st>>>(p.key[p.cur], n, sh, nd, hist));
    for (int d = 0; d < nd; ++d) {
        FL_LAUNCH(cls, k_sort_digit<K><<<(unsigned)tiles, kThreads, 0, st>>>(
                           p.key[p.cur], p.val[p.cur], p.key[p.cur ^ 1], p.val[p.cur ^ 1], n, sh.s[d],
                           hist + (size_t)d * kBins, status + (size_t)d * tiles * kBins, next + d, err));
        p.cur ^= 1;
    }
    FL_CUDA(cudaGetLastError());
    return FL_OK;
}

template int sort_pairs<uint32_t>(SortPairs<uint32_t>&, int64_t, const int*, int, cudaStream_t, DBuf&, int,
                                  unsigned long long*);
template int sort_pairs<uint64_t>(SortPairs<uint64_t>&, int64_t, const int*, int, cudaStream_t, DBuf&, int,
                                  unsigned long long*);

int digit_windows(uint64_t varying, int bits, int* shift) {
    if (!varying) return 0;
    int top = 63, low = 0;
    while (!((varying >> top) & 1)) --top;
    while (!((varying >> low) & 1)) ++low;
    if (bits > 0 && top + 1 - bits > low) low = top + 1 - bits;
    const int nd = (top + 1 - low + 7) / 8;
    const int first = top + 1 - 8 * nd > 0 ? top + 1 - 8 * nd : 0;
    for (int d = 0; d < nd; ++d) shift[d] = first + 8 * d;
    return nd;
}

}  // namespace fl

// order.cu -- longest-first order of a batch from per-system cost estimates.
//
// A counting sort on a 16-bit cost class.  Positive floats order like their
// bit patterns, and the bit pattern is close to a scaled log2 of the value,
// so the classes split the range [lo, hi] of the batch's positive costs'
// bit patterns into 65535 equal steps (about log-uniform): class
// 1 + (bits - lo) * 65535 / (hi - lo + 1); NaN and values <= 0 form class 0.
// Classes that narrow matter: systems of almost equal cost follow almost the
// same step sequence, so a warp of them stays in phase (merging neighbouring
// costs of a few parts in a thousand measurably costs time), and a few
// outliers must not widen the classes much.  One memset and four launches:
//   k_order_range    lo and hi, and how much of their range an average group
//                    of 32 consecutive systems covers (block reductions);
//   k_order_hist     class histogram (global atomics, aggregated over the
//                    lanes of a warp that share a class);
//   k_order_scan     descending exclusive scan, so the most expensive class
//                    starts at position 0: a block per 1,024 classes, which
//                    sums the classes above its own by itself (the histogram
//                    is 256 KB in L2) and needs no other block;
//   k_order_scatter  each system's position from its class's running
//                    offset (lanes of a warp with the same class take
//                    consecutive positions with one atomic).
// Launches and their latencies are what an order costs: with the scan in one
// block, whose threads read 64 scattered classes each, twice, and with three
// memsets 90 us at 20,000 systems and 125 at 1M; so 20 and 65.
// Systems of one class land in an unspecified order; the integration
// results do not depend on it.
//
// Some batches keep their own order (index[i] = i): one whose costs are all
// equal -- a caller's way to ask for its own layout -- and, for an order that
// nobody asked for, one whose consecutive systems are already alike in the
// key.  Thirty-two systems drawn at random cover 0.93 of the range on
// average; systems laid out by their cost, or along a smooth field, much
// less (van der Pol systems by their evaluations 0.12-0.26, networks
// 0.50-0.57, grids 0.55).  Up to kGrouped of the range the layout stays.
#include <cuda_runtime.h>

#include <cstdint>

#include "order.h"

namespace bode {

namespace {

constexpr int kScanThreads = 1024;
static_assert(kOrderBins % kScanThreads == 0 && kScanThreads == 32 * 32, "whole scan blocks, a warp of warp totals");

// a cost as float: float32 estimates, int32 counts (e.g. n_rhs), or an
// FP64 parameter
__device__ __forceinline__ float cost_at(const void* cost, int kind, int64_t i) {
    switch (kind) {
    case kCostInt: return (float)static_cast<const int32_t*>(cost)[i];
    case kCostParam: return (float)static_cast<const double*>(cost)[i];
    default: return static_cast<const float*>(cost)[i];
    }
}

// the batch's keys, from zeroed memory (k_order_range)
struct OrderStat {
    uint32_t not_lo;  // the complement of the smallest positive key's bits (0: no positive key)
    uint32_t hi;      // the largest one's
    unsigned long long spread;  // summed over groups of 32 consecutive systems: largest less smallest key
    uint32_t rest;    // whether a key was NaN or not positive
};
constexpr double kGrouped = 0.75;

// whether the batch keeps its own order
__device__ __forceinline__ bool keeps_order(const OrderStat* st, int kind, int64_t n) {
    if (st->not_lo == 0u) return true;  // one class
    const uint32_t range = st->hi - ~st->not_lo;
    if (range == 0u && !st->rest) return true;
    return kind == kCostParam && (double)st->spread <= kGrouped * (double)range * (double)((n + 31) / 32);
}

__device__ __forceinline__ int cost_class(float c, const OrderStat* st) {
    if (!(c > 0.0f)) return 0;  // NaN, zero and negative estimates: cheapest
    const uint32_t lo = ~st->not_lo, hi = st->hi;
    const uint64_t step = (uint64_t)(__float_as_uint(c) - lo) * (uint64_t)(kOrderBins - 1);
    return 1 + (int)(step / ((uint64_t)(hi - lo) + 1u));
}

__global__ void __launch_bounds__(256) k_order_range(const void* __restrict__ cost, int kind, int64_t n,
                                                     OrderStat* __restrict__ st) {
    uint32_t not_lo = 0u, hi = 0u, rest = 0u;
    unsigned long long spread = 0ull;
    // a warp takes 32 consecutive systems at a time (strides are whole blocks)
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i - (threadIdx.x & 31) < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float c = i < n ? cost_at(cost, kind, i) : 0.0f;
        const bool pos = c > 0.0f;
        const uint32_t bits = pos ? __float_as_uint(c) : 0u;
        hi = max(hi, bits);
        if (pos) not_lo = max(not_lo, ~bits);
        rest |= (uint32_t)(i < n && !pos);
        const uint32_t top = __reduce_max_sync(0xffffffffu, bits);
        const uint32_t low = __reduce_min_sync(0xffffffffu, i < n ? bits : top);
        spread += top - low;  // the same in every lane
    }
    not_lo = __reduce_max_sync(0xffffffffu, not_lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    rest = __reduce_max_sync(0xffffffffu, rest);
    __shared__ uint32_t s_not_lo[8], s_hi[8], s_rest[8];
    __shared__ unsigned long long s_spread[8];
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        s_not_lo[w] = not_lo;
        s_hi[w] = hi;
        s_rest[w] = rest;
        s_spread[w] = spread;
    }
    __syncthreads();
    if (threadIdx.x) return;
    for (int q = 1; q < (int)blockDim.x / 32; ++q) {
        not_lo = max(not_lo, s_not_lo[q]);
        hi = max(hi, s_hi[q]);
        rest |= s_rest[q];
        spread += s_spread[q];
    }
    if (not_lo) atomicMax(&st->not_lo, not_lo);
    if (hi) atomicMax(&st->hi, hi);
    if (rest) atomicOr(&st->rest, 1u);
    if (spread) atomicAdd(&st->spread, spread);
}

__global__ void k_order_hist(const void* __restrict__ cost, int kind, int64_t n, const OrderStat* __restrict__ st,
                             int32_t* __restrict__ hist) {
    if (keeps_order(st, kind, n)) return;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = i < n;
    const unsigned active = __ballot_sync(0xffffffffu, live);
    if (!live) return;
    const int cls = cost_class(cost_at(cost, kind, i), st);
    const unsigned peers = __match_any_sync(active, cls);
    if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&hist[cls], __popc(peers));
}

// offset[b] = number of systems in classes above b; block q takes classes
// kOrderBins - 1 - 1024 q downward, one a thread
__global__ void __launch_bounds__(kScanThreads) k_order_scan(const int32_t* __restrict__ hist, int kind, int64_t n,
                                                             const OrderStat* __restrict__ st,
                                                             int32_t* __restrict__ offset) {
    if (keeps_order(st, kind, n)) return;
    __shared__ int32_t warp_sums[kScanThreads / 32], warp_above[kScanThreads / 32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int cls = kOrderBins - 1 - kScanThreads * (int)blockIdx.x - t;
    const int32_t mine = hist[cls];
    int32_t above = 0;  // classes of the blocks above this one
    const int4* h4 = reinterpret_cast<const int4*>(hist);
#pragma unroll 8
    for (int q = (kOrderBins - kScanThreads * (int)blockIdx.x) / 4 + t; q < kOrderBins / 4; q += kScanThreads) {
        const int4 v = h4[q];
        above += v.x + v.y + v.z + v.w;
    }
    above = (int32_t)__reduce_add_sync(0xffffffffu, (unsigned)above);
    int32_t x = mine;  // inclusive scan over the threads: shuffles, then the warp totals
    for (int d = 1; d < 32; d <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) {
        warp_sums[warp] = x;
        warp_above[warp] = above;
    }
    __syncthreads();
    int32_t before = (int32_t)__reduce_add_sync(0xffffffffu, (unsigned)warp_above[lane]);
    before += (int32_t)__reduce_add_sync(0xffffffffu, lane < warp ? (unsigned)warp_sums[lane] : 0u);
    offset[cls] = before + x - mine;
}

__global__ void k_order_scatter(const void* __restrict__ cost, int kind, int64_t n,
                                 const OrderStat* __restrict__ st, int32_t* __restrict__ offset,
                                 int32_t* __restrict__ index) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = i < n;
    if (keeps_order(st, kind, n)) {
        if (live) index[i] = (int32_t)i;
        return;
    }
    const int cls = live ? cost_class(cost_at(cost, kind, i), st) : -1;
    const unsigned active = __ballot_sync(0xffffffffu, live);
    if (!live) return;
    const unsigned peers = __match_any_sync(active, cls);
    const int leader = __ffs(peers) - 1;
    const int lane = threadIdx.x & 31;
    int32_t base = 0;
    if (lane == leader) base = atomicAdd(&offset[cls], __popc(peers));
    base = __shfl_sync(peers, base, leader);
    index[base + __popc(peers & ((1u << lane) - 1u))] = (int32_t)i;
}

}  // namespace

cudaError_t order_by_cost(const void* cost, int kind, int64_t n, int32_t* bins, int32_t* index, int sm_count,
                          cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    // histogram, keys' range (zeroed together), offsets
    int32_t* hist = bins;
    OrderStat* st = reinterpret_cast<OrderStat*>(bins + kOrderBins);
    int32_t* offset = bins + kOrderBins + kOrderStatWords;
    static_assert(sizeof(OrderStat) <= sizeof(int32_t) * kOrderStatWords, "scratch words");
    cudaError_t e = cudaMemsetAsync(hist, 0, sizeof(int32_t) * (kOrderBins + kOrderStatWords), s);
    if (e != cudaSuccess) return e;
    const int64_t blocks = (n + 255) / 256;
    const unsigned grid = (unsigned)(blocks < 4 * (int64_t)sm_count ? blocks : 4 * (int64_t)sm_count);
    k_order_range<<<grid, 256, 0, s>>>(cost, kind, n, st);
    k_order_hist<<<(unsigned)blocks, 256, 0, s>>>(cost, kind, n, st, hist);
    k_order_scan<<<kOrderBins / kScanThreads, kScanThreads, 0, s>>>(hist, kind, n, st, offset);
    k_order_scatter<<<(unsigned)blocks, 256, 0, s>>>(cost, kind, n, st, offset, index);
    return cudaGetLastError();
}

}  // namespace bode

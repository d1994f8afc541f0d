// scan_device.cuh -- device building blocks of the scans: warp and block prefix sums, and the
// look-back of the single-pass scans.
#pragma once

#include "rgs_internal.cuh"

namespace rgs {
namespace {

__device__ __forceinline__ uint32_t read_count(const uint32_t* n_dev, int64_t n_cap) {
  if (!n_dev) return (uint32_t)n_cap;
  const uint32_t n = *n_dev;
  return n < (uint64_t)n_cap ? n : (uint32_t)n_cap;
}

// Block-wide exclusive scan of one value per thread; returns the block total in *total.
template <int THREADS>
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* total) {
  __shared__ uint32_t warp_sums[THREADS / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < THREADS / 32 ? warp_sums[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < THREADS / 32) warp_sums[lane] = w;  // inclusive warp prefix
  }
  __syncthreads();
  const uint32_t warp_prefix = warp > 0 ? warp_sums[warp - 1] : 0u;
  if (total) *total = warp_sums[THREADS / 32 - 1];
  const uint32_t r = warp_prefix + x - v;
  __syncthreads();  // warp_sums may be reused by the caller's next scan
  return r;
}

// Exclusive prefix of one value per lane; the warp's total in *total.
__device__ __forceinline__ uint32_t warp_exclusive_scan(uint32_t v, uint32_t* total) {
  const int lane = threadIdx.x & 31;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  *total = __shfl_sync(0xffffffffu, x, 31);
  return x - v;
}

// First lane whose inclusive count exceeds idx (31 past the warp total).
__device__ __forceinline__ int lane_of(uint32_t incl, uint32_t idx) {
  int lo = 0, hi = 31;
#pragma unroll
  for (int step = 0; step < 5; ++step) {
    const int mid = (lo + hi) >> 1;
    if (__shfl_sync(0xffffffffu, incl, mid) > idx) hi = mid; else lo = mid + 1;
  }
  return min(lo, 31);
}

// ------------------------------------------------------------------------------------------
// Single-pass scan: the chained scan with decoupled look-back of Merrill and Garland
// ("Single-pass Parallel Prefix Scan with Decoupled Look-back", 2016), in one launch of one
// block per tile of kScanTile elements. A block takes its tile from a ticket counter, so tiles
// are handed out in the order blocks start: a block only ever waits for tiles of blocks that
// are already running, which therefore finish. It scans its tile, publishes the tile total (an
// "aggregate") and, unless it is tile 0, walks back over the earlier tiles 32 at a time (one per
// lane of warp 0), adding aggregates until it meets a published inclusive prefix; then it
// publishes its own inclusive prefix and stores its results. A state word packs the flag in bits 62..63 (0 not yet published, 1 aggregate,
// 2 inclusive prefix) and the value in bits 0..31. It is written and read whole (an aligned
// 64-bit access), and nothing else is published through it, so relaxed accesses suffice. Each
// wait is bounded: past kLookbackSpins polls the block records kStatusScanWait and takes the
// tile as 0 (a wrong result, reported; never expected, since the waited-for block is running).
// ------------------------------------------------------------------------------------------
constexpr unsigned long long kTileAggregate = 1ull << 62, kTileInclusive = 2ull << 62;
constexpr int kLookbackSpins = 1 << 20;  // polls of ~1 us each

__device__ __forceinline__ void store_state(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long load_state(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// Takes a tile from the ticket counter (thread 0; the result is broadcast to the block).
__device__ __forceinline__ uint32_t lookback_ticket(const Lookback& lb) {
  __shared__ uint32_t s_tile;
  if (threadIdx.x == 0) s_tile = atomicAdd(lb.ticket, 1u);
  __syncthreads();
  return s_tile;
}

// Called by the 32 lanes of warp 0 of the block holding tile b, whose elements sum to agg:
// publishes the aggregate, looks back for the exclusive prefix of the tile, publishes the
// inclusive prefix and returns the exclusive one (in every lane).
__device__ uint32_t lookback_prefix(const Lookback& lb, uint32_t b, uint32_t agg) {
  const int lane = threadIdx.x & 31;
  if (b == 0) {
    if (lane == 0) store_state(&lb.tiles[0], kTileInclusive | agg);
    return 0u;
  }
  if (lane == 0) store_state(&lb.tiles[b], kTileAggregate | agg);
  uint32_t prefix = 0;
  bool timed_out = false;
  for (int64_t end = b; end > 0; end -= 32) {
    const int64_t j = end - 1 - lane;  // lane 0 looks at the nearest earlier tile
    unsigned long long w = kTileInclusive;  // before tile 0: an empty inclusive prefix
    if (j >= 0) {
      w = load_state(&lb.tiles[j]);
      for (int spin = 0; (w >> 62) == 0; ++spin) {
        if (spin >= kLookbackSpins) {
          timed_out = true;
          w = kTileInclusive;
          break;
        }
        __nanosleep(32);
        w = load_state(&lb.tiles[j]);
      }
    }
    const uint32_t inclusive = __ballot_sync(0xffffffffu, (w >> 62) == 2ull);
    // Tiles nearer than the nearest inclusive prefix contribute their aggregates, that prefix
    // contributes itself, and the farther tiles nothing.
    const int stop = inclusive ? __ffs(inclusive) - 1 : 32;
    uint32_t x = lane <= stop ? (uint32_t)w : 0u;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    prefix += x;
    if (inclusive) break;
  }
  if (__any_sync(0xffffffffu, timed_out) && lane == 0)
    atomicOr(lb.status, (uint32_t)kStatusScanWait);
  if (lane == 0) store_state(&lb.tiles[b], kTileInclusive | (prefix + agg));
  return prefix;
}

}  // namespace
}  // namespace rgs

// cells.cu -- from the depth-sorted visible entries to the tiles' front-to-back lists (Section
// 3.1: the ordered covering set of every pixel).
//
// A footprint touches many tiles (60 on average in a 16-view 1080p window of 3M Gaussians), so a
// sort of (tile, Gaussian) pairs moves the same Gaussian again and again. The pairs are therefore
// built in two levels:
//   emit     one entry per touched cell of 4 x 4 tiles, with the mask of its touched tiles, in
//            depth order (7 per footprint there);
//   sort     the entries by cell (stable, sort.cu), which leaves each cell's run in depth order;
//   ranges   [first, last + 1) of each cell's run;
//   count    pairs per tile, from the masks of its cell's run; a scan in tile order gives every
//            tile's place in the pair list;
//   expand   each cell's run is written out to its 16 tiles' lists: a warp takes a tile, a ballot
//            of 32 masks' bits ranks the entries that touch it, and their indices are stored side
//            by side. A run's order carries over, so every tile's list is in (depth, index) order.
// The radix passes then move 1/8 of the pairs, nothing reads or writes a key per pair, and each
// pair costs one 4-byte store.
#include <algorithm>

#include "scan_device.cuh"

namespace rgs {
namespace {

// ------------------------------------------------------------------------------------------
// Emission. A block takes a tile of consecutive entries of the depth order (by ticket); its warps
// take 32 at a time. The prefix of the cell counts (warp, block, then look-back over the earlier
// blocks) gives every round its slots, so the list keeps the depth order and no separate scan is
// launched. Each lane sets up its own footprint's cover once; the covers' cell rows are then dealt
// out over the lanes (a lane per footprint would wait for the tallest one of the warp: 3 rows on
// average, 30 at most), whose cells are written in (footprint, row, column) order into shared
// memory, and from there side by side. A round that exceeds the buffer is written directly.
// Long lists take kEmitItems rounds per warp, so that the look-back chain stays short; short ones
// one round, so that every SM has work (59k entries: 231 blocks instead of 58).
// ------------------------------------------------------------------------------------------
constexpr int kEmitThreads = 256;
constexpr int kEmitWarps = kEmitThreads / 32;
constexpr int kEmitItems = 4;
constexpr int64_t kEmitLong = 4 * 152 * kEmitThreads;
constexpr uint32_t kEmitStage = 512;  // cell entries a warp stages per round

int emit_items(int64_t visible) { return visible > kEmitLong ? kEmitItems : 1; }

template <bool kMasks>
__device__ __forceinline__ uint32_t cell_key(uint32_t cell, uint32_t mask) {
  return kMasks ? (cell << 16) | mask : cell;
}

template <bool kMasks, int ITEMS>
__global__ void __launch_bounds__(kEmitThreads) emit_cells_kernel(
    const __grid_constant__ Views views, int n, const uint32_t* __restrict__ order,
    const Record* __restrict__ rec, float log2_alpha_min, uint32_t visible_cap,
    uint32_t capacity, uint32_t* __restrict__ keys, uint32_t* __restrict__ vals, Lookback lb,
    uint32_t n_blocks, Counters* __restrict__ counters) {
  chain_wait();
  __shared__ uint32_t s_key[kEmitWarps][kEmitStage], s_val[kEmitWarps][kEmitStage];
  __shared__ uint32_t s_warp[kEmitWarps];
  const uint32_t b = lookback_ticket(lb);
  if (b >= n_blocks) {  // the ticket counter was not zeroed: report, touch nothing
    if (threadIdx.x == 0) atomicOr(lb.status, (uint32_t)kStatusScanWait);
    return;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // The sorted list holds at most visible_cap entries; more (only possible under stream capture)
  // are dropped from this forward and recorded in the status word.
  const uint32_t n_visible_raw = counters->n_visible;
  const uint32_t n_visible = min(n_visible_raw, visible_cap);
  if (b == 0 && threadIdx.x == 0) {
    if (n_visible_raw > visible_cap) atomicOr(&counters->status, (uint32_t)kStatusVisibleOverflow);
    counters->n_visible_kept = n_visible;
  }
  const uint32_t first = b * (kEmitThreads * ITEMS) + (uint32_t)warp * (32 * ITEMS) + lane;
  uint32_t vi[ITEMS], total[ITEMS], sum = 0;
  unsigned long long tiles = 0;
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) vi[j] = first + 32u * j < n_visible ? order[first + 32u * j] : 0u;
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const uint2 t = first + 32u * j < n_visible ? rec[vi[j]].touched : make_uint2(0u, 0u);
    tiles += t.x;
    total[j] = __reduce_add_sync(0xffffffffu, t.y);
    sum += total[j];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tiles += __shfl_xor_sync(0xffffffffu, tiles, o);
  if (lane == 0) {
    s_warp[warp] = sum;
    if (tiles) atomicAdd(&counters->n_pairs, tiles);
  }
  __syncthreads();
  if (warp == 0) {
    uint32_t agg;
    const uint32_t before = warp_exclusive_scan(lane < kEmitWarps ? s_warp[lane] : 0u, &agg);
    const uint32_t prefix = lookback_prefix(lb, b, agg);
    if (lane < kEmitWarps) s_warp[lane] = prefix + before;
    if (b == n_blocks - 1 && lane == 0) {
      const uint32_t all = prefix + agg;
      counters->n_cells = all;
      counters->n_cells_stored = min(all, capacity);
      if (all > capacity) atomicOr(&counters->status, (uint32_t)kStatusPairOverflow);
    }
  }
  __syncthreads();
  uint32_t out0 = s_warp[warp];  // first slot of the round
#pragma unroll 1
  for (int j = 0; j < ITEMS; ++j) {
    const uint32_t round = total[j];
    if (round == 0) continue;  // warp-uniform
    const uint32_t my_vi = vi[j];
    const bool staged = round <= kEmitStage;  // warp-uniform
    auto put = [&](uint32_t slot, uint32_t key, uint32_t val) {
      if (staged) {
        s_key[warp][slot] = key;
        s_val[warp][slot] = val;
      } else if (out0 + slot < capacity) {
        keys[out0 + slot] = key;
        vals[out0 + slot] = val;
      }
    };
    TileCover tc{};
    uint32_t rows = 0;
    int cell_base = 0, cells_x = 0;
    if (first + 32u * j < n_visible) {
      Ellipse e;
      const ViewParams& vp = views.v[my_vi / (uint32_t)max(n, 1)];
      cell_base = vp.cell_base;
      cells_x = vp.cells_x;
      if (make_ellipse(rec[my_vi].mean, rec[my_vi].conic, log2_alpha_min, e) &&
          tc.init(e, views.tile_w, views.tile_h, vp.tiles_x, vp.tiles_y))
        rows = (uint32_t)((tc.ty1 >> kCellShift) - (tc.ty0 >> kCellShift) + 1);
    }
    uint32_t row_total, done = 0;  // rows of the round; slots filled
    const uint32_t row_first = warp_exclusive_scan(rows, &row_total);
    for (uint32_t r0 = 0; r0 < row_total; r0 += 32) {
      const uint32_t task = r0 + lane;
      const int from = lane_of(row_first + rows, task);
      const TileCover tb = tc.from_lane(from, views.tile_w, views.tile_h);
      const uint32_t vib = __shfl_sync(0xffffffffu, my_vi, from);
      const int cy = (tb.ty0 >> kCellShift) +
                     (int)(task - __shfl_sync(0xffffffffu, row_first, from));
      const int base = __shfl_sync(0xffffffffu, cell_base, from) +
                       cy * __shfl_sync(0xffffffffu, cells_x, from);
      CellRow row;
      uint32_t w = 0;
      if (task < row_total && cell_row(tb, cy, row)) w = (uint32_t)(row.c1 - row.c0 + 1);
      uint32_t filled;
      uint32_t slot = done + warp_exclusive_scan(w, &filled);
      for (uint32_t k = 0; k < w && slot < round; ++k, ++slot) {
        const int c = row.c0 + (int)k;
        put(slot, cell_key<kMasks>((uint32_t)(base + c), kMasks ? cell_mask(row.span, c) : 0u),
            vib);
      }
      done += filled;
    }
    // The projection counted the same cells with the same operations, so every slot is filled; if
    // that ever failed, the rest get an id past the last cell, which no run holds.
    for (uint32_t slot = done + lane; slot < round; slot += 32)
      put(slot, cell_key<kMasks>((uint32_t)views.total_cells, 0u), 0u);
    __syncwarp();
    if (staged) {
      for (uint32_t t = lane; t < round; t += 32)
        if (out0 + t < capacity) {
          keys[out0 + t] = s_key[warp][t];
          vals[out0 + t] = s_val[warp][t];
        }
    }
    __syncwarp();
    out0 += round;
  }
}

// No visible-list capacity: nothing to emit, but a visible entry that is dropped is recorded.
__global__ void no_cells_kernel(Counters* counters) {
  chain_wait();
  if (counters->n_visible > 0) atomicOr(&counters->status, (uint32_t)kStatusVisibleOverflow);
}

// ------------------------------------------------------------------------------------------
// Cell ranges: thread t looks at the eight sorted keys 8t .. 8t + 7 (two 16-byte loads; the key
// arrays are 256-byte aligned) and the key before them, and writes the run boundaries among them
// into `ranges` (zero on entry: cells without entries keep [0, 0)).
// ------------------------------------------------------------------------------------------
constexpr int kRangesThreads = 256;
constexpr int kRangesKeys = 8;

__global__ void __launch_bounds__(kRangesThreads) cell_ranges_kernel(
    const uint32_t* __restrict__ keys, int shift, uint32_t total_cells,
    uint2* __restrict__ ranges, const Counters* __restrict__ counters) {
  chain_wait();
  const uint32_t np = counters->n_cells_stored;
  const uint32_t p0 = (uint32_t)kRangesKeys * (blockIdx.x * kRangesThreads + threadIdx.x);
  if (p0 >= np) return;
  uint32_t k[kRangesKeys + 2];  // k[0] = key before p0 (or none), k[1..8] = keys p0 .., the next
  k[0] = p0 > 0 ? keys[p0 - 1] : 0xffffffffu;
  if (p0 + kRangesKeys <= np) {
#pragma unroll
    for (int h = 0; h < kRangesKeys / 4; ++h) {
      const uint4 q = *reinterpret_cast<const uint4*>(keys + p0 + 4 * h);
      k[4 * h + 1] = q.x;
      k[4 * h + 2] = q.y;
      k[4 * h + 3] = q.z;
      k[4 * h + 4] = q.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < kRangesKeys; ++j) k[j + 1] = p0 + j < np ? keys[p0 + j] : 0xffffffffu;
  }
  k[kRangesKeys + 1] = p0 + kRangesKeys < np ? keys[p0 + kRangesKeys] : 0xffffffffu;
#pragma unroll
  for (int j = 0; j < kRangesKeys + 2; ++j) k[j] >>= shift;
#pragma unroll
  for (int j = 1; j <= kRangesKeys; ++j) {
    const uint32_t p = p0 + j - 1;
    if (p >= np || k[j] >= total_cells) continue;
    if (p == 0 || k[j - 1] != k[j]) ranges[k[j]].x = p;
    if (p == np - 1 || k[j + 1] != k[j]) ranges[k[j]].y = p + 1;
  }
}

// ------------------------------------------------------------------------------------------
// Count and expand: one block per cell walks the cell's run in chunks of kCellThreads entries,
// whose masks it stages in shared memory; warp w answers for tiles w and w + 8 of the cell.
// ------------------------------------------------------------------------------------------
constexpr int kCellThreads = 256;
constexpr int kCellWarps = kCellThreads / 32;
constexpr int kCellArea = kCellTiles * kCellTiles;
static_assert(kCellArea == 2 * kCellWarps, "two tiles per warp");

// The cell's place: its view, and tile (row, column) of its first tile.
struct CellPlace {
  const ViewParams* vp;
  int v, cy, cx;
};
__device__ __forceinline__ CellPlace place_of(const Views& views, int cell) {
  CellPlace p;
  p.v = view_of_cell(views, cell);
  p.vp = &views.v[p.v];
  const int local = cell - p.vp->cell_base;
  p.cy = local / p.vp->cells_x;
  p.cx = local - p.cy * p.vp->cells_x;
  return p;
}
// Global id of tile t (4 row + column) of the cell, -1 past the edge of the view.
__device__ __forceinline__ int tile_of(const CellPlace& p, int t) {
  const int ty = p.cy * kCellTiles + t / kCellTiles, tx = p.cx * kCellTiles + t % kCellTiles;
  return ty < p.vp->tiles_y && tx < p.vp->tiles_x ? p.vp->tile_base + ty * p.vp->tiles_x + tx : -1;
}

// Tile mask of list entry (key, vi) in the cell.
template <bool kMasks>
__device__ __forceinline__ uint32_t entry_mask(const Views& views, const CellPlace& p,
                                               uint32_t key, uint32_t vi, const Record* rec,
                                               float log2_alpha_min) {
  if constexpr (kMasks) {
    return key & 0xffffu;
  } else {
    Ellipse e;
    TileCover tc;
    CellRow row;
    if (!make_ellipse(rec[vi].mean, rec[vi].conic, log2_alpha_min, e) ||
        !tc.init(e, views.tile_w, views.tile_h, p.vp->tiles_x, p.vp->tiles_y) ||
        !cell_row(tc, p.cy, row))
      return 0u;
    return cell_mask(row.span, p.cx);
  }
}

// Launch order of the blends' tiles: longest run first. A CTA's time grows with its tile's run,
// and runs differ by two orders of magnitude (a few tiles near dense structure hold thousands of
// Gaussians); launched in tile order, a long run that starts late holds its SM after the others
// have drained. Ordered by decreasing octave of the length, the long runs start first and the
// short ones fill the end; inside an octave the tiles come cell by cell, roughly in the order the
// blocks run, so neighbouring tiles, which share Gaussians (their records, and in the backward
// their gradient atomics), still run together. Finer classes (16 per octave) made the backward
// 3 % slower; octaves made it 1 % faster than plain tile order. The count kernel adds up how many
// tiles each class holds, the expand kernel takes places in them.
constexpr int kOrderClasses = 33;
__device__ __forceinline__ int length_class(uint32_t len) {
  return 32 - (31 - __clz(len + 1u));  // 0 (longest) .. 32 (empty); len < 2^32 - 1
}

template <bool kMasks>
__global__ void __launch_bounds__(kCellThreads) cell_count_kernel(
    const __grid_constant__ Views views, const uint2* __restrict__ cell_ranges,
    const uint32_t* __restrict__ keys, const uint32_t* __restrict__ vals,
    const Record* __restrict__ rec, float log2_alpha_min,
    uint32_t* __restrict__ tile_counts, uint32_t* __restrict__ class_sizes) {
  chain_wait();
  __shared__ uint32_t s_mask[2][kCellThreads];  // the chunk in use and the next
  __shared__ uint32_t s_count[kCellArea];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const CellPlace place = place_of(views, blockIdx.x);
  const uint2 range = cell_ranges[blockIdx.x];
  uint32_t n0 = 0, n1 = 0;
  auto load = [&](uint32_t p) {
    return p < range.y ? entry_mask<kMasks>(views, place, keys[p], kMasks ? 0u : vals[p], rec,
                                            log2_alpha_min)
                       : 0u;
  };
  uint32_t m = load(range.x + threadIdx.x);
  int buf = 0;
  for (uint32_t start = range.x; start < range.y; start += kCellThreads, buf ^= 1) {
    s_mask[buf][threadIdx.x] = m;
    m = load(start + kCellThreads + threadIdx.x);  // in flight while this chunk is counted
    __syncthreads();
    const uint32_t cnt = min((uint32_t)kCellThreads, range.y - start);
#pragma unroll 4
    for (uint32_t g = 0; g < cnt; g += 32) {
      const uint32_t mm = s_mask[buf][g + lane];
      n0 += __popc(__ballot_sync(0xffffffffu, (mm >> warp) & 1u));
      n1 += __popc(__ballot_sync(0xffffffffu, (mm >> (warp + kCellWarps)) & 1u));
    }
  }
  if (lane == 0) {
    s_count[warp] = n0;
    s_count[warp + kCellWarps] = n1;
  }
  __syncthreads();
  if (threadIdx.x < kCellArea) {
    const int tile = tile_of(place, threadIdx.x);
    const uint32_t count = s_count[threadIdx.x];
    const int cls = tile >= 0 ? length_class(count) : -1;
    const unsigned peers = __match_any_sync(0xffffu, cls);
    if (tile >= 0) {
      tile_counts[tile] = count;
      if (lane == __ffs(peers) - 1) atomicAdd(class_sizes + cls, (uint32_t)__popc(peers));
    }
  }
}

template <bool kMasks>
__global__ void __launch_bounds__(kCellThreads) cell_expand_kernel(
    const __grid_constant__ Views views, const uint2* __restrict__ cell_ranges,
    const uint32_t* __restrict__ keys, const uint32_t* __restrict__ vals,
    const Record* __restrict__ rec, float log2_alpha_min,
    const uint32_t* __restrict__ tile_counts, const uint2* __restrict__ ranges,
    uint32_t* __restrict__ pairs, uint32_t capacity, const uint32_t* __restrict__ class_sizes,
    uint32_t* __restrict__ class_taken, uint32_t* __restrict__ tile_order,
    Counters* __restrict__ counters) {
  chain_wait();
  __shared__ uint32_t s_mask[2][kCellThreads], s_val[2][kCellThreads];
  __shared__ uint2 s_run[kCellArea];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const CellPlace place = place_of(views, blockIdx.x);
  const uint2 range = cell_ranges[blockIdx.x];
  if (blockIdx.x == 0 && threadIdx.x == 0 && counters->n_pairs > capacity) {
    atomicOr(&counters->status, (uint32_t)kStatusPairOverflow);
    if (counters->n_pairs > 0xffffffffull) counters->n_pairs_listed = 0;  // the scan wrapped
  }
  if (warp == 0) {
    // The cell's tiles, their runs, and their places in the launch order.
    const int tile = lane < kCellArea ? tile_of(place, lane) : -1;
    if (lane < kCellArea) s_run[lane] = tile >= 0 ? ranges[tile] : make_uint2(0u, 0u);
    uint32_t sum;
    const uint32_t base = warp_exclusive_scan(class_sizes[lane], &sum);  // classes 0 .. 31
    const int cls = tile >= 0 ? length_class(tile_counts[tile]) : -1;
    const unsigned peers = __match_any_sync(0xffffffffu, cls);
    const int leader = __ffs(peers) - 1;
    uint32_t at = 0;
    if (tile >= 0 && lane == leader) at = atomicAdd(class_taken + cls, (uint32_t)__popc(peers));
    at = __shfl_sync(0xffffffffu, at, leader) + __popc(peers & ((1u << lane) - 1u));
    const uint32_t class_base = __shfl_sync(0xffffffffu, base, cls & 31);
    if (tile >= 0) tile_order[(cls < 32 ? class_base : sum) + at] = (uint32_t)tile;
  }
  __syncthreads();
  uint2 run0 = s_run[warp], run1 = s_run[warp + kCellWarps];
  const unsigned lt = (1u << lane) - 1u;
  uint32_t m = 0, val = 0;
  auto load = [&](uint32_t p) {
    m = val = 0;
    if (p < range.y) {
      val = vals[p];
      m = entry_mask<kMasks>(views, place, kMasks ? keys[p] : 0u, val, rec, log2_alpha_min);
    }
  };
  load(range.x + threadIdx.x);
  int buf = 0;
  for (uint32_t start = range.x; start < range.y; start += kCellThreads, buf ^= 1) {
    s_mask[buf][threadIdx.x] = m;
    s_val[buf][threadIdx.x] = val;
    load(start + kCellThreads + threadIdx.x);  // in flight while this chunk is written out
    __syncthreads();
    const uint32_t cnt = min((uint32_t)kCellThreads, range.y - start);
#pragma unroll 4
    for (uint32_t g = 0; g < cnt; g += 32) {
      const uint32_t mm = s_mask[buf][g + lane], vi = s_val[buf][g + lane];
      const bool in0 = (mm >> warp) & 1u, in1 = (mm >> (warp + kCellWarps)) & 1u;
      const unsigned b0 = __ballot_sync(0xffffffffu, in0), b1 = __ballot_sync(0xffffffffu, in1);
      const uint32_t p0 = run0.x + __popc(b0 & lt), p1 = run1.x + __popc(b1 & lt);
      if (in0 && p0 < run0.y) pairs[p0] = vi;
      if (in1 && p1 < run1.y) pairs[p1] = vi;
      run0.x += __popc(b0);
      run1.x += __popc(b1);
    }
  }
}

}  // namespace

// Blocks of the emission over up to `visible` entries.
int64_t emit_blocks(int64_t visible) {
  const int64_t tile = (int64_t)kEmitThreads * emit_items(visible);
  return (visible + tile - 1) / tile;
}
// The most blocks that any number of entries up to `visible` takes.
int64_t max_emit_blocks(int64_t visible) {
  return std::max(emit_blocks(visible), emit_blocks(std::min(visible, kEmitLong)));
}
int order_words() { return 2 * kOrderClasses; }

cudaError_t launch_emit_cells(const Views& views, int n, const uint32_t* order,
                              const Record* rec, float log2_alpha_min, int64_t visible_cap, uint32_t capacity,
                              uint32_t* keys, uint32_t* vals, Lookback lb, Counters* counters,
                              cudaStream_t stream) {
  const int64_t blocks = emit_blocks(visible_cap);
  cudaError_t e;
  if (blocks == 0) {
    e = launch_chained(no_cells_kernel, dim3(1), dim3(1), stream, counters);
  } else if (blocks > lb.capacity) {
    return cudaErrorInvalidValue;
  } else {
    const bool masks = cells_masked(views.total_cells);
    auto kernel = emit_items(visible_cap) == 1
                      ? (masks ? emit_cells_kernel<true, 1> : emit_cells_kernel<false, 1>)
                      : (masks ? emit_cells_kernel<true, kEmitItems>
                               : emit_cells_kernel<false, kEmitItems>);
    e = launch_chained(kernel, dim3((unsigned)blocks), dim3(kEmitThreads), stream, views, n, order,
                       rec, log2_alpha_min,
                       (uint32_t)std::min<int64_t>(visible_cap, 0xffffffffll), capacity, keys,
                       vals, lb, (uint32_t)blocks, counters);
  }
  RGS_LAUNCHED();
  return e;
}

cudaError_t launch_cell_ranges(const Views& views, const uint32_t* keys, int64_t n_keys,
                               uint2* ranges, const Counters* counters, cudaStream_t stream) {
  const int64_t per_block = kRangesKeys * kRangesThreads;
  if (n_keys <= 0) return cudaSuccess;
  const cudaError_t e =
      launch_chained(cell_ranges_kernel, dim3((unsigned)((n_keys + per_block - 1) / per_block)),
                     dim3(kRangesThreads), stream, keys, cells_masked(views.total_cells) ? 16 : 0,
                     (uint32_t)views.total_cells, ranges, counters);
  RGS_LAUNCHED();
  return e;
}

cudaError_t launch_tile_lists(const Views& views, const uint2* cell_ranges, const uint32_t* keys,
                              const uint32_t* vals, const Record* rec, float log2_alpha_min, uint32_t* tile_counts, uint2* ranges,
                              uint32_t* pairs, uint32_t capacity, uint32_t* order_words,
                              uint32_t* tile_order, Lookback lb, Counters* counters,
                              cudaStream_t stream) {
  const dim3 grid(views.total_cells), block(kCellThreads);
  const bool masks = cells_masked(views.total_cells);
  cudaError_t e = launch_chained(masks ? cell_count_kernel<true> : cell_count_kernel<false>, grid,
                                 block, stream, views, cell_ranges, keys, vals, rec,
                                 log2_alpha_min, tile_counts, order_words);
  RGS_LAUNCHED();
  if (e == cudaSuccess)
    e = launch_tile_ranges_scan(tile_counts, ranges, views.total_tiles, capacity,
                                &counters->n_pairs, &counters->n_pairs_listed, lb, stream);
  if (e == cudaSuccess) {
    e = launch_chained(masks ? cell_expand_kernel<true> : cell_expand_kernel<false>, grid, block,
                       stream, views, cell_ranges, keys, vals, rec, log2_alpha_min,
                       (const uint32_t*)tile_counts, (const uint2*)ranges, pairs, capacity,
                       (const uint32_t*)order_words, order_words + kOrderClasses, tile_order,
                       counters);
    RGS_LAUNCHED();
  }
  return e;
}

}  // namespace rgs

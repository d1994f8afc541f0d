// Stand-ins for the library's launchers: they check that the buffers they are given lie in live
// memory of the fake device and are large enough.
#pragma once

#include <cstdio>
#include <cstdlib>
#include <string>
#include <vector>

#include "fake_state.h"
#include "rgs_internal.cuh"

namespace rgs {
using fake::check;
int64_t cluster_sort_capacity(int) { return 0; }
int order_words() { return 66; }
int64_t max_emit_blocks(int64_t n) { return (n + 255) / 256; }
int preprocess_backward_blocks(int64_t n) { return (int)((n + 127) / 128); }

cudaError_t launch_preprocess_forward(const Views& views, const Consts&, const rgs_gaussians& g,
                                      Record* rec, uint32_t* depths, uint32_t* cand,
                                      uint32_t* vis_bits, bool, Counters* counters, cudaStream_t) {
  const size_t vn = (size_t)views.n_views * g.n;
  check(rec, sizeof(Record) * vn, "records");
  check(depths, 4 * vn, "depths");
  check(cand, 4 * vn, "candidates");
  check(vis_bits, 4 * views.n_views * vis_bit_words_per_view(g.n), "visibility bits");
  check(counters, sizeof(Counters), "counters");
  counters->all_visible = fake::visible;
  counters->all_cells = fake::cells;
  counters->all_pairs = fake::pairs;
  return cudaSuccess;
}
cudaError_t launch_colour(const Views&, const rgs_gaussians&, const uint32_t*, int64_t, Record*,
                          Counters*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_compact_visible(const uint32_t*, int n_views, int n, const uint32_t*,
                                   uint32_t* keys, uint32_t* vals, uint32_t* list, uint32_t*,
                                   Lookback, cudaStream_t) {
  const size_t vn = (size_t)n_views * n;
  check(keys, 4 * vn, "depth keys");
  check(vals, 4 * vn, "depth values");
  check(list, 4 * vn, "visible list");
  return cudaSuccess;
}
cudaError_t launch_radix_sort(uint32_t* keys, uint32_t* vals, uint32_t* keys_alt,
                              uint32_t* vals_alt, int64_t n, const uint32_t*, int, int,
                              uint32_t* hist, uint32_t* sums, bool* alt, cudaStream_t, int items) {
  for (uint32_t* p : {keys, vals, keys_alt, vals_alt})
    if (p) check(p, 4 * (size_t)n, "sort buffer");
  check(hist, 4 * (size_t)sort_hist_entries(n, items), "sort counts");
  check(sums, 4 * (size_t)(scan_blocks(sort_hist_entries(n, items)) + 1), "sort sums");
  *alt = n % 2 == 0;
  return cudaSuccess;
}
bool radix_sort_in_alt(int64_t n, int, int, int) { return n % 2 == 0; }
cudaError_t launch_emit_cells(const Views&, int, const uint32_t*, const Record*, float, int64_t,
                              uint32_t capacity, uint32_t* keys, uint32_t* vals, Lookback,
                              Counters*, cudaStream_t) {
  check(keys, 4 * (size_t)capacity, "cell keys");
  check(vals, 4 * (size_t)capacity, "cell values");
  return cudaSuccess;
}
cudaError_t launch_cell_ranges(const Views& views, const uint32_t*, int64_t, uint2* ranges,
                               const Counters*, cudaStream_t) {
  check(ranges, 8 * (size_t)views.total_cells, "cell ranges");
  return cudaSuccess;
}
cudaError_t launch_tile_lists(const Views& views, const uint2*, const uint32_t* keys,
                              const uint32_t* vals, const Record*, float, uint32_t* tile_counts,
                              uint2* ranges, uint32_t* pairs, uint32_t capacity, uint32_t*,
                              uint32_t* tile_order, Lookback, Counters*, cudaStream_t) {
  check(tile_counts, 4 * (size_t)views.total_tiles, "tile counts");
  check(ranges, 8 * (size_t)views.total_tiles, "tile ranges");
  check(tile_order, 4 * (size_t)views.total_tiles, "tile order");
  if (capacity) check(pairs, 4 * (size_t)capacity, "pairs");
  if (fake::one_place && fake::wrote_pairs && pairs != fake::wrote_pairs)
    check(nullptr, 0, "pairs written to another place than before");
  if (fake::one_place) fake::wrote_pairs = pairs;
  const char *a = reinterpret_cast<const char*>(pairs), *b = a + 4 * (size_t)capacity;
  for (const uint32_t* in : {keys, vals}) {  // the lists are read while the pairs are written
    const char* c = reinterpret_cast<const char*>(in);
    if (capacity && c >= a && c < b) fake::check(nullptr, 0, "pairs over the sorted cell list");
  }
  return cudaSuccess;
}
cudaError_t launch_blend(bool forward, const Views& views, const Consts&, const uint2* ranges,
                         const uint32_t* pairs, const Record* rec, float*, float*, float*,
                         float* t_final, int32_t* last, const float*, const float*, const float*,
                         float* g2d, const uint32_t*, Counters*, cudaStream_t) {
  check(ranges, 8 * (size_t)views.total_tiles, "blend's ranges");
  check(rec, sizeof(Record), "blend's records");
  check(pairs, 4 * (size_t)fake::pairs, "blend's pairs");
  if (fake::wrote_pairs && pairs != fake::wrote_pairs)
    check(nullptr, 0, "blend's pairs are not where a forward on this state wrote them");
  check(t_final, 4 * (size_t)views.total_pixels, "transmittances");
  check(last, 4 * (size_t)views.total_pixels, "last indices");
  if (!forward) check(g2d, 64, "gradient records");
  return cudaSuccess;
}
cudaError_t launch_preprocess_backward(const Views& views, const Consts&, const rgs_gaussians& g,
                                       unsigned long long* vis_mask, const uint32_t*,
                                       const Counters*, int64_t vn, float* g2d, uint32_t, float*,
                                       float*, float*, float*, float*, float* partial, float*,
                                       const MapReg* reg, cudaStream_t) {
  check(vis_mask, 8 * (size_t)g.n, "visibility masks");
  check(g2d, 64 * (size_t)vn, "gradient records");
  check(partial, 4 * (size_t)preprocess_backward_blocks(vn) * views.n_views * 6, "pose partials");
  if (reg && reg->values) check(reg->values, 4 * (size_t)g.n, "regulariser values");
  return cudaSuccess;
}
// Not reached by these tests.
cudaError_t launch_pose_prepare(const float*, int, float*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_grad_weight(const Views&, const float*, float, float*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_track_loss(const Views&, const float*, const float*, const float*, const float*, float, bool, double*, float*, double*, float*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_pose_adam(int, float, float, float, float, int, const float*, float*, int32_t*, float*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_covisibility(const float*, const float*, int64_t, int, float, unsigned long long*, float*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_map_ema(int64_t, const float*, float*, float, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_prune_mask(int64_t, const float*, const float*, const uint32_t*, const float*, float, float, uint32_t, float, uint8_t*, uint32_t*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_exclusive_scan(const uint32_t*, uint32_t*, int64_t, const uint32_t*, uint32_t*, uint32_t*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_exclusive_scan_single_pass(const uint32_t*, uint32_t*, int64_t, uint32_t*, Lookback, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_triangulate(const SeedCams&, const SeedConsts&, int64_t, int, const int32_t*, const double*, const int32_t*, const double*, const float*, uint32_t*, double*, int32_t*, double*, double*, float*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_accept_points(const SeedScratch&, int64_t, int, const uint32_t*, const int32_t*, const double*, double, double, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_seeds(const SeedScratch&, const SeedCams&, const SeedConsts&, const CellPack (&)[2], int, int, int, const int32_t*, const int32_t*, const double*, const double*, const double*, const float*, const float*, const float*, int32_t*, float*, float*, float*, float*, float*, float*, cudaStream_t) { return cudaSuccess; }
}  // namespace rgs

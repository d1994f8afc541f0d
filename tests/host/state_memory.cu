// Host-side scenarios of the context's states on the fake device; one per run, named by argv[1].
#include <cstring>

#include "fake_launchers.h"

using namespace rgs;

namespace {

struct Images {
  std::vector<float> color, depth, alpha;
  rgs_images get(int pixels) {
    color.resize(3 * pixels);
    depth.resize(pixels);
    alpha.resize(pixels);
    return rgs_images{color.data(), depth.data(), alpha.data()};
  }
};

rgs_ctx* make_context() {
  rgs_ctx* ctx = nullptr;
  if (rgs_create(&ctx, 0) != RGS_OK) std::exit(2);
  return ctx;
}

// A forward of `views` views of w x w pixels and n Gaussians that counts `count` of everything.
rgs_status forward(rgs_ctx* ctx, int n, int w, unsigned long long count, uint64_t* state,
                   int views = 1) {
  static Images images;
  alignas(16) static float parameters[4];
  fake::visible = count < (unsigned long long)n * views ? count : (unsigned long long)n * views;
  fake::cells = count;
  fake::pairs = fake::pairs_per_cell * count;
  std::vector<rgs_camera> cams(views);
  for (rgs_camera& c : cams) {
    c = rgs_camera{};
    c.width = c.height = w;
    c.fx = c.fy = 100.0f;
    c.world_to_cam[0] = c.world_to_cam[5] = c.world_to_cam[10] = 1.0f;
  }
  const rgs_gaussians g{n, 0, parameters, parameters, parameters, parameters, parameters};
  rgs_images out = images.get(views * w * w);
  return rgs_render_forward(ctx, &g, cams.data(), views, nullptr, &out, state, nullptr);
}

rgs_status backward(rgs_ctx* ctx, uint64_t state, bool reg = false) {
  alignas(16) static float grads[4];
  static double value;
  const rgs_image_grads up{grads, nullptr, nullptr};
  rgs_map_reg r{};
  r.value = &value;
  return rgs_render_backward_mapping(ctx, state, &up, RGS_GRAD_ALL, grads, grads, grads, grads,
                                     grads, grads, reg ? &r : nullptr, nullptr);
}

int failures = 0;
#define EXPECT(x)                                            \
  do {                                                       \
    if (!(x)) {                                              \
      ++failures;                                            \
      std::printf("line %d: %s does not hold\n", __LINE__, #x); \
    }                                                        \
  } while (0)

// A forward that runs out of memory at any of its allocations leaves nothing behind that a later,
// smaller forward on the same state would use.
void failed_growth() {
  const struct { int n, w, views; unsigned long long count; } larger[] = {
      {5000, 64, 1, 6000},    // per Gaussian
      {1000, 64, 8, 6000},    // per entry
      {1000, 300, 1, 6000},   // per pixel and tile
      {1000, 64, 1, 900000},  // the lists and the sort's scratch
  };
  for (const auto& l : larger) {
    for (size_t room = 0;; room += 4096) {
      rgs_ctx* ctx = make_context();
      uint64_t s = 0;
      EXPECT(forward(ctx, 1000, 64, 6000, &s) == RGS_OK);
      EXPECT(backward(ctx, s, true) == RGS_OK);
      fake::limit = fake::live + room;
      const rgs_status st = forward(ctx, l.n, l.w, l.count, &s, l.views);
      EXPECT(st == RGS_OK || st == RGS_ERR_NOMEM);
      if (st == RGS_OK) backward(ctx, s, true);  // its scratch may fail, too
      rgs_stats stats;
      EXPECT(rgs_query_stats(ctx, s, &stats, nullptr) == RGS_OK);
      fake::limit = SIZE_MAX;
      EXPECT(forward(ctx, 1000, 64, 6000, &s) == RGS_OK);
      EXPECT(backward(ctx, s, true) == RGS_OK);
      rgs_destroy(ctx);
      EXPECT(fake::live == 0);
      if (st == RGS_OK) break;
    }
  }
}

// A forward that fails after it created its state leaves none: the handle stays 0, the memory is
// free again (a kept state that it took, too), and a capture is not disturbed.
void failed_first() {
  for (int kept = 0; kept < 2; ++kept) {
    for (size_t room = 0;; room += 4096) {
      rgs_ctx* ctx = make_context();
      const size_t bare = fake::live;
      uint64_t s = 0;
      if (kept) {
        EXPECT(forward(ctx, 1000, 64, 6000, &s) == RGS_OK);
        EXPECT(rgs_release_state(ctx, s) == RGS_OK);
        s = 0;
      }
      fake::limit = bare + room;
      const rgs_status st = forward(ctx, 2000, 100, 20000, &s);
      fake::limit = SIZE_MAX;
      if (st != RGS_OK) {
        EXPECT(st == RGS_ERR_NOMEM && s == 0 && fake::live == bare);
        EXPECT(std::strlen(rgs_last_error(ctx)) > 0);
      }
      rgs_destroy(ctx);
      if (st == RGS_OK) break;
    }
  }
  rgs_ctx* ctx = make_context();
  uint64_t s = 0;
  fake::capturing = true;
  EXPECT(forward(ctx, 1000, 64, 6000, &s) == RGS_ERR_CAPACITY && s == 0);
  EXPECT(forward(ctx, 0, 64, 0, &s) == RGS_ERR_CAPACITY && s == 0);
  EXPECT(fake::unsafe == 0);
  fake::capturing = false;
  // A named state outlives a call that fails on it.
  EXPECT(forward(ctx, 1000, 64, 6000, &s) == RGS_OK);
  fake::limit = fake::live;
  const uint64_t named = s;
  EXPECT(forward(ctx, 2000, 100, 20000, &s) == RGS_ERR_NOMEM && s == named);
  fake::limit = SIZE_MAX;
  EXPECT(rgs_release_state(ctx, s) == RGS_OK);
  rgs_destroy(ctx);
}

// Every allocation of the library frees the kept states before it fails, and the bound on what is
// kept counts all that a state holds.
void kept_states_give_way() {
  void *keys, *vals;
  cudaMalloc(&keys, 4 * 5000);
  cudaMalloc(&vals, 4 * 5000);
  for (int call = 0; call < 3; ++call) {
    rgs_ctx* ctx = make_context();
    const size_t bare = fake::live;
    uint64_t s = 0;
    EXPECT(forward(ctx, 200000, 64, 6000, &s) == RGS_OK);
    const size_t before = fake::live;
    EXPECT(backward(ctx, s, true) == RGS_OK);
    rgs_stats stats;
    EXPECT(rgs_query_stats(ctx, s, &stats, nullptr) == RGS_OK);
    EXPECT(fake::live - before == 4 * 200000);  // the regulariser's scratch
    EXPECT((size_t)stats.state_bytes == fake::live - bare);
    EXPECT(rgs_release_state(ctx, s) == RGS_OK);
    EXPECT(fake::live > bare);
    fake::limit = fake::live;  // nothing is left but what is kept
    rgs_status st = RGS_ERR_INVALID_ARG;
    uint32_t *k = static_cast<uint32_t*>(keys), *v = static_cast<uint32_t*>(vals);
    if (call == 0) st = rgs_radix_sort_u32(ctx, k, v, 5000, 0, 32, nullptr);
    if (call == 1) st = rgs_exclusive_scan_u32(ctx, k, v, 5000, nullptr, nullptr);
    if (call == 2) {
      alignas(16) static float parameters[4];
      const rgs_gaussians g{100, 0, parameters, parameters, parameters, parameters, parameters};
      rgs_camera cam{};
      cam.width = cam.height = 32;
      cam.fx = cam.fy = 100.0f;
      rgs_config cfg;
      rgs_config_default(&cfg);
      fake::visible = fake::cells = fake::pairs = 100;
      st = rgs_autotune(ctx, &g, &cam, 1, &cfg, nullptr, nullptr);
    }
    EXPECT(st == RGS_OK);
    fake::limit = SIZE_MAX;
    rgs_destroy(ctx);
    EXPECT(fake::live == 2 * 4 * 5000);
  }
  cudaFree(keys);
  cudaFree(vals);
}

// List positions are signed 32-bit numbers in the blends: more pairs or cell entries than those
// hold are refused, by the forward and by rgs_reserve, and capacities with their slack stay below.
void list_limits() {
  const unsigned long long most = 2147483647ull;
  rgs_ctx* ctx = make_context();
  const size_t bare = fake::live;
  uint64_t s = 0;
  EXPECT(rgs_reserve(ctx, &s, (int64_t)most + 1, nullptr) == RGS_ERR_INVALID_ARG);
  EXPECT(s == 0 && fake::live == bare);
  for (unsigned long long count : {most + 1, 3000000000ull, 4294967294ull, 5000000000ull}) {
    EXPECT(forward(ctx, 1000, 64, count, &s) == RGS_ERR_INVALID_ARG);
    EXPECT(s == 0 && fake::live == bare);
  }
  for (unsigned long long count : {1800000000ull, most}) {
    EXPECT(forward(ctx, 1000, 64, count, &s) == RGS_OK);
    rgs_stats stats;
    EXPECT(rgs_query_stats(ctx, s, &stats, nullptr) == RGS_OK);
    EXPECT(stats.pair_capacity == (int64_t)most);
  }
  rgs_destroy(ctx);
}

// Reserved pairs take 16 bytes each (and a quarter more of them), and serve forwards under capture
// with as many pairs and cells, whichever of the two is larger, before and after eager ones.
void reserved_pairs() {
  const int64_t asked = 1000000;
  rgs_ctx* ctx = make_context();
  uint64_t s = 0;
  EXPECT(forward(ctx, 1000, 64, 100, &s) == RGS_OK);
  const size_t before = fake::live;
  EXPECT(rgs_reserve(ctx, &s, asked, nullptr) == RGS_OK);
  const size_t grown = fake::live - before;
  const size_t scratch = 1 << 20;  // the sort's tables
  EXPECT(grown >= 16 * (size_t)asked && grown <= 20 * (size_t)asked + scratch);
  rgs_stats stats;
  EXPECT(rgs_query_stats(ctx, s, &stats, nullptr) == RGS_OK);
  EXPECT(stats.pair_capacity >= asked);
  for (int round = 0; round < 2; ++round) {
    fake::capturing = true;
    EXPECT(forward(ctx, 1000, 64, asked, &s) == RGS_OK);
    EXPECT(backward(ctx, s) == RGS_OK);
    fake::capturing = false;
    EXPECT(fake::live - before == grown);
    EXPECT(forward(ctx, 1000, 64, asked, &s) == RGS_OK);  // nothing grows
    EXPECT(backward(ctx, s) == RGS_OK);
    EXPECT(fake::live - before == grown);
  }
  // Eager and captured forwards write to one place: a backward after a replay reads what it wrote.
  fake::one_place = true;
  for (unsigned long long count : {50ull, 51ull, 999999ull}) {
    EXPECT(forward(ctx, 1000, 64, count, &s) == RGS_OK);
    fake::capturing = true;
    EXPECT(forward(ctx, 1000, 64, count, &s) == RGS_OK);
    fake::capturing = false;
    EXPECT(backward(ctx, s) == RGS_OK);
  }
  fake::one_place = false;
  fake::wrote_pairs = nullptr;
  fake::pairs_per_cell = 8;
  EXPECT(forward(ctx, 1000, 64, asked, &s) == RGS_OK);
  EXPECT(rgs_query_stats(ctx, s, &stats, nullptr) == RGS_OK);
  EXPECT(stats.pair_capacity >= 8 * asked);
  fake::pairs_per_cell = 1;
  EXPECT(forward(ctx, 1000, 64, asked, &s) == RGS_OK);
  EXPECT(fake::unsafe == 0);
  rgs_destroy(ctx);
}

// A reserve between a forward and its backward leaves the forward's pairs readable, wherever they
// lie, also when it fails; one that fails on a state it created leaves none.
void reserve_after_forward() {
  for (unsigned long long per_cell : {1ull, 8ull}) {
    for (size_t room = 0;; room += 1 << 16) {
      fake::pairs_per_cell = per_cell;
      rgs_ctx* ctx = make_context();
      uint64_t s = 0;
      EXPECT(forward(ctx, 1000, 64, 20000, &s) == RGS_OK);
      fake::limit = fake::live + room;
      const rgs_status st = rgs_reserve(ctx, &s, 1000000, nullptr);
      fake::limit = SIZE_MAX;
      EXPECT(st == RGS_OK || st == RGS_ERR_NOMEM);
      EXPECT(backward(ctx, s) == RGS_OK);
      EXPECT(forward(ctx, 1000, 64, 20000, &s) == RGS_OK);
      EXPECT(backward(ctx, s) == RGS_OK);
      rgs_destroy(ctx);
      EXPECT(fake::live == 0);
      if (st == RGS_OK) break;
    }
  }
  fake::pairs_per_cell = 1;
  rgs_ctx* ctx = make_context();
  const size_t bare = fake::live;
  uint64_t s = 0;
  fake::limit = bare + 1000;
  EXPECT(rgs_reserve(ctx, &s, 1000000, nullptr) == RGS_ERR_NOMEM && s == 0 && fake::live == bare);
  fake::limit = SIZE_MAX;
  rgs_destroy(ctx);
}

// What is kept after a release is bounded, is not kept while memory is scarce, and is given back.
void kept_memory() {
  for (size_t room : {(size_t)0, fake::total / 8 - (1u << 20), fake::total / 8 + (1u << 20)}) {
    rgs_ctx* ctx = make_context();
    const size_t bare = fake::live;
    uint64_t a = 0, b = 0, c = 0;
    EXPECT(forward(ctx, 1000, 64, 6000, &a) == RGS_OK);
    EXPECT(forward(ctx, 1000000, 64, 6000, &b) == RGS_OK);   // 150 MB
    EXPECT(forward(ctx, 60000000, 64, 6000, &c) == RGS_OK);  // 9 GB
    fake::limit = fake::live + room;
    EXPECT(rgs_release_state(ctx, a) == RGS_OK);  // small: kept
    EXPECT(fake::live > bare + (150u << 20));
    EXPECT(rgs_release_state(ctx, c) == RGS_OK);  // beyond the bound
    fake::limit = fake::live + room;
    const size_t with_b = fake::live;
    EXPECT(rgs_release_state(ctx, b) == RGS_OK);
    const bool scarce = room < fake::total / 8;
    EXPECT(scarce ? fake::live == bare : fake::live == with_b);
    EXPECT(fake::live - bare <= fake::total / 64);
    EXPECT(rgs_trim(ctx) == RGS_OK);
    EXPECT(fake::live == bare);
    uint64_t s = 0;
    fake::limit = SIZE_MAX;
    EXPECT(forward(ctx, 1000, 64, 6000, &s) == RGS_OK);
    EXPECT(backward(ctx, s) == RGS_OK);
    rgs_destroy(ctx);
    EXPECT(fake::live == 0);
  }
  EXPECT(rgs_trim(nullptr) == RGS_ERR_INVALID_ARG);
}

}  // namespace

int main(int argc, char** argv) {
  const std::string which = argc > 1 ? argv[1] : "";
  if (which == "failed_growth") failed_growth();
  else if (which == "failed_first") failed_first();
  else if (which == "kept_states_give_way") kept_states_give_way();
  else if (which == "list_limits") list_limits();
  else if (which == "reserved_pairs") reserved_pairs();
  else if (which == "kept_memory") kept_memory();
  else if (which == "reserve_after_forward") reserve_after_forward();
  else return 2;
  EXPECT(fake::stale == 0);
  return failures ? 1 : 0;
}

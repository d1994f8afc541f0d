// raster.cu -- the forward and backward alpha blends.
//
// Forward blend (Section 3.1, Eq. alpha; Section 3.2.2): one CTA per (view, tile), the tiles
// taken longest run first; the tile's Gaussians, already in near-to-far order, are staged
// through shared memory in batches of one Gaussian per thread and every thread composites its
// pixels front to back with early exit.
// Backward blend: the same tiles are walked back to front from each pixel's last contributor,
// recovering the transmittance by division from the saved final value, so no per-pixel list is
// stored; per-Gaussian screen-space gradient sums are reduced per warp through shared memory, in
// groups of Gaussians, before one atomic per value and Gaussian.
#include <algorithm>
#include <type_traits>

#include "rgs_internal.cuh"

namespace rgs {
namespace {

// ------------------------------------------------------------------------------------------
// Staging of a batch of Gaussians in shared memory, with the row terms of the tile's anchor row
// y_a (anchor_terms), as 16-byte rows:
//   column  (mx hi, mx lo), (l11, c21): what a thread needs once for its column
//   shape   (l21, l22), (s_a, -log2 o)
//   colour  (r, g), (b, z)
// For an even number of pixels per thread the packed f32x2 arithmetic of two pixels reads shape
// and colour as (x, x) pairs. Stored doubled (two rows in place of one) they arrive paired; stored
// once, a thread pairs them with register moves. The blends are bound by instruction issue and
// wait on their shared-memory reads in between (a 16-byte broadcast row is one instruction and two
// wavefronts of a pipe that is 44 to 52 % busy), so what is best depends on how many pixel pairs
// share a read, and was measured:
// Blends of 16 views of 1080p, by rows per Gaussian (column row single, the others as said):
//   forward, 4 pixels: all doubled, column row too 2.97 ms, 2.82 with it single; shape single 2.64;
//     shape and colour single 2.86
//   forward, 8 pixels: 2.98, 2.93, 2.81, 2.56
//   backward, 8 pixels: 4.39, 4.32, 4.50, 4.47
// For the backward the z of a doubled colour gives its place to r_g: (b, b), (z, r_g), with r_g the
// row of the tile nearest to where the footprint's ridge (in each column the point of largest
// weight, dy = -l11 l21 dx / (l21^2 + l22^2)) crosses the tile's middle column, relative to the
// anchor row. The backward sums its moments about that row: the pixels that a tilted footprint
// covers lie around its ridge, not around its centre, which may be many tiles away. Error of the
// second moment across thin footprints of any tilt, in units of the moment: 2.0e-6 about the
// ridge's row, 6.0e-6 about the row nearest to the centre, 3.7e-6 about the anchor row.
// ------------------------------------------------------------------------------------------
template <bool kBackward, int PPT>
struct StageLayout {
  static constexpr bool kPacked = PPT % 2 == 0;
  static constexpr bool kShapeTwice = kPacked && kBackward;
  static constexpr bool kColourTwice = kPacked && (kBackward || PPT < 8);
  static constexpr int kShape = 1;
  static constexpr int kColour = kShape + (kShapeTwice ? 2 : 1);
  static constexpr int kRows = kColour + (kColourTwice ? 2 : 1);
};

template <int kTileH, bool kBackward, int PPT, int R, int N>
__device__ __forceinline__ void stage_gaussian(ulonglong2 (&sp)[R][N], int t, float4 r0,
                                               float4 r1, float4 r2, float x_m, float y_a) {
  using L = StageLayout<kBackward, PPT>;
  static_assert(R == L::kRows, "rows of the layout");
  const AnchorTerms at = anchor_terms(r0, r1, y_a);
  const float nlo = -r1.w;
  sp[0][t] = make_ulonglong2(f2_make(r0.x, r0.z), f2_make(r1.x, at.c21));
  if constexpr (L::kShapeTwice) {
    sp[L::kShape][t] = make_ulonglong2(f2_make(r1.y, r1.y), f2_make(r1.z, r1.z));
    sp[L::kShape + 1][t] = make_ulonglong2(f2_make(at.s_a, at.s_a), f2_make(nlo, nlo));
  } else {
    sp[L::kShape][t] = make_ulonglong2(f2_make(r1.y, r1.z), f2_make(at.s_a, nlo));
  }
  if constexpr (L::kColourTwice) {
    float last = r2.w;
    if constexpr (kBackward) {
      // An undefined quotient (an exponent that underflows) leaves the tile's first row.
      const float ridge = __fdividef(r1.x * r1.y * (r0.x - x_m), fmaf(r1.y, r1.y, r1.z * r1.z));
      last = fminf(fmaxf(rintf(ridge - at.dya), (float)(-kTileH / 2)),
                   (float)(kTileH - 1 - kTileH / 2));
    }
    sp[L::kColour][t] = make_ulonglong2(f2_make(r2.x, r2.x), f2_make(r2.y, r2.y));
    sp[L::kColour + 1][t] = make_ulonglong2(f2_make(r2.z, r2.z), f2_make(r2.w, last));
  } else {
    sp[L::kColour][t] = make_ulonglong2(f2_make(r2.x, r2.y), f2_make(r2.z, r2.w));
  }
}

// Two values of a row as (x, x), (y, y).
__device__ __forceinline__ ulonglong2 f2_spread(f32x2 v) {
  return make_ulonglong2(f2_make(f2_lo(v), f2_lo(v)), f2_make(f2_hi(v), f2_hi(v)));
}
// Staged Gaussian g for the packed arithmetic: column row, (l21, l22), (s_a, -log2 o), (r, g),
// (b, z or (z, r_g)), each value of the last four twice.
struct Staged {
  ulonglong2 column, l2, sn, rg, bz;
};
template <bool kBackward, int PPT, int R, int N>
__device__ __forceinline__ Staged staged(const ulonglong2 (&sp)[R][N], int g) {
  using L = StageLayout<kBackward, PPT>;
  Staged s;
  s.column = sp[0][g];
  s.l2 = sp[L::kShape][g];
  if constexpr (L::kShapeTwice) {
    s.sn = sp[L::kShape + 1][g];
  } else {
    s.sn = f2_spread(s.l2.y);
    s.l2 = f2_spread(s.l2.x);
  }
  s.rg = sp[L::kColour][g];
  if constexpr (L::kColourTwice) {
    s.bz = sp[L::kColour + 1][g];
  } else {
    s.bz = f2_spread(s.rg.y);
    s.rg = f2_spread(s.rg.x);
  }
  return s;
}
// t of a thread's column at the anchor row, from the column row.
__device__ __forceinline__ float column_t(float fx, ulonglong2 x) {
  return __fmaf_rn(f2_lo(x.y), __fsub_rn(__fsub_rn(fx, f2_lo(x.x)), f2_hi(x.x)), f2_hi(x.y));
}

// ------------------------------------------------------------------------------------------
// Forward blend. A CTA covers one TW x TH tile with TW * TH / PPT threads; thread t owns the
// PPT vertically adjacent pixels (x, y0 + k), k < PPT, of column x = t % TW, so every Gaussian
// staged in shared memory is read once per thread and evaluated for PPT pixels. With an even PPT
// the pixels go in pairs through packed f32x2 arithmetic: a pixel that does not composite a
// Gaussian gets weight +0, which leaves its colour, depth and transmittance bit-identical, so the
// result equals the one-pixel-per-thread kernel's. Alpha is zeroed where it is below alpha_min
// before the weight is formed, so a live pixel composites its weight unconditionally and only
// the rare stop (its transmittance would fall below t_min) branches. A pixel that has stopped, or
// lies off the image, gets a row offset of 1e18 from the anchor row: its exponent is then
// astronomically large, its alpha 0, and it keeps its colour and transmittance with no per-pixel
// test in the loop.
// For the backward each pixel saves the last list position it may composite: the one before its
// stop, or the tile's last position if it never stops (between its last contributor and that
// position no Gaussian covers it, so the backward takes the same decisions there).
// ------------------------------------------------------------------------------------------
template <int TW, int TH, int PPT>
__global__ void __launch_bounds__(TW * TH / PPT) blend_forward_kernel(
    const __grid_constant__ Views views, const Consts c, const uint2* __restrict__ ranges,
    const uint32_t* __restrict__ pair_vals, const Record* __restrict__ rec, float* __restrict__ color,
    float* __restrict__ depth, float* __restrict__ alpha_out, float* __restrict__ t_final,
    int32_t* __restrict__ last_index, const uint32_t* __restrict__ tile_order,
    Counters* __restrict__ counters) {
  chain_wait();
  constexpr int kThreads = TW * TH / PPT;
  constexpr bool kPacked = PPT % 2 == 0;
  constexpr int P2 = kPacked ? PPT / 2 : 1;
  static_assert(kThreads % 32 == 0, "whole warps only");
  __shared__ ulonglong2 sp[StageLayout<false, PPT>::kRows][kThreads];
  __shared__ unsigned long long s_eval[kThreads / 32];
  const int gtile = (int)tile_order[blockIdx.x];
  const int v = view_of_tile(views, gtile);
  const ViewParams& vp = views.v[v];
  const int local = gtile - vp.tile_base;
  const int ty = local / vp.tiles_x, tx = local - ty * vp.tiles_x;
  const int px = tx * TW + (int)(threadIdx.x % TW);
  const int py0 = ty * TH + (int)(threadIdx.x / TW) * PPT;
  const float fx = (float)px;
  // Anchor row of the tile's row terms, and the thread's first row relative to it.
  const float x_m = (float)(tx * TW) + 0.5f * (float)(TW - 1), y_a = (float)(ty * TH + TH / 2);
  const int r0_ = (int)(threadIdx.x / TW) * PPT - TH / 2;
  const uint2 range = ranges[gtile];

  float T[PPT], C0[PPT], C1[PPT], C2[PPT], D[PPT];
  f32x2 T2[P2], C02[P2], C12[P2], C22[P2], D2[P2], FR[P2];
  uint32_t visited_end[PPT];  // one past the last list position the pixel visited
  bool done[PPT];             // the pixel has stopped (or is off the image)
  int live = 0;               // pixels of the thread that have not stopped
  // Row offset of a pixel that takes no further part: every Gaussian's alpha there is 0.
  constexpr float kFarRow = 1e18f;
#pragma unroll
  for (int k = 0; k < PPT; ++k) {
    done[k] = !(px < vp.width && py0 + k < vp.height);
    T[k] = 1.0f;
    C0[k] = C1[k] = C2[k] = D[k] = 0.0f;
    visited_end[k] = done[k] ? range.x : range.y;
    live += done[k] ? 0 : 1;
  }
#pragma unroll
  for (int q = 0; q < P2; ++q) {
    const int k0 = kPacked ? 2 * q : 0, k1 = kPacked ? 2 * q + 1 : 0;
    T2[q] = f2_make(1.0f, 1.0f);
    C02[q] = C12[q] = C22[q] = D2[q] = f2_make(0.0f, 0.0f);
    FR[q] = f2_make(done[k0] ? kFarRow : (float)(r0_ + k0), done[k1] ? kFarRow : (float)(r0_ + k1));
  }

  // One staged Gaussian (list position pos, slot g) against the thread's pixel pairs.
  auto composite_pairs = [&](uint32_t pos, int g) {
    const Staged st = staged<false, PPT>(sp, g);
    // Whitened offset t at the anchor row of the thread's column (Eq. alpha's exponent).
    const float ta = column_t(fx, st.column);
    const f32x2 TA = f2_make(ta, ta);
#pragma unroll
    for (int q = 0; q < P2; ++q) {
      const int k0 = 2 * q, k1 = 2 * q + 1;
      const f32x2 tt = f2_fma(FR[q], st.l2.x, TA);
      const f32x2 ss = f2_fma(FR[q], st.l2.y, st.sn.x);
      const f32x2 nq = f2_fma(tt, tt, f2_fma(ss, ss, st.sn.y));  // -log2(o G)
      const float a0 = fminf(c.alpha_max, ex2_neg_approx(f2_lo(nq)));
      const float a1 = fminf(c.alpha_max, ex2_neg_approx(f2_hi(nq)));
      // w = alpha T and the transmittance after this Gaussian T' = T - w; an uncovered pixel
      // (alpha < alpha_min) has w = +0 and T' = T.
      f32x2 w = f2_mul(f2_make(a0 >= c.alpha_min ? a0 : 0.0f, a1 >= c.alpha_min ? a1 : 0.0f),
                       T2[q]);
      f32x2 Tn = f2_sub(T2[q], w);
      const bool stop0 = f2_lo(Tn) < c.t_min, stop1 = f2_hi(Tn) < c.t_min;
      if (stop0 || stop1) {  // once per pixel: it composites nothing from here on
        const float t0 = f2_lo(T2[q]), t1 = f2_hi(T2[q]);
        w = f2_make(stop0 ? 0.0f : f2_lo(w), stop1 ? 0.0f : f2_hi(w));
        Tn = f2_make(stop0 ? t0 : f2_lo(Tn), stop1 ? t1 : f2_hi(Tn));
        FR[q] = f2_make(stop0 ? kFarRow : f2_lo(FR[q]), stop1 ? kFarRow : f2_hi(FR[q]));
        if (stop0) visited_end[k0] = pos + 1;
        if (stop1) visited_end[k1] = pos + 1;
        live -= (int)stop0 + (int)stop1;
      }
      C02[q] = f2_fma(w, st.rg.x, C02[q]);
      C12[q] = f2_fma(w, st.rg.y, C12[q]);
      C22[q] = f2_fma(w, st.bz.x, C22[q]);
      D2[q] = f2_fma(w, st.bz.y, D2[q]);
      T2[q] = Tn;
    }
  };

  for (uint32_t start = range.x; start < range.y; start += kThreads) {
    if (__syncthreads_count(live == 0) == kThreads) break;
    const uint32_t j = start + threadIdx.x;
    if (j < range.y) {
      const uint32_t vi = pair_vals[j];
      stage_gaussian<TH, false, PPT>(sp, threadIdx.x, rec[vi].mean, rec[vi].conic,
                                     rec[vi].colour, x_m, y_a);
    }
    __syncthreads();
    const int cnt = (int)min((uint32_t)kThreads, range.y - start);
    // The warp leaves the batch together, once none of its pixels is live: a stopped pixel
    // composites nothing more (its alpha is 0), and a loop without per-thread exits ran 9 %
    // faster than one that let each thread leave on its own. The vote is taken before a visit and
    // followed after it, so that it waits for nothing (a view of 160x120: 33 -> 29 us; the one
    // visit more changes nothing).
    for (int g = 0; g < cnt; ++g) {
      const bool go_on = __any_sync(0xffffffffu, live > 0);
      const uint32_t pos = start + g;
      if constexpr (kPacked) {
        // Always with the clamp: a warp-uniform clamp-free variant (as in the backward) made
        // this loop slower (two copies of its body), measured 3.64 against 3.21 ms on the
        // 16-view 1080p window.
        composite_pairs(pos, g);
      } else {
        const float4 g0 = reinterpret_cast<const float4*>(sp[0])[g];
        const float4 g1 = reinterpret_cast<const float4*>(sp[1])[g];
        const float4 g2 = reinterpret_cast<const float4*>(sp[2])[g];
        const float ta = __fmaf_rn(g0.z, __fsub_rn(__fsub_rn(fx, g0.x), g0.y), g0.w);
#pragma unroll
        for (int k = 0; k < PPT; ++k) {
          if (!done[k]) {
            const float nq = neg_log2_og(ta, g1.z, g1.x, g1.y, g1.w, (float)(r0_ + k));
            const float a = fminf(c.alpha_max, ex2_neg_approx(nq));
            if (a >= c.alpha_min) {
              const float w = __fmul_rn(a, T[k]);
              const float Tn = __fsub_rn(T[k], w);
              if (Tn < c.t_min) {
                done[k] = true;
                visited_end[k] = pos + 1;
                --live;
              } else {
                C0[k] = fmaf(w, g2.x, C0[k]);
                C1[k] = fmaf(w, g2.y, C1[k]);
                C2[k] = fmaf(w, g2.z, C2[k]);
                D[k] = fmaf(w, g2.w, D[k]);
                T[k] = Tn;
              }
            }
          }
        }
      }
      if (!go_on) break;
    }
  }
  if constexpr (kPacked) {
#pragma unroll
    for (int q = 0; q < P2; ++q) {
      done[2 * q] = f2_lo(FR[q]) == kFarRow;
      done[2 * q + 1] = f2_hi(FR[q]) == kFarRow;
      T[2 * q] = f2_lo(T2[q]);
      T[2 * q + 1] = f2_hi(T2[q]);
      C0[2 * q] = f2_lo(C02[q]);
      C0[2 * q + 1] = f2_hi(C02[q]);
      C1[2 * q] = f2_lo(C12[q]);
      C1[2 * q + 1] = f2_hi(C12[q]);
      C2[2 * q] = f2_lo(C22[q]);
      C2[2 * q + 1] = f2_hi(C22[q]);
      D[2 * q] = f2_lo(D2[q]);
      D[2 * q + 1] = f2_hi(D2[q]);
    }
  }
  uint32_t evals = 0;
#pragma unroll
  for (int k = 0; k < PPT; ++k) {
    evals += visited_end[k] - range.x;
    const int py = py0 + k;
    if (px < vp.width && py < vp.height) {
      const long long pix = vp.pixel_offset + (long long)py * vp.width + px;
      color[3 * pix + 0] = fmaf(T[k], c.bg[0], C0[k]);
      color[3 * pix + 1] = fmaf(T[k], c.bg[1], C1[k]);
      color[3 * pix + 2] = fmaf(T[k], c.bg[2], C2[k]);
      depth[pix] = D[k];
      alpha_out[pix] = 1.0f - T[k];
      t_final[pix] = T[k];
      // The last position the pixel may composite (stop position - 1, or the tile's last).
      last_index[pix] = done[k] ? (int32_t)visited_end[k] - 2 : (int32_t)range.y - 1;
    }
  }
  // Visited (pixel, Gaussian) positions, for the roofline accounting.
  unsigned long long e = evals;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  if ((threadIdx.x & 31) == 0) s_eval[threadIdx.x >> 5] = e;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long s = 0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) s += s_eval[w];
    atomicAdd(&counters->n_eval, s);
  }
}

// ------------------------------------------------------------------------------------------
// Per-warp reduction of the visited Gaussians' gradient sums through shared memory. Each visit
// writes the lane's sums, two by two, as one 8-byte column of kPairs rows (row kPairs b + p for
// pair p of the b-th Gaussian of the group, RedLayout); after kBatch visits (or at the end of a
// staged batch) every lane adds up one row (sixteen 16-byte reads of a row of 32 pairs padded to
// 68 floats: the column writes and the row reads are both free of bank conflicts) and parks the
// totals in the padding. Lane b then turns Gaussian b's totals into its whitened moments and
// issues the atomics. Per visit this costs kPairs shared stores and a share of the row sums, in
// place of a shuffle butterfly with its selects after every Gaussian; single values in rows of 32
// floats took nine stores and two row passes per seven Gaussians (+3 % on the 16-view 1080p window,
// +8 % on ten 640x480 views).
//
// The lane's values: sdp, sr | srr, t_a sdp | t_a sr, t_a^2 sdp | gr, gg | gb, gz, with sdp, sr,
// srr the sums of dp, dp r and dp r^2 over its pixels (r the row offset from row r_g; from the
// tile's anchor row with one pixel per thread), t_a the whitened offset of its column at that row, and gr .. gz the colour and depth weights (gz 0 without a depth
// or opacity gradient).
// ------------------------------------------------------------------------------------------
constexpr int kRedPad = 68;  // floats per row of 32 lane pairs, padded

struct RedLayout {
  static constexpr int kPairs = 5;
  static constexpr int kBatch = 6;  // kPairs * kBatch <= 32: one row pass
  static constexpr int kRows = kPairs * kBatch;
};

// Adds up row r (32 lane pairs) and parks the totals in its first two padding floats.
__device__ __forceinline__ void reduce_row(float* red, int r) {
  const ulonglong2* row = reinterpret_cast<const ulonglong2*>(red + r * kRedPad);
  f32x2 s[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const ulonglong2 v = row[c], w = row[c + 8];
    s[c] = f2_add(f2_add(v.x, v.y), f2_add(w.x, w.y));
  }
#pragma unroll
  for (int h = 4; h > 0; h >>= 1)
#pragma unroll
    for (int c = 0; c < h; ++c) s[c] = f2_add(s[c], s[c + h]);
  *reinterpret_cast<f32x2*>(red + r * kRedPad + 64) = s[0];
}

// ------------------------------------------------------------------------------------------
// Backward blend (same pixel layout as the forward).
// ------------------------------------------------------------------------------------------
// kAux: a depth or accumulated-opacity upstream gradient is present. Without one (a colour-only
// loss) the per-pixel depth / opacity gradient state and its arithmetic drop out; the results
// are those of the general kernel with those gradients zero.
template <int TW, int TH, int PPT, bool kAux>
__global__ void __launch_bounds__(TW * TH / PPT) blend_backward_kernel(
    const __grid_constant__ Views views, const Consts c, const uint2* __restrict__ ranges,
    const uint32_t* __restrict__ pair_vals, const Record* __restrict__ rec,
    const float* __restrict__ t_final, const int32_t* __restrict__ last_index,
    const float* __restrict__ d_color, const float* __restrict__ d_depth,
    const float* __restrict__ d_alpha, const uint32_t* __restrict__ tile_order,
    float* __restrict__ g2d) {
  chain_wait();
  constexpr int kThreads = TW * TH / PPT;
  constexpr bool kPacked = PPT % 2 == 0;
  constexpr int P2 = kPacked ? PPT / 2 : 1;
  static_assert(kThreads % 32 == 0, "whole warps only");
  using RL = RedLayout;
  using SL = StageLayout<true, PPT>;
  __shared__ ulonglong2 sp[SL::kRows][kThreads];
  __shared__ uint32_t s_vi[kThreads];
  __shared__ int s_max_last[kThreads / 32];
  __shared__ __align__(16) float s_red[kThreads / 32][RL::kRows * kRedPad];
  const int gtile = (int)tile_order[blockIdx.x];
  const int v = view_of_tile(views, gtile);
  const ViewParams& vp = views.v[v];
  const int local = gtile - vp.tile_base;
  const int ty = local / vp.tiles_x, tx = local - ty * vp.tiles_x;
  const int px = tx * TW + (int)(threadIdx.x % TW);
  const int py0 = ty * TH + (int)(threadIdx.x / TW) * PPT;
  const float fx = (float)px;
  // Anchor row of the tile's row terms, and the thread's first row relative to it (as in the
  // forward, so both blends compute every pixel's exponent to the same bits).
  const float x_m = (float)(tx * TW) + 0.5f * (float)(TW - 1), y_a = (float)(ty * TH + TH / 2);
  const int r0_ = (int)(threadIdx.x / TW) * PPT - TH / 2;
  const uint2 range = ranges[gtile];
  const int lane = threadIdx.x & 31;
  float* const red = s_red[threadIdx.x >> 5];

  // Per pixel: the transmittance T behind the current position, the upstream gradients, and the
  // gradient-weighted value seen behind it per unit of transmittance,
  //   U = dL/dC . C_behind + dL/dD D_behind  (dL/dC . background - dL/dA at the far end),
  // so that with q = dL/dC . c + dL/dD z of a Gaussian and w = alpha T its weight,
  //   alpha dL/dalpha = w (q - U),  U <- U + alpha (q - U)
  // (three operations; the running sum of w q, divided by 1 - alpha at each step, took five).
  float T[PPT], U[PPT], gC0[PPT], gC1[PPT], gC2[PPT], gD[PPT];
  int32_t last[PPT];
  int thread_last = -1;
#pragma unroll
  for (int k = 0; k < PPT; ++k) {
    float Tfin = 1.0f;
    gC0[k] = gC1[k] = gC2[k] = gD[k] = 0.0f;
    float gA = 0.0f;
    last[k] = -1;
    const int py = py0 + k;
    if (px < vp.width && py < vp.height) {
      const long long pix = vp.pixel_offset + (long long)py * vp.width + px;
      Tfin = t_final[pix];
      last[k] = last_index[pix];
      if (d_color) {
        gC0[k] = d_color[3 * pix + 0];
        gC1[k] = d_color[3 * pix + 1];
        gC2[k] = d_color[3 * pix + 2];
      }
      if (kAux && d_depth) gD[k] = d_depth[pix];
      if (kAux && d_alpha) gA = d_alpha[pix];
    }
    T[k] = Tfin;
    U[k] = gC0[k] * c.bg[0] + gC1[k] * c.bg[1] + gC2[k] * c.bg[2] - gA;
    thread_last = max(thread_last, last[k]);
  }
  // The same state as (pixel 2q, pixel 2q + 1) pairs for the packed arithmetic.
  f32x2 T2[P2], U2[P2], GC02[P2], GC12[P2], GC22[P2], GD2[P2], FR[P2];
#pragma unroll
  for (int q = 0; q < P2; ++q) {
    const int k0 = kPacked ? 2 * q : 0, k1 = kPacked ? 2 * q + 1 : 0;
    T2[q] = f2_make(T[k0], T[k1]);
    U2[q] = f2_make(U[k0], U[k1]);
    GC02[q] = f2_make(gC0[k0], gC0[k1]);
    GC12[q] = f2_make(gC1[k0], gC1[k1]);
    GC22[q] = f2_make(gC2[k0], gC2[k1]);
    GD2[q] = f2_make(gD[k0], gD[k1]);
    FR[q] = f2_make((float)(r0_ + k0), (float)(r0_ + k1));
  }
  const f32x2 ONE2 = f2_make(1.0f, 1.0f), ZERO2 = f2_make(0.0f, 0.0f);
  // Only list positions up to the largest last-contributor index of the tile matter.
  int m = thread_last;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) s_max_last[threadIdx.x >> 5] = m;
  // At or below the smallest last-contributor index of the warp every pixel of the warp is
  // live, and the per-pixel test of the list position drops out (warp-uniform).
  int thread_min_last = last[0];
#pragma unroll
  for (int k = 1; k < PPT; ++k) thread_min_last = min(thread_min_last, last[k]);
  const int warp_min_last = __reduce_min_sync(0xffffffffu, thread_min_last);
  __syncthreads();
  int max_last = -1;
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) max_last = max(max_last, s_max_last[w]);
  if (max_last < (int)range.x) return;

  // One Gaussian (list position jj, staged at g) against the thread's pixels; kCheckLast tests
  // each pixel's last-contributor index.
  // kClamp: the Gaussian may reach alpha_max somewhere (clamp, and no gradient through a
  // clamped alpha); without it neither can happen and both tests drop out. The lane's partial
  // sums go to column `lane` of the rows from `rows` on (zeros where it covers nothing).
  auto visit = [&](int jj, int g, float* rows, auto check_last, auto clamp_tag) {
    constexpr bool kCheckLast = decltype(check_last)::value;
    constexpr bool kClamp = decltype(clamp_tag)::value;
    (void)kClamp;  // the one-pixel path always clamps
    // Per-thread sums of dp = dL/dpower over the thread's pixels, weighted by their row offset
    // r from row r_g (0, the anchor row, with one pixel per thread): sdp = sum dp, sr = sum dp r,
    // srr = sum dp r^2. Every pixel of the column has w = (t, s) = (t_a + r l21, s_a + r l22) with
    // t_a, s_a at that row, so the whitened moments follow from
    // these three and t_a once per Gaussian.
    float sdp = 0.0f, sr = 0.0f, srr = 0.0f, ta = 0.0f, gr = 0.0f, gg = 0.0f, gb = 0.0f,
          gz = 0.0f;
    if (!kCheckLast || jj <= thread_last) {
      if constexpr (kPacked) {
        const Staged st = staged<true, PPT>(sp, g);
        const float ta0 = column_t(fx, st.column);
        const f32x2 TA = f2_make(ta0, ta0);
        const f32x2 Z2 = f2_make(f2_lo(st.bz.y), f2_lo(st.bz.y));
        (void)Z2;
        f32x2 aR = ZERO2, aG = ZERO2, aB = ZERO2, aZ = ZERO2, dps[P2];
        (void)aZ;
#pragma unroll
        for (int q = P2 - 1; q >= 0; --q) {
          const int k0 = 2 * q, k1 = 2 * q + 1;
          const f32x2 tt = f2_fma(FR[q], st.l2.x, TA);
          const f32x2 ss = f2_fma(FR[q], st.l2.y, st.sn.x);
          const f32x2 nq = f2_fma(tt, tt, f2_fma(ss, ss, st.sn.y));  // -log2(o G)
          const float oG0 = ex2_neg_approx(f2_lo(nq)), oG1 = ex2_neg_approx(f2_hi(nq));
          const float a0 = kClamp ? fminf(c.alpha_max, oG0) : oG0;
          const float a1 = kClamp ? fminf(c.alpha_max, oG1) : oG1;
          const bool cov0 = (!kCheckLast || jj <= last[k0]) && a0 >= c.alpha_min;
          const bool cov1 = (!kCheckLast || jj <= last[k1]) && a1 >= c.alpha_min;
          // A pixel this Gaussian does not cover gets alpha 0 and 1 / (1 - alpha) = 1 (the
          // hardware reciprocal of 1 is exactly 1 on sm_103a, measured), so its transmittance,
          // U and every accumulator stay bit-identical.
          const f32x2 am = f2_make(cov0 ? a0 : 0.0f, cov1 ? a1 : 0.0f);
          const f32x2 om = f2_sub(ONE2, am);
          const f32x2 rom = f2_make(rcp_approx(f2_lo(om)), rcp_approx(f2_hi(om)));
          T2[q] = f2_mul(T2[q], rom);  // transmittance in front of this Gaussian
          const f32x2 w = f2_mul(am, T2[q]);
          aR = q == P2 - 1 ? f2_mul(GC02[q], w) : f2_fma(GC02[q], w, aR);
          aG = q == P2 - 1 ? f2_mul(GC12[q], w) : f2_fma(GC12[q], w, aG);
          aB = q == P2 - 1 ? f2_mul(GC22[q], w) : f2_fma(GC22[q], w, aB);
          f32x2 qv;
          if constexpr (kAux) {
            aZ = q == P2 - 1 ? f2_mul(GD2[q], w) : f2_fma(GD2[q], w, aZ);
            qv = f2_fma(GC02[q], st.rg.x,
                        f2_fma(GC12[q], st.rg.y, f2_fma(GC22[q], st.bz.x, f2_mul(GD2[q], Z2))));
          } else {
            qv = f2_fma(GC02[q], st.rg.x,
                        f2_fma(GC12[q], st.rg.y, f2_mul(GC22[q], st.bz.x)));
          }
          const f32x2 diff = f2_sub(qv, U2[q]);
          U2[q] = f2_fma(am, diff, U2[q]);
          // dL/dpower = dL/dalpha * alpha (d alpha / d power = o G = alpha), unclamped only
          // (an uncovered pixel has weight 0 here, so its share is 0 already).
          f32x2 dp = f2_mul(w, diff);
          if constexpr (kClamp) {
            const bool m0 = oG0 < c.alpha_max, m1 = oG1 < c.alpha_max;
            dp = f2_make(m0 ? f2_lo(dp) : 0.0f, m1 ? f2_hi(dp) : 0.0f);
          }
          dps[q] = dp;
        }
        gr = f2_lo(aR) + f2_hi(aR);
        gg = f2_lo(aG) + f2_hi(aG);
        gb = f2_lo(aB) + f2_hi(aB);
        if constexpr (kAux) gz = f2_lo(aZ) + f2_hi(aZ);
        // Moments about the middle of the thread's rows, folded by symmetry: pair q's middle lies
        // p_q = 2 q - (P2 - 1) rows from there and its pixels half a row to either side, so with
        // mP = sum dp, mF = sum p_q dp, mQ = sum p_q^2 dp the first and second moments are
        // k1 = sum mF + (hi - lo) mP / 2 and k2 = sum mQ + (hi - lo) mF + sum mP / 4 (seven
        // packed operations for four pairs). Sums from the thread's first row took as many and
        // cancelled up to 225 : 1 in the shift to another row, these 64 : 1.
        f32x2 mP, mF = ZERO2, mQ = ZERO2;
        if constexpr (P2 == 4) {
          const f32x2 A = f2_add(dps[3 % P2], dps[0]), B = f2_add(dps[2 % P2], dps[1 % P2]);
          const f32x2 C = f2_sub(dps[3 % P2], dps[0]), D = f2_sub(dps[2 % P2], dps[1 % P2]);
          mP = f2_add(A, B);
          mF = f2_fma(f2_make(3.0f, 3.0f), C, D);
          mQ = f2_fma(f2_make(9.0f, 9.0f), A, B);
        } else if constexpr (P2 == 2) {
          mP = mQ = f2_add(dps[1 % P2], dps[0]);
          mF = f2_sub(dps[1 % P2], dps[0]);
        } else {
          mP = dps[0];
        }
        sdp = f2_lo(mP) + f2_hi(mP);
        const float k1 = fmaf(0.5f, f2_hi(mP) - f2_lo(mP), f2_lo(mF) + f2_hi(mF));
        const float k2 =
            fmaf(0.25f, sdp, (f2_lo(mQ) + f2_hi(mQ)) + (f2_hi(mF) - f2_lo(mF)));
        // Then over the rows' offsets r - r_g from the row of the footprint's ridge: the lanes'
        // sums and the whitened moments formed from them are then about the size of the result.
        // About the tile's middle row a footprint seven rows away cancelled 50 : 1.
        const float r_g = f2_hi(st.bz.y);
        const float rc = ((float)r0_ + 0.5f * (float)(PPT - 1)) - r_g;
        sr = fmaf(rc, sdp, k1);
        srr = fmaf(rc, k1 + sr, k2);
        ta = fmaf(r_g, f2_lo(st.l2.x), ta0);
      } else {
        const float4 g0 = reinterpret_cast<const float4*>(sp[0])[g];
        const float4 g1 = reinterpret_cast<const float4*>(sp[1])[g];
        const float4 g2 = reinterpret_cast<const float4*>(sp[2])[g];
        ta = __fmaf_rn(g0.z, __fsub_rn(__fsub_rn(fx, g0.x), g0.y), g0.w);
#pragma unroll
        for (int k = 0; k < PPT; ++k) {
          if (kCheckLast && jj > last[k]) continue;
          const float fr = (float)(r0_ + k);
          const float oG = ex2_neg_approx(neg_log2_og(ta, g1.z, g1.x, g1.y, g1.w, fr));
          const float a = fminf(c.alpha_max, oG);
          if (a < c.alpha_min) continue;
          const float rom = rcp_approx(__fsub_rn(1.0f, a));
          T[k] = T[k] * rom;  // transmittance in front of this Gaussian
          const float w = a * T[k];
          gr = fmaf(gC0[k], w, gr);
          gg = fmaf(gC1[k], w, gg);
          gb = fmaf(gC2[k], w, gb);
          float q;
          if constexpr (kAux) {
            gz = fmaf(gD[k], w, gz);
            q = fmaf(gC0[k], g2.x, fmaf(gC1[k], g2.y, fmaf(gC2[k], g2.z, gD[k] * g2.w)));
          } else {
            q = fmaf(gC0[k], g2.x, fmaf(gC1[k], g2.y, gC2[k] * g2.z));
          }
          const float diff = q - U[k];
          U[k] = fmaf(a, diff, U[k]);
          if (oG < c.alpha_max) {
            const float dp = w * diff;
            sdp += dp;
            const float t = dp * fr;
            sr += t;
            srr = fmaf(t, fr, srr);
          }
        }
      }
    }
    const float tsdp = ta * sdp;
    auto put = [&](int p, float x, float y) {
      *reinterpret_cast<f32x2*>(rows + p * kRedPad + 2 * lane) = f2_make(x, y);
    };
    put(0, sdp, sr);
    put(1, srr, tsdp);
    put(2, ta * sr, ta * tsdp);
    put(3, gr, gg);
    put(4, gb, gz);
  };

  // Row sums of the last nb visits (staged at g_first, g_first - 1, ...), then one lane per
  // Gaussian forms its whitened moments (with w = (t_a + r l21, s_a + r l22):
  // sum dp w = (S3 + l21 S1, s_a S0 + l22 S1) and
  // sum dp w w^T = (S5 + l21 (2 S4 + l21 S2), s_a W_t + l22 (S4 + l21 S2),
  // s_a W_s + l22 (s_a S1 + l22 S2)) for the lane values S0..S5) and adds them to its record.
  auto flush = [&](int nb, int g_first) {
    __syncwarp();
    const int nrows = nb * RL::kPairs;
    for (int r = lane; r < nrows; r += 32) reduce_row(red, r);
    __syncwarp();
    if (lane < nb) {
      const int g = g_first - lane;
      const float* tot = red + lane * RL::kPairs * kRedPad + 64;
      float S[2 * RL::kPairs];
#pragma unroll
      for (int k = 0; k < RL::kPairs; ++k) {
        const f32x2 t = *reinterpret_cast<const f32x2*>(tot + k * kRedPad);
        S[2 * k] = f2_lo(t);
        S[2 * k + 1] = f2_hi(t);
      }
      float l21, l22, s_a;
      if constexpr (kPacked) {
        l21 = f2_lo(sp[SL::kShape][g].x);
        l22 = f2_lo(sp[SL::kShape][g].y);
        s_a = fmaf(f2_hi(sp[SL::kRows - 1][g].y), l22, f2_lo(sp[SL::kShape + 1][g].x));
      } else {
        const float4 g1 = reinterpret_cast<const float4*>(sp[1])[g];
        l21 = g1.x;
        l22 = g1.y;
        s_a = g1.z;
      }
      bool any = false;
#pragma unroll
      for (int k = 0; k < 2 * RL::kPairs; ++k) any = any || S[k] != 0.0f;
      if (any) {
        const float wt = fmaf(l21, S[1], S[3]);
        const float ws = fmaf(s_a, S[0], l22 * S[1]);
        const float u = fmaf(l21, S[2], S[4]);
        float* dst = g2d + (size_t)s_vi[g] * kG2Stride;
        // Three vector additions to the 64-byte record in place of nine or ten single ones.
        static_assert(kM0 == 0 && kWt == 1 && kWs == 2 && kWtt == 3 && kWts == 4 && kWss == 5 &&
                          kGR == 6 && kGG == 7 && kGB == 8 && kGZ == 9 && kG2Stride % 4 == 0,
                      "the sums' order in the record");
        atomicAdd(reinterpret_cast<float4*>(dst),
                  make_float4(S[0], wt, ws, fmaf(l21, S[4] + u, S[5])));
        atomicAdd(reinterpret_cast<float4*>(dst) + 1,
                  make_float4(fmaf(s_a, wt, l22 * u),
                              fmaf(s_a, ws, l22 * fmaf(s_a, S[1], l22 * S[2])), S[6], S[7]));
        if constexpr (kAux)
          atomicAdd(reinterpret_cast<float2*>(dst) + 4, make_float2(S[8], S[9]));
        else
          atomicAdd(dst + kGB, S[8]);
      }
    }
    __syncwarp();
  };

  const int first = (int)range.x;
  for (int bend = max_last + 1; bend > first; bend -= kThreads) {
    const int bstart = max(first, bend - kThreads);
    __syncthreads();
    const int j = bstart + (int)threadIdx.x;
    bool may_clamp = false;
    if (j < bend) {
      const uint32_t vi = pair_vals[j];
      s_vi[threadIdx.x] = vi;
      const float4 r1 = rec[vi].conic;
      may_clamp = !(-r1.w > c.unclamped_neg_lo);
      stage_gaussian<TH, true, PPT>(sp, threadIdx.x, rec[vi].mean, r1, rec[vi].colour,
                                    x_m, y_a);
    }
    const unsigned clamp_bits = __ballot_sync(0xffffffffu, may_clamp);
    __syncthreads();
    // Positions above the warp's smallest last index test each pixel; the rest do not. Whether
    // the staged Gaussian can reach alpha_max is warp-uniform. Where the block is one warp it is a
    // bit of the staging vote, so that no load stands between two visits (16 views of 1080p: 4.51
    // -> 4.40 ms); otherwise every thread reads its opacity.
    auto clamps = [&](int g) {
      if constexpr (!kPacked) return true;
      if constexpr (kThreads == 32) return ((clamp_bits >> g) & 1u) != 0u;
      return !(f2_lo(sp[SL::kShape + 1][g].y) > c.unclamped_neg_lo);
    };
    int nb = 0, g_first = bend - 1 - bstart;
    auto next = [&](int g) {
      if (++nb == RL::kBatch) {
        flush(nb, g_first);
        nb = 0;
        g_first = g - 1;
      }
    };
    const int split = max(bstart - 1, min(bend - 1, warp_min_last));
    for (int jj = bend - 1; jj > split; --jj) {
      const int g = jj - bstart;
      float* rows = red + nb * RL::kPairs * kRedPad;
      if (clamps(g))
        visit(jj, g, rows, std::true_type{}, std::true_type{});
      else
        visit(jj, g, rows, std::true_type{}, std::false_type{});
      next(g);
    }
    for (int jj = split; jj >= bstart; --jj) {
      const int g = jj - bstart;
      float* rows = red + nb * RL::kPairs * kRedPad;
      if (clamps(g))
        visit(jj, g, rows, std::false_type{}, std::true_type{});
      else
        visit(jj, g, rows, std::false_type{}, std::false_type{});
      next(g);
    }
    if (nb > 0) flush(nb, g_first);
  }
}

template <int TW, int TH, int PPT>
cudaError_t launch_blends_t(bool forward, const Views& views, const Consts& c,
                            const uint2* ranges, const uint32_t* pair_vals, const Record* rec, float* color, float* depth,
                            float* alpha, float* t_final, int32_t* last_index,
                            const float* d_color, const float* d_depth, const float* d_alpha,
                            float* g2d, const uint32_t* tile_order, Counters* counters,
                            cudaStream_t stream) {
  if (views.total_tiles == 0) return cudaSuccess;
  constexpr int kThreads = TW * TH / PPT;
  cudaError_t e;
  if (forward) {
    e = launch_chained(blend_forward_kernel<TW, TH, PPT>, dim3(views.total_tiles), dim3(kThreads),
                       stream, views, c, ranges, pair_vals, rec, color, depth, alpha,
                       t_final, last_index, tile_order, counters);
  } else {
    const bool aux = d_depth != nullptr || d_alpha != nullptr;
    e = launch_chained(aux ? blend_backward_kernel<TW, TH, PPT, true>
                           : blend_backward_kernel<TW, TH, PPT, false>,
                       dim3(views.total_tiles), dim3(kThreads), stream, views, c, ranges,
                       pair_vals, rec, (const float*)t_final,
                       (const int32_t*)last_index, d_color, d_depth, d_alpha, tile_order, g2d);
  }
  RGS_LAUNCHED();
  return e;
}

}  // namespace

cudaError_t launch_blend(bool forward, const Views& views, const Consts& c, const uint2* ranges,
                         const uint32_t* pair_vals, const Record* rec, float* color, float* depth, float* alpha,
                         float* t_final, int32_t* last_index, const float* d_color,
                         const float* d_depth, const float* d_alpha, float* g2d,
                         const uint32_t* tile_order, Counters* counters, cudaStream_t stream) {
  const int tw = views.tile_w, th = views.tile_h;
  const int ppt = forward ? views.pixels_per_thread : views.bwd_pixels_per_thread;
#define RGS_BLEND(W, H, P)                                                                        \
  if (tw == W && th == H && ppt == P)                                                             \
  return launch_blends_t<W, H, P>(forward, views, c, ranges, pair_vals, rec, color, \
                                  depth, alpha, t_final, last_index, d_color, d_depth, d_alpha,   \
                                  g2d, tile_order, counters, stream)
  RGS_BLEND(16, 16, 1);
  RGS_BLEND(16, 16, 2);
  RGS_BLEND(16, 16, 4);
  RGS_BLEND(16, 16, 8);
  RGS_BLEND(8, 8, 1);
  RGS_BLEND(8, 8, 2);
  RGS_BLEND(32, 8, 1);
  RGS_BLEND(32, 8, 2);
  RGS_BLEND(32, 8, 4);
  RGS_BLEND(32, 8, 8);
#undef RGS_BLEND
  return cudaErrorInvalidValue;
}

}  // namespace rgs

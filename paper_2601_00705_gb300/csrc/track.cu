// track.cu -- the tracking step around the renderer (Section 3.2 and its appendix: Eq.
// app-bright, app-ls, app-trackloss, app-weight; Eq. leftupdate):
//   * pose records: device poses [V][12] -> R, t and the camera centre -R^T t per view, so
//     the projection kernels can read a pose that only the device holds;
//   * gradient weights w_grad(x) = clip(||grad I(x)||_2 / tau_grad, 0, 1) of an observed frame;
//   * the exposure fit (g, b) = argmin sum_x ||I(x) - g I^(x) - b||^2 per view, the weighted L1
//     loss sum_x w_alpha(x) w_grad(x) ||I(x) - (g I^(x) + b)||_1 and its gradient with respect to
//     the rendered colour, which is the upstream gradient of the backward;
//   * one Adam step on the twist xi of every view, applied as T <- exp(xi^) T;
//   * co-visibility of frame pairs for the keyframe test (Eq. iou): intersection and union of
//     the pixels whose accumulated opacity exceeds a threshold.
// All passes are elementwise or reductions over the images (HBM-bound) except the pose update
// (six lanes per view).
#include <math.h>

#include <algorithm>

#include "rgs_internal.cuh"

namespace rgs {
namespace {

constexpr int kTrackThreads = 256;

// ------------------------------------------------------------------------------------------
// Pose records: R (9), t (3), c = -R^T t (3), pad. The centre is accumulated in double and
// rounded once, as the host does for poses given in rgs_camera, so both routes give the same
// records bit for bit.
// ------------------------------------------------------------------------------------------
__global__ void pose_prepare_kernel(const float* __restrict__ world_to_cam, int n_views,
                                    float* __restrict__ records) {
  chain_wait();
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n_views) return;
  const float* w = world_to_cam + 12 * v;
  float R[9], t[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
#pragma unroll
    for (int b = 0; b < 3; ++b) R[3 * a + b] = w[4 * a + b];
    t[a] = w[4 * a + 3];
  }
  float* r = records + 16 * v;
#pragma unroll
  for (int k = 0; k < 9; ++k) r[k] = R[k];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    r[9 + a] = t[a];
    double s = 0.0;
#pragma unroll
    for (int b = 0; b < 3; ++b) s -= (double)R[3 * b + a] * (double)t[b];
    r[12 + a] = (float)s;
  }
  r[15] = 0.0f;
}

// Pixel k of view v's pixels, walked by the blocks of grid row v.
__device__ __forceinline__ void view_pixels(const Views& views, int v, long long& first,
                                            int& count, int& width, int& height) {
  const ViewParams& vp = views.v[v];
  first = vp.pixel_offset;
  width = vp.width;
  height = vp.height;
  count = vp.width * vp.height;
}

// ------------------------------------------------------------------------------------------
// Gradient weights (Eq. app-weight): per channel, central differences inside the image and
// one-sided differences on its border (zero along an axis of extent 1); the norm is taken over
// both axes and the three channels.
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kTrackThreads) grad_weight_kernel(
    const __grid_constant__ Views views, const float* __restrict__ obs, float inv_tau,
    float* __restrict__ w_out) {
  chain_wait();
  const int v = blockIdx.y;
  long long first;
  int count, W, H;
  view_pixels(views, v, first, count, W, H);
  for (int k = blockIdx.x * kTrackThreads + threadIdx.x; k < count;
       k += gridDim.x * kTrackThreads) {
    const int y = k / W, x = k - y * W;
    const int xl = x > 0 ? x - 1 : x, xr = x < W - 1 ? x + 1 : x;
    const int yu = y > 0 ? y - 1 : y, yd = y < H - 1 ? y + 1 : y;
    const float sx = (xr - xl) == 2 ? 0.5f : 1.0f, sy = (yd - yu) == 2 ? 0.5f : 1.0f;
    const float* row = obs + 3 * (first + (long long)y * W);
    const float* up = obs + 3 * (first + (long long)yu * W);
    const float* dn = obs + 3 * (first + (long long)yd * W);
    float s = 0.0f;
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
      const float gx = (xr == xl) ? 0.0f : (row[3 * xr + ch] - row[3 * xl + ch]) * sx;
      const float gy = (yd == yu) ? 0.0f : (dn[3 * x + ch] - up[3 * x + ch]) * sy;
      s = fmaf(gx, gx, fmaf(gy, gy, s));
    }
    w_out[first + k] = fminf(fmaxf(sqrtf(s) * inv_tau, 0.0f), 1.0f);
  }
}

// ------------------------------------------------------------------------------------------
// The two loss passes walk the images four consecutive pixels a thread: kLossThreads threads take
// kTrackThreads pixels of a row of blocks at a time, so that a colour quadruple is three 16-byte
// words (where the quadruple starts on 16 bytes). Each of the four keeps its own FP32 partial sums,
// and a group of eight threads adds its 32 as a warp with one pixel per thread would (offsets 16,
// 8, 4 across the threads, 2 and 1 inside), so every sum is the same float as pixel by pixel; FP64
// from there on.
// ------------------------------------------------------------------------------------------
constexpr int kLossThreads = kTrackThreads / 4;

// Calls one(p, e) for every pixel p (index e of its quadruple) or four(p) for whole quadruples
// that start on 16 bytes (vec: the arrays do).
template <typename One, typename Four>
__device__ __forceinline__ void for_quads(const Views& views, int v, int vec, One&& one,
                                          Four&& four) {
  long long first;
  int count, W, H;
  view_pixels(views, v, first, count, W, H);
  const bool wide = vec && (first & 3) == 0;
  for (int k = 4 * (blockIdx.x * kLossThreads + threadIdx.x); k < count;
       k += gridDim.x * kTrackThreads) {
    if (wide && k + 3 < count) {
      four(first + k);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (k + e < count) one(first + k + e, e);
    }
  }
}

__device__ __forceinline__ void load12(const float* __restrict__ p, float (&x)[12]) {
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const float4 w = reinterpret_cast<const float4*>(p)[q];
    x[4 * q] = w.x;
    x[4 * q + 1] = w.y;
    x[4 * q + 2] = w.z;
    x[4 * q + 3] = w.w;
  }
}

// Block-wide sums of NV values of each of a thread's four pixels, into (double) accumulators with
// atomics.
template <int NV>
__device__ __forceinline__ void block_sum_to(const float (&x)[4][NV], double* __restrict__ acc) {
  constexpr int kGroups = kLossThreads / 8;
  __shared__ double s_part[kGroups][NV];
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    float q[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      q[e] = x[e][j];
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) q[e] += __shfl_xor_sync(0xffffffffu, q[e], o);
    }
    const float sum = (q[0] + q[2]) + (q[1] + q[3]);
    if ((threadIdx.x & 7) == 0) s_part[threadIdx.x >> 3][j] = (double)sum;
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    double t = 0.0;
#pragma unroll
    for (int g = 0; g < kGroups; ++g) t += s_part[g][threadIdx.x];
    atomicAdd(acc + threadIdx.x, t);
  }
}

// ------------------------------------------------------------------------------------------
// Exposure fit, pass 1 (Eq. app-ls): per view, sum r, sum r^2, sum o, sum r o over the three
// channels of every pixel (r rendered, o observed).
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kLossThreads) track_sums_kernel(
    const __grid_constant__ Views views, const float* __restrict__ color,
    const float* __restrict__ obs, int vec, double* __restrict__ sums,
    double* __restrict__ loss) {
  chain_wait();
  const int v = blockIdx.y;
  if (blockIdx.x == 0 && threadIdx.x == 0) loss[v] = 0.0;  // for the next pass
  float x[4][4] = {};
  auto add = [](float (&s)[4], float r, float o) {
    s[0] += r;
    s[1] = fmaf(r, r, s[1]);
    s[2] += o;
    s[3] = fmaf(r, o, s[3]);
  };
  for_quads(
      views, v, vec,
      [&](long long p, int e) {
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) add(x[e], color[3 * p + ch], obs[3 * p + ch]);
      },
      [&](long long p) {
        float r[12], o[12];
        load12(color + 3 * p, r);
        load12(obs + 3 * p, o);
#pragma unroll
        for (int e = 0; e < 12; ++e) add(x[e / 3], r[e], o[e]);
      });
  block_sum_to<4>(x, sums + 4 * v);
}

// (g, b) of view v from its sums; without a unique fit (a constant render) g = 1 and b matches
// the means.
__device__ __forceinline__ void exposure_of(const double* s, double n, bool fit, double& g,
                                            double& b) {
  if (!fit) {
    g = 1.0;
    b = 0.0;
    return;
  }
  const double sr = s[0], srr = s[1], so = s[2], sro = s[3];
  const double den = n * srr - sr * sr;
  if (n > 0.0 && den > 1e-12 * n * n) {
    g = (n * sro - sr * so) / den;
    b = (so - g * sr) / n;
  } else {
    g = 1.0;
    b = n > 0.0 ? (so - sr) / n : 0.0;
  }
}

// ------------------------------------------------------------------------------------------
// Pass 2 (Eq. app-bright, app-trackloss, app-weight): with r' = g r + b,
//   loss_v = sum_x w(x) sum_ch |o - r'|,  w = clip(alpha / tau_alpha, 0, 1) w_grad,
//   dL/dr_ch = -w g sign(o - r'),
// with (g, b) and w held fixed (they are re-estimated from every render, and no gradient flows
// into them). Writes the upstream colour gradient, the loss per view and (g, b) per view.
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kLossThreads) track_loss_kernel(
    const __grid_constant__ Views views, const float* __restrict__ color,
    const float* __restrict__ alpha, const float* __restrict__ obs,
    const float* __restrict__ w_grad, const double* __restrict__ sums, float inv_tau_alpha,
    int fit_exposure, int vec, float* __restrict__ d_color, double* __restrict__ loss,
    float* __restrict__ gain_bias) {
  chain_wait();
  const int v = blockIdx.y;
  double gd, bd;
  // One thread fits the exposure: a double-precision instruction costs a warp 64 cycles.
  __shared__ float s_fit[2];
  if (threadIdx.x == 0) {
    exposure_of(sums + 4 * v, 3.0 * (double)views.v[v].width * (double)views.v[v].height,
                fit_exposure != 0, gd, bd);
    s_fit[0] = (float)gd;
    s_fit[1] = (float)bd;
    if (blockIdx.x == 0) {
      gain_bias[2 * v] = (float)gd;
      gain_bias[2 * v + 1] = (float)bd;
    }
  }
  __syncthreads();
  const float g = s_fit[0], b = s_fit[1];
  float part[4][1] = {};
  // Pixel e of the quadruple: gradient and share of the loss, from its residuals (r rendered, o
  // observed).
  auto pixel = [&](int e, float a, float wg, const float* r, const float* o, float* d) {
    const float w = fminf(fmaxf(a * inv_tau_alpha, 0.0f), 1.0f) * wg;
    float l1 = 0.0f;
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
      const float res = o[ch] - fmaf(g, r[ch], b);
      l1 += fabsf(res);
      const float sg = res > 0.0f ? 1.0f : (res < 0.0f ? -1.0f : 0.0f);
      d[ch] = -w * g * sg;
    }
    part[e][0] = fmaf(w, l1, part[e][0]);
  };
  for_quads(
      views, v, vec,
      [&](long long p, int e) {
        float r[3], o[3], d[3];
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
          r[ch] = color[3 * p + ch];
          o[ch] = obs[3 * p + ch];
        }
        pixel(e, alpha[p], w_grad ? w_grad[p] : 1.0f, r, o, d);
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) d_color[3 * p + ch] = d[ch];
      },
      [&](long long p) {
        float r[12], o[12], d[12];
        load12(color + 3 * p, r);
        load12(obs + 3 * p, o);
        const float4 a = *reinterpret_cast<const float4*>(alpha + p);
        const float4 wg = w_grad ? *reinterpret_cast<const float4*>(w_grad + p)
                                 : make_float4(1.0f, 1.0f, 1.0f, 1.0f);
        pixel(0, a.x, wg.x, r, o, d);
        pixel(1, a.y, wg.y, r + 3, o + 3, d + 3);
        pixel(2, a.z, wg.z, r + 6, o + 6, d + 6);
        pixel(3, a.w, wg.w, r + 9, o + 9, d + 9);
        float4* out = reinterpret_cast<float4*>(d_color + 3 * p);
        out[0] = make_float4(d[0], d[1], d[2], d[3]);
        out[1] = make_float4(d[4], d[5], d[6], d[7]);
        out[2] = make_float4(d[8], d[9], d[10], d[11]);
      });
  block_sum_to<1>(part, loss + v);
}

// ------------------------------------------------------------------------------------------
// Pose update: one Adam step on the twist xi = (rho, omega) of every view from dL/dxi at
// xi = 0, then T <- exp(xi^) T (Eq. leftupdate) with the closed-form SE(3) exponential:
//   R_d = I + A W + B W^2,  V = I + B W + C W^2,  t_d = V rho,  W = [omega]_x,
//   A = sin(th) / th, B = (1 - cos(th)) / th^2, C = (th - sin(th)) / th^3, th = |omega|
// (Taylor series for small th); R <- R_d R, t <- R_d t + t_d. The learning rate of step k
// (k = 0, 1, ...) is lr * (1 + cos(pi min(k, K) / K)) / 2 with K = iterations, or lr when
// K = 0. In FP64; the pose is stored back in FP32.
// ------------------------------------------------------------------------------------------
// Six lanes per view (five views per warp), lane j with component j: a double-precision
// instruction costs a warp 64 cycles whatever its lanes do, so the views' components go through
// each one together and what a view shares is computed by its six lanes alike (27 us with a thread
// per view and the pow, sin and cos of the general case, now 10).
constexpr int kAdamViews = 5;  // views per warp

// x^n by squaring. n follows from the caller's step counter in device memory, so it may be anything:
// the loop runs over an unsigned exponent, at most 32 times.
__device__ __forceinline__ double power(double x, int64_t n) {
  double r = 1.0;
  for (uint32_t e = (uint32_t)(n < 0 ? -n : n); e; e >>= 1) {
    if (e & 1) r *= x;
    x *= x;
  }
  return n < 0 ? 1.0 / r : r;
}

__global__ void pose_adam_kernel(int n_views, float lr, float beta1, float beta2, float eps,
                                 int iterations, const float* __restrict__ d_pose,
                                 float* __restrict__ adam_state, int32_t* __restrict__ step,
                                 float* __restrict__ world_to_cam) {
  chain_wait();
  const int lane = threadIdx.x & 31;
  const int j = lane % 6, first = lane - j;
  const int v = (threadIdx.x >> 5) * kAdamViews + lane / 6;
  const bool on = lane < 6 * kAdamViews && v < n_views;
  const int k = *step;
  __syncthreads();  // every thread has read the step count before it advances
  double lr_k = lr;
  if (iterations > 0)
    lr_k = 0.5 * (double)lr * (1.0 + cospi((double)min(k, iterations) / (double)iterations));
  // Even lanes hold 1 - beta1^(k + 1), odd ones 1 - beta2^(k + 1).
  const double bias = 1.0 - power((lane & 1) ? (double)beta2 : (double)beta1, (int64_t)k + 1);
  const double c1 = __shfl_sync(0xffffffffu, bias, 0), c2 = __shfl_sync(0xffffffffu, bias, 1);
  double xi = 0.0;
  if (on) {
    float* m = adam_state + 12 * v;
    const double gj = d_pose[6 * v + j];
    const double mj = (double)beta1 * m[j] + (1.0 - (double)beta1) * gj;
    const double vj = (double)beta2 * m[6 + j] + (1.0 - (double)beta2) * gj * gj;
    m[j] = (float)mj;
    m[6 + j] = (float)vj;
    xi = -lr_k * (mj / c1) / (sqrt(vj / c2) + (double)eps);
  }
  double rho[3], w[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    rho[a] = __shfl_sync(0xffffffffu, xi, first + a);
    w[a] = __shfl_sync(0xffffffffu, xi, (first + 3 + a) & 31);
  }
  const double th2 = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
  // A = sin(th) / th, B = (1 - cos(th)) / th^2, C = (th - sin(th)) / th^3: their Taylor series up
  // to th = 1/2 (eight terms leave 1e-17; no cancellation for small th), else sin and cos.
  double A, B, C;
  if (th2 <= 0.25) {
    A = B = C = 0.0;
#pragma unroll
    for (int q = 7; q >= 0; --q) {  // coefficients (-1)^q / (2q + 1)!, (2q + 2)!, (2q + 3)!
      constexpr double kFact[18] = {1., 1., 2., 6., 24., 120., 720., 5040., 40320., 362880.,
                                    3628800., 39916800., 479001600., 6227020800., 87178291200.,
                                    1307674368000., 20922789888000., 355687428096000.};
      const double sg = (q & 1) ? -1.0 : 1.0;
      A = fma(A, th2, sg / kFact[2 * q + 1]);
      B = fma(B, th2, sg / kFact[2 * q + 2]);
      C = fma(C, th2, sg / kFact[2 * q + 3]);
    }
  } else {
    const double th = sqrt(th2);
    double sn, cs;
    sincos(th, &sn, &cs);
    A = sn / th;
    B = (1.0 - cs) / th2;
    C = (th - sn) / (th2 * th);
  }
  // Lane j answers for two entries of row a = j / 2 of the new pose: columns 0 and 1, or column 2
  // and the translation. Row a of W = [omega]_x and of W^2 = omega omega^T - th^2 I.
  const int a = j >> 1;
  const double wa = a == 0 ? w[0] : a == 1 ? w[1] : w[2];
  const double W[3] = {a == 0 ? 0.0 : a == 1 ? w[2] : -w[1], a == 0 ? -w[2] : a == 1 ? 0.0 : w[0],
                       a == 0 ? w[1] : a == 1 ? -w[0] : 0.0};
  double Rd[3], Vm[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    const double id = a == b ? 1.0 : 0.0;
    const double W2 = wa * w[b] - id * th2;
    Rd[b] = id + A * W[b] + B * W2;
    Vm[b] = id + B * W[b] + C * W2;
  }
  float* T = world_to_cam + 12 * (on ? v : 0);
  double n0 = 0.0, n1 = 0.0;
  const int col = (j & 1) ? 2 : 0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    n0 += Rd[c] * (double)T[4 * c + col];
    n1 += Rd[c] * (double)T[4 * c + col + 1];
    if (j & 1) n1 += Vm[c] * rho[c];
  }
  __syncthreads();  // every lane of a view has read the old pose
  if (on) {
    T[4 * a + col] = (float)n0;
    T[4 * a + col + 1] = (float)n1;
  }
  if (threadIdx.x == 0) *step = (int32_t)((uint32_t)k + 1u);
}

// ------------------------------------------------------------------------------------------
// Co-visibility (Eq. iou, with the per-pixel visibility masks of the keyframe scheduling): for
// pair j, V_a = {p : alpha_a(p) > tau}, V_b likewise, counts |V_a n V_b| and |V_a u V_b| over
// the n pixels of the pair's two images; IoU = intersection / union (0 for an empty union).
// Grid rows are pairs; each block reduces its share with ballots and one atomic per count.
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kTrackThreads) covis_count_kernel(
    const float* __restrict__ alpha_a, const float* __restrict__ alpha_b, int64_t n, float tau,
    unsigned long long* __restrict__ counts) {
  chain_wait();
  const int j = blockIdx.y;
  const float* a = alpha_a + (size_t)j * n;
  const float* b = alpha_b + (size_t)j * n;
  unsigned long long inter = 0, uni = 0;
  auto add = [&](float x, float y) {
    const bool va = x > tau, vb = y > tau;
    inter += (va && vb) ? 1u : 0u;
    uni += (va || vb) ? 1u : 0u;
  };
  // Four pixels per load where both images start on 16 bytes.
  const bool vec = ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15) == 0;
  const int64_t t = (int64_t)blockIdx.x * kTrackThreads + threadIdx.x,
                step = (int64_t)gridDim.x * kTrackThreads, groups = vec ? n >> 2 : 0;
  for (int64_t p = t; p < groups; p += step) {
    const float4 x = reinterpret_cast<const float4*>(a)[p];
    const float4 y = reinterpret_cast<const float4*>(b)[p];
    add(x.x, y.x);
    add(x.y, y.y);
    add(x.z, y.z);
    add(x.w, y.w);
  }
  for (int64_t p = 4 * groups + t; p < n; p += step) add(a[p], b[p]);
  __shared__ unsigned long long s_i[kTrackThreads / 32], s_u[kTrackThreads / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    inter += __shfl_xor_sync(0xffffffffu, inter, o);
    uni += __shfl_xor_sync(0xffffffffu, uni, o);
  }
  if ((threadIdx.x & 31) == 0) {
    s_i[threadIdx.x >> 5] = inter;
    s_u[threadIdx.x >> 5] = uni;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long ti = 0, tu = 0;
    for (int w = 0; w < kTrackThreads / 32; ++w) {
      ti += s_i[w];
      tu += s_u[w];
    }
    atomicAdd(counts + 2 * j, ti);
    atomicAdd(counts + 2 * j + 1, tu);
  }
}

__global__ void covis_iou_kernel(int n_pairs, const unsigned long long* __restrict__ counts,
                                 float* __restrict__ iou) {
  chain_wait();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < n_pairs)
    iou[j] = counts[2 * j + 1] ? (float)((double)counts[2 * j] / (double)counts[2 * j + 1]) : 0.0f;
}

// Grid rows per view, columns enough to cover the largest view (at most 2 waves of blocks). The
// loss passes' partial sums follow this grid.
dim3 view_grid(const Views& views) {
  int max_px = 1;
  for (int v = 0; v < views.n_views; ++v)
    max_px = max(max_px, views.v[v].width * views.v[v].height);
  const int want = (max_px + kTrackThreads * 4 - 1) / (kTrackThreads * 4);
  const int cap = max(1, 2 * 152 * 4 / views.n_views);
  return dim3((unsigned)min(want, cap), (unsigned)views.n_views);
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace

cudaError_t launch_pose_prepare(const float* world_to_cam, int n_views, float* records,
                                cudaStream_t stream) {
  const cudaError_t e = launch_chained(pose_prepare_kernel, dim3(1), dim3(kMaxViews), stream,
                                       world_to_cam, n_views, records);
  RGS_LAUNCHED();
  return e;
}

cudaError_t launch_grad_weight(const Views& views, const float* obs, float tau_grad, float* w_out,
                               cudaStream_t stream) {
  const cudaError_t e = launch_chained(grad_weight_kernel, view_grid(views), dim3(kTrackThreads),
                                       stream, views, obs, 1.0f / tau_grad, w_out);
  RGS_LAUNCHED();
  return e;
}

cudaError_t launch_track_loss(const Views& views, const float* color, const float* alpha,
                              const float* obs, const float* w_grad, float tau_alpha,
                              bool fit_exposure, double* sums, float* d_color, double* loss,
                              float* gain_bias, cudaStream_t stream) {
  const int V = views.n_views;
  const dim3 grid = view_grid(views);
  const int vec = aligned16(color) && aligned16(alpha) && aligned16(obs) && aligned16(d_color) &&
                  (!w_grad || aligned16(w_grad));
  cudaError_t e;
  if (fit_exposure) {
    e = cudaMemsetAsync(sums, 0, sizeof(double) * 4 * V, stream);
    if (e != cudaSuccess) return e;
    e = launch_chained(track_sums_kernel, grid, dim3(kLossThreads), stream, views, color, obs,
                       vec, sums, loss);
    RGS_LAUNCHED();
  } else {
    e = cudaMemsetAsync(loss, 0, sizeof(double) * V, stream);
  }
  if (e != cudaSuccess) return e;
  e = launch_chained(track_loss_kernel, grid, dim3(kLossThreads), stream, views, color, alpha,
                     obs, w_grad, (const double*)sums, 1.0f / tau_alpha, fit_exposure ? 1 : 0,
                     vec, d_color, loss, gain_bias);
  RGS_LAUNCHED();
  return e;
}

cudaError_t launch_covisibility(const float* alpha_a, const float* alpha_b, int64_t n,
                                int n_pairs, float tau, unsigned long long* counts, float* iou,
                                cudaStream_t stream) {
  cudaError_t e = cudaMemsetAsync(counts, 0, sizeof(unsigned long long) * 2 * n_pairs, stream);
  if (e != cudaSuccess || n_pairs == 0) return e;
  if (n > 0) {
    const int64_t want = (n + kTrackThreads * 4 - 1) / (kTrackThreads * 4);
    const unsigned gx = (unsigned)std::max<int64_t>(1, std::min<int64_t>(want, 4 * 152 / n_pairs + 1));
    e = launch_chained(covis_count_kernel, dim3(gx, (unsigned)n_pairs), dim3(kTrackThreads),
                       stream, alpha_a, alpha_b, n, tau, counts);
    RGS_LAUNCHED();
    if (e != cudaSuccess) return e;
  }
  e = launch_chained(covis_iou_kernel, dim3((unsigned)((n_pairs + 255) / 256)), dim3(256), stream,
                     n_pairs, (const unsigned long long*)counts, iou);
  RGS_LAUNCHED();
  return e;
}

cudaError_t launch_pose_adam(int n_views, float lr, float beta1, float beta2, float eps,
                             int iterations, const float* d_pose, float* adam_state,
                             int32_t* step, float* world_to_cam, cudaStream_t stream) {
  const cudaError_t e = launch_chained(pose_adam_kernel, dim3(1),
                                       dim3(32 * ((n_views + kAdamViews - 1) / kAdamViews)),
                                       stream, n_views, lr, beta1, beta2, eps, iterations, d_pose,
                                       adam_state, step, world_to_cam);
  RGS_LAUNCHED();
  return e;
}

}  // namespace rgs

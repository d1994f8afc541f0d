// map.cu -- maintenance of the Gaussian set between mapping steps (appendix "Gaussian
// Initialization and Joint Mapping": Eq. app-ema and the pruning bounds on the observation
// count, visibility score, covariance trace and opacity). Elementwise over the Gaussians.
#include <math.h>

#include <algorithm>

#include "rgs_internal.cuh"

namespace rgs {
namespace {

constexpr int kMapThreads = 256;

// Eq. app-ema: mu_bar <- (1 - eta) mu_bar + eta mu, four floats at a time where both arrays are
// 16-byte aligned (vec).
__global__ void __launch_bounds__(kMapThreads) map_ema_kernel(int64_t n3,
                                                              const float* __restrict__ means,
                                                              float* __restrict__ ema, float eta,
                                                              int vec) {
  chain_wait();
  auto step_to = [&](float e, float m) { return fmaf(eta, m - e, e); };
  const int64_t t = (int64_t)blockIdx.x * kMapThreads + threadIdx.x,
                step = (int64_t)gridDim.x * kMapThreads, groups = vec ? n3 >> 2 : 0;
  for (int64_t k = t; k < groups; k += step) {
    const float4 m = reinterpret_cast<const float4*>(means)[k];
    float4 e = reinterpret_cast<float4*>(ema)[k];
    e = make_float4(step_to(e.x, m.x), step_to(e.y, m.y), step_to(e.z, m.z), step_to(e.w, m.w));
    reinterpret_cast<float4*>(ema)[k] = e;
  }
  for (int64_t k = 4 * groups + t; k < n3; k += step) ema[k] = step_to(ema[k], means[k]);
}

// Kept iff alpha >= min_opacity, tr(Sigma) <= max_trace and not (observed at least
// min_observations times with a visibility score below min_visibility). Four Gaussians per thread
// and step where every array allows wide accesses (vec); the kept ones are counted per block and
// added once (an atomic per warp on the one counter took most of 25 us per million Gaussians).
__global__ void __launch_bounds__(kMapThreads) prune_mask_kernel(
    int n, const float* __restrict__ log_scales, const float* __restrict__ logits,
    const uint32_t* __restrict__ obs_count, const float* __restrict__ vis_score,
    float min_opacity, float max_trace, uint32_t min_observations, float min_visibility, int vec,
    uint8_t* __restrict__ keep, uint32_t* __restrict__ n_keep) {
  chain_wait();
  uint32_t kept = 0;
  auto decide = [&](float l0, float l1, float l2, float logit, uint32_t obs, float vis) {
    const float alpha = 1.0f / (1.0f + expf(-logit));
    const float tr = expf(2.0f * l0) + expf(2.0f * l1) + expf(2.0f * l2);
    const bool weak = obs >= min_observations && vis < min_visibility;
    const bool k = alpha >= min_opacity && tr <= max_trace && !weak;
    kept += k ? 1u : 0u;
    return (uint8_t)(k ? 1 : 0);
  };
  const int64_t t = (int64_t)blockIdx.x * kMapThreads + threadIdx.x,
                step = (int64_t)gridDim.x * kMapThreads, groups = vec ? n >> 2 : 0;
  for (int64_t k = t; k < groups; k += step) {
    const float4* ls = reinterpret_cast<const float4*>(log_scales) + 3 * k;
    const float4 a = ls[0], b = ls[1], c = ls[2];
    const float4 lg = reinterpret_cast<const float4*>(logits)[k];
    const uint4 ob = reinterpret_cast<const uint4*>(obs_count)[k];
    const float4 vs = reinterpret_cast<const float4*>(vis_score)[k];
    reinterpret_cast<uchar4*>(keep)[k] =
        make_uchar4(decide(a.x, a.y, a.z, lg.x, ob.x, vs.x), decide(a.w, b.x, b.y, lg.y, ob.y, vs.y),
                    decide(b.z, b.w, c.x, lg.z, ob.z, vs.z), decide(c.y, c.z, c.w, lg.w, ob.w, vs.w));
  }
  for (int64_t i = 4 * groups + t; i < n; i += step)
    keep[i] = decide(log_scales[3 * i], log_scales[3 * i + 1], log_scales[3 * i + 2], logits[i],
                     obs_count[i], vis_score[i]);
  __shared__ uint32_t s_kept;
  if (threadIdx.x == 0) s_kept = 0;
  __syncthreads();
  kept = __reduce_add_sync(0xffffffffu, kept);
  if ((threadIdx.x & 31) == 0 && kept) atomicAdd(&s_kept, kept);
  __syncthreads();
  if (threadIdx.x == 0 && s_kept) atomicAdd(n_keep, s_kept);
}

bool aligned(const void* p, uintptr_t bytes) {
  return (reinterpret_cast<uintptr_t>(p) & (bytes - 1)) == 0;
}

}  // namespace

cudaError_t launch_map_ema(int64_t n, const float* means, float* ema, float eta,
                           cudaStream_t stream) {
  const int64_t n3 = 3 * n;
  const int vec = aligned(means, 16) && aligned(ema, 16);
  const int64_t items = vec ? (n3 + 3) / 4 : n3;
  const unsigned blocks =
      (unsigned)std::min<int64_t>((items + kMapThreads - 1) / kMapThreads, 8 * 152);
  const cudaError_t e = launch_chained(map_ema_kernel, dim3(blocks), dim3(kMapThreads), stream,
                                       n3, means, ema, eta, vec);
  RGS_LAUNCHED();
  return e;
}

cudaError_t launch_prune_mask(int64_t n, const float* log_scales, const float* logits,
                              const uint32_t* obs_count, const float* vis_score, float min_opacity,
                              float max_trace, uint32_t min_observations, float min_visibility,
                              uint8_t* keep, uint32_t* n_keep, cudaStream_t stream) {
  cudaError_t e = cudaMemsetAsync(n_keep, 0, sizeof(uint32_t), stream);
  if (e != cudaSuccess || n == 0) return e;
  const int vec = aligned(log_scales, 16) && aligned(logits, 16) && aligned(obs_count, 16) &&
                  aligned(vis_score, 16) && aligned(keep, 4);
  const int64_t items = vec ? (n + 3) / 4 : n;
  const unsigned blocks =
      (unsigned)std::min<int64_t>((items + kMapThreads - 1) / kMapThreads, 8 * 152);
  e = launch_chained(prune_mask_kernel, dim3(blocks), dim3(kMapThreads), stream, (int)n,
                     log_scales, logits, obs_count, vis_score, min_opacity, max_trace,
                     min_observations, min_visibility, vec, keep, n_keep);
  RGS_LAUNCHED();
  return e;
}

}  // namespace rgs

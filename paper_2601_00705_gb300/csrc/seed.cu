// seed.cu -- the single-step dense initialisation (Section 3.3 "Multi-view Triangulation" and
// "Gaussian Parameter Initialization"; appendix "Gaussian Initialization and Joint Mapping",
// Eq. app-sigma-init, Eq. app-alpha-init), in FP64 where the paper asks for double precision:
//   triangulate_kernel  one thread per retained reference pixel: for each neighbour the 4x4
//                       linear system of the two-view DLT, its smallest right singular vector in
//                       FP64, reprojection error and baseline angle; the best accepted hypothesis;
//   voxel thinning      optional: one seed per cube (highest confidence, then lowest index);
//   cell keys + sort    the accepted points grouped by cubic cells of the plane-fit radius;
//   moments_kernel      per accepted point: count and moments of the points within the radius (27
//                       cells, binary search in the sorted keys), a warp per point;
//   seed_kernel         per seed: plane fit by a 3x3 Jacobi eigen-solve, tangent frame, scales
//                       from the reference projection Jacobian, colour as the median of
//                       exposure-corrected bilinear samples, opacity from the confidence.
#include <math.h>

#include <algorithm>

#include "scan_device.cuh"

namespace rgs {

namespace {

constexpr int kSeedThreads = 128;
constexpr int kMaxNb = 8;      // neighbours per reference pixel
constexpr int kJacobiSweeps = 16;

// Pixel of X in view v and its camera-space point.
__device__ __forceinline__ void project_pt(const SeedCams& cams, int v, const double X[3],
                                           double& u, double& w, double xc[3]) {
  const double* R = cams.R[v];
  for (int a = 0; a < 3; ++a)
    xc[a] = R[3 * a] * X[0] + R[3 * a + 1] * X[1] + R[3 * a + 2] * X[2] + cams.t[v][a];
  const double iz = 1.0 / xc[2];
  u = cams.fx[v] * xc[0] * iz + cams.cx[v];
  w = cams.fy[v] * xc[1] * iz + cams.cy[v];
}

// Smallest right singular vector of the 4x4 matrix A (row-major), up to scale:
//   * A P = Q R by Householder reflections with column pivoting;
//   * one-sided Jacobi (Hestenes) on the columns of R^T: its left singular vectors are A P's right
//     ones, so nothing but the four columns is rotated, and the pivoted triangle needs about two
//     sweeps where A itself takes five (preconditioned Jacobi, Drmac and Veselic, SIAM J. Matrix
//     Anal. Appl. 2008);
//   * the vector orthogonal to the three larger columns, so that a vanishing singular value (exact
//     matches) does no harm;
//   * one correction from the residual A w, w -= sum_j v_j (v_j . A^T A w) / (s_j^2 - s_min^2),
//     which takes out what the factorisation rounded off: against 80-bit arithmetic the points'
//     error is half of plain one-sided Jacobi's on A (median 0.9e-15 against 1.5e-15 relative,
//     99.9th percentile 5.6e-14 against 1.3e-13; 0.3 px noise, 5 % outliers).
// About 1200 FP64 operations a system instead of 2700: the FP64 pipe bounds the kernel.
__device__ __forceinline__ void swap_if(bool c, double& a, double& b) {
  const double t = c ? b : a;
  b = c ? a : b;
  a = t;
}

__device__ void smallest_right_singular_vector(const double (&A)[16], double (&out)[4]) {
  // a[c] is column c of A P; perm[c] its column in A.
  double a[4][4];
  int perm[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    perm[c] = c;
#pragma unroll
    for (int r = 0; r < 4; ++r) a[c][r] = A[4 * r + c];
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    // The longest remaining column comes first.
    double best = 0.0;
    int at = k;
#pragma unroll
    for (int c = k; c < 4; ++c) {
      double n = 0.0;
#pragma unroll
      for (int r = k; r < 4; ++r) n = fma(a[c][r], a[c][r], n);
      if (c == k || n > best) {
        best = n;
        at = c;
      }
    }
#pragma unroll
    for (int c = k + 1; c < 4; ++c) {
      const bool sw = at == c;
#pragma unroll
      for (int r = 0; r < 4; ++r) swap_if(sw, a[k][r], a[c][r]);
      const int t = sw ? perm[c] : perm[k];
      perm[c] = sw ? perm[k] : perm[c];
      perm[k] = t;
    }
    if (best == 0.0) continue;
    const double norm = sqrt(best);
    const double diag = a[k][k] >= 0.0 ? -norm : norm;
    const double v0 = a[k][k] - diag;
    const double beta = 1.0 / (diag * v0);
#pragma unroll
    for (int c = k + 1; c < 4; ++c) {
      double d = v0 * a[c][k];
#pragma unroll
      for (int r = k + 1; r < 4; ++r) d = fma(a[k][r], a[c][r], d);
      d *= beta;
      a[c][k] = fma(d, v0, a[c][k]);
#pragma unroll
      for (int r = k + 1; r < 4; ++r) a[c][r] = fma(d, a[k][r], a[c][r]);
    }
    a[k][k] = diag;
  }
  // Columns of R^T: x[j] = row j of R.
  double x[4][4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int c = 0; c < 4; ++c) x[j][c] = c >= j ? a[c][j] : 0.0;
  double n2[4];
  for (int sweep = 0; sweep < kJacobiSweeps; ++sweep) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      n2[j] = 0.0;
#pragma unroll
      for (int i = 0; i < 4; ++i) n2[j] = fma(x[j][i], x[j][i], n2[j]);
    }
    bool rotated = false;
#pragma unroll
    for (int p = 0; p < 3; ++p) {
#pragma unroll
      for (int q = p + 1; q < 4; ++q) {
        double g = 0.0;
#pragma unroll
        for (int i = 0; i < 4; ++i) g = fma(x[p][i], x[q][i], g);
        // Orthogonal to 1e-13: the correction below squares what is left.
        if (!(g * g > 1e-26 * (n2[p] * n2[q]))) continue;
        rotated = true;
        const double d = n2[q] - n2[p], g2 = 2.0 * g;
        const double t = (d >= 0.0 ? g2 : -g2) / (fabs(d) + sqrt(fma(d, d, g2 * g2)));
        const double cs = rsqrt(fma(t, t, 1.0)), sn = cs * t;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const double u = x[p][i], w = x[q][i];
          x[p][i] = cs * u - sn * w;
          x[q][i] = sn * u + cs * w;
        }
        n2[p] = fma(-t, g, n2[p]);
        n2[q] = fma(t, g, n2[q]);
      }
    }
    if (!rotated) break;
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    n2[j] = 0.0;
#pragma unroll
    for (int i = 0; i < 4; ++i) n2[j] = fma(x[j][i], x[j][i], n2[j]);
  }
  // The shortest column goes last.
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const bool sw = n2[j] < n2[3];
    swap_if(sw, n2[j], n2[3]);
#pragma unroll
    for (int i = 0; i < 4; ++i) swap_if(sw, x[j][i], x[3][i]);
  }
  // Generalised cross product of the other three, from the 2x2 minors of the first two.
  const double m01 = x[0][0] * x[1][1] - x[0][1] * x[1][0];
  const double m02 = x[0][0] * x[1][2] - x[0][2] * x[1][0];
  const double m03 = x[0][0] * x[1][3] - x[0][3] * x[1][0];
  const double m12 = x[0][1] * x[1][2] - x[0][2] * x[1][1];
  const double m13 = x[0][1] * x[1][3] - x[0][3] * x[1][1];
  const double m23 = x[0][2] * x[1][3] - x[0][3] * x[1][2];
  double w[4];
  w[0] = x[2][1] * m23 - x[2][2] * m13 + x[2][3] * m12;
  w[1] = -(x[2][0] * m23 - x[2][2] * m03 + x[2][3] * m02);
  w[2] = x[2][0] * m13 - x[2][1] * m03 + x[2][3] * m01;
  w[3] = -(x[2][0] * m12 - x[2][1] * m02 + x[2][2] * m01);
  auto unpermute = [&](const double (&v)[4], double (&o)[4]) {
#pragma unroll
    for (int c = 0; c < 4; ++c)
      o[c] = perm[0] == c ? v[0] : perm[1] == c ? v[1] : perm[2] == c ? v[2] : v[3];
  };
  double y[4], grad[4] = {0.0, 0.0, 0.0, 0.0}, ww = 0.0;
  unpermute(w, y);
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    double res = 0.0;
#pragma unroll
    for (int c = 0; c < 4; ++c) res = fma(A[4 * r + c], y[c], res);
#pragma unroll
    for (int c = 0; c < 4; ++c) grad[c] = fma(A[4 * r + c], res, grad[c]);
    ww = fma(w[r], w[r], ww);
  }
  double z[4];  // grad in the order of w
#pragma unroll
  for (int c = 0; c < 4; ++c)
    z[c] = perm[c] == 0 ? grad[0] : perm[c] == 1 ? grad[1] : perm[c] == 2 ? grad[2] : grad[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    double d = 0.0;
#pragma unroll
    for (int i = 0; i < 4; ++i) d = fma(x[j][i], z[i], d);
    d /= n2[j] * (n2[j] - n2[3]);
    // Two (nearly) equal singular values leave the vector undetermined: no correction then.
    if (!(d * d * n2[j] <= 1e-6 * ww)) d = 0.0;
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = fma(-d, x[j][i], w[i]);
  }
  unpermute(w, out);
}

__global__ void __launch_bounds__(kSeedThreads) triangulate_kernel(
    const __grid_constant__ SeedCams cams, const SeedConsts c, int64_t m, int k,
    const int32_t* __restrict__ ref_view, const double* __restrict__ ref_xy,
    const int32_t* __restrict__ nb_view, const double* __restrict__ nb_xy,
    const float* __restrict__ nb_conf, uint32_t* __restrict__ valid, double* __restrict__ X_out,
    int32_t* __restrict__ best_out, double* __restrict__ err_out,
    double* __restrict__ angle_out, float* __restrict__ kappa_out) {
  chain_wait();
  const int64_t i = (int64_t)blockIdx.x * kSeedThreads + threadIdx.x;
  if (i >= m) return;
  const int r = ref_view[i];
  if (r < 0 || r >= cams.n_views) {  // not a view of this batch: no hypothesis
    valid[i] = 0u;
    best_out[i] = -1;
    kappa_out[i] = 0.0f;
    return;
  }
  const double xr = ref_xy[2 * i], yr = ref_xy[2 * i + 1];
  double kap = 0.0;
  int n_match = 0;
  // Accepted hypotheses of this pixel (slot order).
  double h_err[kMaxNb], h_ang[kMaxNb], h_X[kMaxNb][3];
  bool h_ok[kMaxNb];
  double emin = 0.0;
  bool any = false;
  for (int s = 0; s < k; ++s) {
    h_ok[s] = false;
    const int n = nb_view[i * k + s];
    if (n < 0 || n >= cams.n_views) continue;
    kap += (double)nb_conf[i * k + s];
    ++n_match;
    const double xn = nb_xy[2 * (i * k + s)], yn = nb_xy[2 * (i * k + s) + 1];
    double A[16];
    const double* Pr = cams.P[r];
    const double* Pn = cams.P[n];
    for (int j = 0; j < 4; ++j) {
      A[j] = xr * Pr[8 + j] - Pr[j];
      A[4 + j] = yr * Pr[8 + j] - Pr[4 + j];
      A[8 + j] = xn * Pn[8 + j] - Pn[j];
      A[12 + j] = yn * Pn[8 + j] - Pn[4 + j];
    }
    double Xh[4];
    smallest_right_singular_vector(A, Xh);
    if (Xh[3] == 0.0) continue;
    const double iw = 1.0 / Xh[3];
    const double X[3] = {Xh[0] * iw, Xh[1] * iw, Xh[2] * iw};
    double ur, wr, un, wn, cr[3], cn[3];
    project_pt(cams, r, X, ur, wr, cr);
    project_pt(cams, n, X, un, wn, cn);
    if (!(cr[2] > 0.0 && cn[2] > 0.0)) continue;
    const double err = sqrt(0.5 * ((ur - xr) * (ur - xr) + (wr - yr) * (wr - yr) +
                                   (un - xn) * (un - xn) + (wn - yn) * (wn - yn)));
    if (err > c.max_reproj) continue;
    double d1[3], d2[3], dot = 0.0, n1 = 0.0, n2 = 0.0;
    for (int a = 0; a < 3; ++a) {
      d1[a] = X[a] - cams.c[r][a];
      d2[a] = X[a] - cams.c[n][a];
      dot += d1[a] * d2[a];
      n1 += d1[a] * d1[a];
      n2 += d2[a] * d2[a];
    }
    const double cosang = fmin(1.0, fmax(-1.0, dot * rsqrt(n1 * n2)));
    const double ang = acos(cosang);
    if (ang < c.min_parallax) continue;
    h_ok[s] = true;
    h_err[s] = err;
    h_ang[s] = ang;
    h_X[s][0] = X[0];
    h_X[s][1] = X[1];
    h_X[s][2] = X[2];
    emin = any ? fmin(emin, err) : err;
    any = true;
  }
  // The lowest error wins; errors within tie_eps of the lowest are ties, decided by the larger
  // angle, then the earlier slot.
  bool found = false;
  double b_err = 0.0, b_ang = 0.0, bX[3] = {0.0, 0.0, 0.0};
  int b_k = -1;
  for (int s = 0; s < k; ++s) {
    if (!h_ok[s] || h_err[s] > emin + c.tie_eps) continue;
    if (!found || h_ang[s] > b_ang) {
      found = true;
      b_err = h_err[s];
      b_ang = h_ang[s];
      b_k = s;
      bX[0] = h_X[s][0];
      bX[1] = h_X[s][1];
      bX[2] = h_X[s][2];
    }
  }
  valid[i] = found ? 1u : 0u;
  X_out[3 * i] = bX[0];
  X_out[3 * i + 1] = bX[1];
  X_out[3 * i + 2] = bX[2];
  best_out[i] = b_k;
  err_out[i] = b_err;
  angle_out[i] = b_ang;
  kappa_out[i] = n_match ? (float)(kap / n_match) : 0.0f;
}

// Exact cell of X for cubes of edge h: 21 bits per axis (offset 2^20, clamped), as one 63-bit key.
constexpr int kCellMax = 2097151;
__device__ __forceinline__ int cell_coord(double x, double h) {
  return (int)fmin(fmax(floor(x / h) + 1048576.0, 0.0), (double)kCellMax);
}
__device__ __forceinline__ unsigned long long cell_key(int c0, int c1, int c2) {
  return ((unsigned long long)c0 << 42) | ((unsigned long long)c1 << 21) | (unsigned long long)c2;
}

// Entries to seed: valid, with a reference view of this batch.
__global__ void __launch_bounds__(kSeedThreads) seed_flags_kernel(
    int64_t m, int n_views, const uint32_t* __restrict__ valid,
    const int32_t* __restrict__ ref_view, uint32_t* __restrict__ flags) {
  chain_wait();
  const int64_t i = (int64_t)blockIdx.x * kSeedThreads + threadIdx.x;
  if (i < m) flags[i] = (valid[i] && ref_view[i] >= 0 && ref_view[i] < n_views) ? 1u : 0u;
}

// The accepted points in order, and the boxes of their cells on both grids (edges h0 and, if > 0,
// h1): box[g] = (max of kCellMax - c, max of c) per axis, zero on entry.
__global__ void __launch_bounds__(kSeedThreads) compact_points_kernel(
    int64_t m, const uint32_t* __restrict__ flags, const uint32_t* __restrict__ pos,
    const double* __restrict__ X, double h0, double h1, uint32_t* __restrict__ vidx,
    uint32_t (*__restrict__ box)[6]) {
  chain_wait();
  const int64_t i = (int64_t)blockIdx.x * kSeedThreads + threadIdx.x;
  const bool on = i < m && flags[i];
  if (on) vidx[pos[i]] = (uint32_t)i;
  for (int g = 0; g < 2; ++g) {
    const double h = g ? h1 : h0;
    if (!(h > 0.0)) continue;
    for (int a = 0; a < 3; ++a) {
      const int c = on ? cell_coord(X[3 * i + a], h) : 0;
      const uint32_t low = __reduce_max_sync(0xffffffffu, on ? (uint32_t)(kCellMax - c) : 0u);
      const uint32_t high = __reduce_max_sync(0xffffffffu, on ? (uint32_t)c : 0u);
      // Most warps widen nothing: they look before they take the one address all share.
      if ((threadIdx.x & 31) == 0) {
        if (low > *(volatile uint32_t*)&box[g][a]) atomicMax(&box[g][a], low);
        if (high > *(volatile uint32_t*)&box[g][3 + a]) atomicMax(&box[g][3 + a], high);
      }
    }
  }
}

// Cell keys of the accepted points, value = compact slot: one word relative to the box's corner
// when its cells fit in 32 bits (pack.on), else the low and high words of the 63-bit key. Both
// sort alike.
__global__ void __launch_bounds__(kSeedThreads) cell_keys_kernel(
    int s, const uint32_t* __restrict__ vidx, const double* __restrict__ X, double h,
    const CellPack pack, uint32_t* __restrict__ lo, uint32_t* __restrict__ hi,
    uint32_t* __restrict__ slot) {
  chain_wait();
  const int j = blockIdx.x * kSeedThreads + threadIdx.x;
  if (j >= s) return;
  const size_t i = vidx[j];
  int c[3];
  for (int a = 0; a < 3; ++a) c[a] = cell_coord(X[3 * i + a], h);
  if (pack.on) {
    lo[j] = ((uint32_t)(c[0] - pack.corner[0]) << (pack.bits[1] + pack.bits[2])) |
            ((uint32_t)(c[1] - pack.corner[1]) << pack.bits[2]) | (uint32_t)(c[2] - pack.corner[2]);
  } else {
    const unsigned long long key = cell_key(c[0], c[1], c[2]);
    lo[j] = (uint32_t)key;
    hi[j] = (uint32_t)(key >> 32);
  }
  slot[j] = (uint32_t)j;
}

__global__ void __launch_bounds__(kSeedThreads) gather_u32_kernel(int s,
                                                                  const uint32_t* __restrict__ src,
                                                                  const uint32_t* __restrict__ perm,
                                                                  uint32_t* __restrict__ dst) {
  chain_wait();
  const int j = blockIdx.x * kSeedThreads + threadIdx.x;
  if (j < s) dst[j] = src[perm[j]];
}

// Sorted cell keys (63-bit) and, unless null, points in sorted order: in double, and in cell units
// relative to their cell's corner (x, y, z in [0, 1)) with the cell's z index (exact in float). A
// point whose cell was clamped gets NaN there.
__global__ void __launch_bounds__(kSeedThreads) sorted_cells_kernel(
    int s, const uint32_t* __restrict__ perm, const uint32_t* __restrict__ vidx,
    const double* __restrict__ X, double h, unsigned long long* __restrict__ skey,
    double* __restrict__ sX, float4* __restrict__ local) {
  chain_wait();
  const int j = blockIdx.x * kSeedThreads + threadIdx.x;
  if (j >= s) return;
  const size_t i = vidx[perm[j]];
  int c[3];
  float off[3];
  for (int a = 0; a < 3; ++a) {
    const double x = X[3 * i + a];
    c[a] = cell_coord(x, h);
    const double o = x / h + 1048576.0 - (double)c[a];
    off[a] = o >= 0.0 && o < 1.0 ? (float)(x / h - (double)(c[a] - 1048576)) : NAN;
    if (sX) sX[3 * (size_t)j + a] = x;
  }
  skey[j] = cell_key(c[0], c[1], c[2]);
  if (local) local[j] = make_float4(off[0], off[1], off[2], (float)c[2]);
}

// Eigenvector of the smallest eigenvalue of the symmetric 3x3 matrix S (cyclic Jacobi).
__device__ void smallest_eigenvector3(double S[9], double v[3]) {
  double V[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1};
  for (int sweep = 0; sweep < kJacobiSweeps; ++sweep) {
    const double off = S[1] * S[1] + S[2] * S[2] + S[5] * S[5];
    const double diag = S[0] * S[0] + S[4] * S[4] + S[8] * S[8];
    if (off <= 1e-30 * diag || off == 0.0) break;
    for (int p = 0; p < 2; ++p) {
      for (int q = p + 1; q < 3; ++q) {
        const double apq = S[3 * p + q];
        if (apq == 0.0) continue;
        const double theta = (S[3 * q + q] - S[3 * p + p]) / (2.0 * apq);
        const double tt = (theta >= 0.0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
        const double cs = 1.0 / sqrt(tt * tt + 1.0), sn = tt * cs;
        // S <- J^T S J with J the rotation in the (p, q) plane.
        for (int kk = 0; kk < 3; ++kk) {
          const double skp = S[3 * kk + p], skq = S[3 * kk + q];
          S[3 * kk + p] = cs * skp - sn * skq;
          S[3 * kk + q] = sn * skp + cs * skq;
        }
        for (int kk = 0; kk < 3; ++kk) {
          const double spk = S[3 * p + kk], sqk = S[3 * q + kk];
          S[3 * p + kk] = cs * spk - sn * sqk;
          S[3 * q + kk] = sn * spk + cs * sqk;
        }
        for (int kk = 0; kk < 3; ++kk) {
          const double vkp = V[3 * kk + p], vkq = V[3 * kk + q];
          V[3 * kk + p] = cs * vkp - sn * vkq;
          V[3 * kk + q] = sn * vkp + cs * vkq;
        }
      }
    }
  }
  int j = 0;
  if (S[4] < S[3 * j + j]) j = 1;
  if (S[8] < S[3 * j + j]) j = 2;
  for (int a = 0; a < 3; ++a) v[a] = V[3 * a + j];
}

__device__ __forceinline__ int lower_bound_key(const unsigned long long* __restrict__ keys, int s,
                                               unsigned long long key) {
  int lo = 0, hi = s;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (keys[mid] < key) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Bilinear sample of view v at (x, y) (pixel (i, j) at (i, j)); false if the 2x2 footprint
// leaves the image.
__device__ __forceinline__ bool bilinear(const SeedCams& cams, const float* __restrict__ obs,
                                         int v, double x, double y, double out[3]) {
  const double fx0 = floor(x), fy0 = floor(y);
  const int W = cams.width[v], H = cams.height[v];
  if (!(fx0 >= 0.0 && fy0 >= 0.0 && fx0 + 1.0 <= W - 1 && fy0 + 1.0 <= H - 1)) return false;
  const int x0 = (int)fx0, y0 = (int)fy0;
  const double ax = x - fx0, ay = y - fy0;
  const float* base = obs + 3 * (cams.pixel_offset[v] + (long long)y0 * W + x0);
  for (int ch = 0; ch < 3; ++ch) {
    const double p00 = base[ch], p01 = base[3 + ch];
    const double p10 = base[3 * W + ch], p11 = base[3 * W + 3 + ch];
    out[ch] = (1 - ax) * (1 - ay) * p00 + ax * (1 - ay) * p01 + (1 - ax) * ay * p10 +
              ax * ay * p11;
  }
  return true;
}

__device__ __forceinline__ double median_of(double* a, int n) {
  for (int i = 1; i < n; ++i) {  // insertion sort of at most kMaxNb + 1 values
    const double x = a[i];
    int j = i - 1;
    while (j >= 0 && a[j] > x) {
      a[j + 1] = a[j];
      --j;
    }
    a[j + 1] = x;
  }
  return (n & 1) ? a[n / 2] : 0.5 * (a[n / 2 - 1] + a[n / 2]);
}

// ------------------------------------------------------------------------------------------
// Moments of the accepted points within the radius of each point (about the point): a warp per
// point, in cell order, so that neighbouring warps read the same cells.
// The points of a 3x3 column of cells along z are contiguous in the sorted order: lanes 0..8 and
// 16..24 find the nine ranges' ends, and the warp walks them as one sequence, 32 candidates at a
// time. Float coordinates in cell units decide most candidates (their error in d^2 is below 2e-6;
// within 4e-6 of the radius, or where a cell was clamped, the double test decides as before); the
// ones inside are queued in shared memory and accumulated in double 32 at a time, so that the FP64
// pipe, which bounds the kernel (16 cycles of an SM for each warp instruction), only sees points
// that count: 12 operations each. One thread per point with a double test per candidate kept a
// third of the lanes busy and searched 27 cells; with 100k points on a near wall it took 19.4 ms.
// ------------------------------------------------------------------------------------------
constexpr int kMomentThreads = 256;
constexpr int kMoments = 10;  // count, sum d (3), sum d d^T (6)

__global__ void __launch_bounds__(kMomentThreads) moments_kernel(
    int s, double h, const uint32_t* __restrict__ perm, const uint32_t* __restrict__ keep,
    const unsigned long long* __restrict__ skey, const double* __restrict__ sX,
    const float4* __restrict__ local, double* __restrict__ mom) {
  chain_wait();
  __shared__ int s_queue[kMomentThreads / 32][64];
  const int lane = threadIdx.x & 31;
  int* queue = s_queue[threadIdx.x >> 5];
  const int64_t q = ((int64_t)blockIdx.x * kMomentThreads + threadIdx.x) >> 5;
  if (q >= s) return;
  const uint32_t slot = perm[q];
  if (keep && !keep[slot]) return;
  const unsigned long long key = skey[q];
  const int a2 = (int)(key & kCellMax);
  // Lane r < 9 (and 16 + r): the column at (dx, dy) = (r / 3 - 1, r % 3 - 1).
  const int r = lane & 15;
  const int c0 = (int)(key >> 42) + r / 3 - 1, c1 = (int)((key >> 21) & kCellMax) + r % 3 - 1;
  const bool column = r < 9 && c0 >= 0 && c1 >= 0 && c0 <= kCellMax && c1 <= kCellMax;
  int end = 0;
  if (column) {
    const unsigned long long target = lane < 16 ? cell_key(c0, c1, max(a2 - 1, 0))
                                                : cell_key(c0, c1, min(a2 + 1, kCellMax)) + 1;
    end = lower_bound_key(skey, s, target);
  }
  const int begin = end;
  end = __shfl_down_sync(0xffffffffu, end, 16);
  const uint32_t len = column && lane < 16 ? (uint32_t)(end - begin) : 0u;
  uint32_t total;
  const uint32_t first = warp_exclusive_scan(len, &total);
  const double X0 = sX[3 * q], X1 = sX[3 * q + 1], X2 = sX[3 * q + 2];
  const float4 me = local[q];
  const double h2 = h * h;
  double v[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  auto add = [&](int p) {
    const double d0 = sX[3 * (size_t)p] - X0, d1 = sX[3 * (size_t)p + 1] - X1,
                 d2 = sX[3 * (size_t)p + 2] - X2;
    v[0] += d0;
    v[1] += d1;
    v[2] += d2;
    v[3] = fma(d0, d0, v[3]);
    v[4] = fma(d0, d1, v[4]);
    v[5] = fma(d0, d2, v[5]);
    v[6] = fma(d1, d1, v[6]);
    v[7] = fma(d1, d2, v[7]);
    v[8] = fma(d2, d2, v[8]);
  };
  int queued = 0, count = 0;
  for (uint32_t t0 = 0; t0 < total; t0 += 32) {
    const uint32_t t = t0 + lane;
    const int from = lane_of(first + len, t);
    const int p = __shfl_sync(0xffffffffu, begin, from) +
                  (int)(t - __shfl_sync(0xffffffffu, first, from));
    bool in = false;
    if (t < total) {
      const float4 o = local[p];
      const float f0 = (o.x - me.x) + (float)(from / 3 - 1);
      const float f1 = (o.y - me.y) + (float)(from % 3 - 1);
      const float f2 = (o.z - me.z) + (o.w - me.w);
      const float d2f = fmaf(f0, f0, fmaf(f1, f1, f2 * f2));
      in = d2f < 1.0f - 4e-6f;
      if (!in && !(d2f > 1.0f + 4e-6f)) {
        const double d0 = sX[3 * (size_t)p] - X0, d1 = sX[3 * (size_t)p + 1] - X1,
                     d2 = sX[3 * (size_t)p + 2] - X2;
        in = d0 * d0 + d1 * d1 + d2 * d2 <= h2;
      }
    }
    const unsigned inside = __ballot_sync(0xffffffffu, in);
    if (in) queue[queued + __popc(inside & ((1u << lane) - 1u))] = p;
    queued += __popc(inside);
    count += __popc(inside);
    __syncwarp();
    if (queued >= 32) {
      add(queue[lane]);
      queued -= 32;
      const int moved = lane < queued ? queue[32 + lane] : 0;
      __syncwarp();
      if (lane < queued) queue[lane] = moved;
      __syncwarp();
    }
  }
  if (lane < queued) add(queue[lane]);
  // Sum over the lanes, halving the values a lane answers for at each step (9, 5, 3, 2, 1): 12
  // additions instead of 45. Lane bits 4..1 select the value that ends up there.
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
  auto fold = [&](bool upper, double lo_v, double hi_v, int o) {
    const double give = upper ? lo_v : hi_v, held = upper ? hi_v : lo_v;
    return held + __shfl_xor_sync(0xffffffffu, give, o);
  };
  double w[5], u[3], y[2];
#pragma unroll
  for (int k = 0; k < 5; ++k) w[k] = fold(b4, v[k], k < 4 ? v[5 + k] : 0.0, 16);
#pragma unroll
  for (int k = 0; k < 3; ++k) u[k] = fold(b3, w[k], k < 2 ? w[3 + k] : 0.0, 8);
#pragma unroll
  for (int k = 0; k < 2; ++k) y[k] = fold(b2, u[k], k < 1 ? u[2] : 0.0, 4);
  double sum = fold(b1, y[0], y[1], 2);
  sum += __shfl_xor_sync(0xffffffffu, sum, 1);
  const int part = (b2 ? 2 : 0) + (b1 ? 1 : 0);
  const int which = (b4 ? 5 : 0) + (b3 ? 3 : 0) + part;
  double* out = mom + (size_t)kMoments * slot;
  if (!(lane & 1) && part < (b3 ? 2 : 3) && which < 9) out[1 + which] = sum;
  if (lane == 0) out[0] = (double)count;
}

// Per accepted point j (compact order): the seed's parameters, at its place among the kept ones
// (keep and place null: all are kept, in order). The SH coefficients beyond the DC term are set by
// zero_sh_kernel.
__global__ void __launch_bounds__(kSeedThreads) seed_kernel(
    const __grid_constant__ SeedCams cams, const SeedConsts c, int s, int k, int sh_k,
    const uint32_t* __restrict__ vidx, const uint32_t* __restrict__ keep,
    const uint32_t* __restrict__ place, const int32_t* __restrict__ ref_view,
    const int32_t* __restrict__ nb_view, const double* __restrict__ X_all,
    const double* __restrict__ err_all, const double* __restrict__ ang_all,
    const float* __restrict__ kappa_all, const double* __restrict__ mom,
    const float* __restrict__ obs, const float* __restrict__ gain_bias,
    int32_t* __restrict__ index, float* __restrict__ means, float* __restrict__ log_scales,
    float* __restrict__ quats, float* __restrict__ logits, float* __restrict__ sh,
    float* __restrict__ normals) {
  chain_wait();
  const int j = blockIdx.x * kSeedThreads + threadIdx.x;
  if (j >= s || (keep && !keep[j])) return;
  const size_t i = vidx[j];
  const size_t at = place ? place[j] : (size_t)j;
  const double X[3] = {X_all[3 * i], X_all[3 * i + 1], X_all[3 * i + 2]};
  const int r = ref_view[i];
  // Plane fit over the accepted points within the radius (moments about X).
  const double* mj = mom + (size_t)kMoments * j;
  const double cnt = mj[0];
  const double m1[3] = {mj[1], mj[2], mj[3]};
  const double m2[6] = {mj[4], mj[5], mj[6], mj[7], mj[8], mj[9]};
  const double* cr = cams.c[r];
  double toc[3] = {cr[0] - X[0], cr[1] - X[1], cr[2] - X[2]};
  const double tn = sqrt(toc[0] * toc[0] + toc[1] * toc[1] + toc[2] * toc[2]);
  double v[3];
  if (cnt >= 3.0) {
    const double mu[3] = {m1[0] / cnt, m1[1] / cnt, m1[2] / cnt};
    double S[9];
    S[0] = m2[0] / cnt - mu[0] * mu[0];
    S[1] = S[3] = m2[1] / cnt - mu[0] * mu[1];
    S[2] = S[6] = m2[2] / cnt - mu[0] * mu[2];
    S[4] = m2[3] / cnt - mu[1] * mu[1];
    S[5] = S[7] = m2[4] / cnt - mu[1] * mu[2];
    S[8] = m2[5] / cnt - mu[2] * mu[2];
    smallest_eigenvector3(S, v);
    const double nv = sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    for (int a = 0; a < 3; ++a) v[a] /= nv;
    if (v[0] * toc[0] + v[1] * toc[1] + v[2] * toc[2] < 0.0)
      for (int a = 0; a < 3; ++a) v[a] = -v[a];
  } else {
    for (int a = 0; a < 3; ++a) v[a] = toc[a] / tn;
  }
  // Tangent frame (Duff et al., JCGT 2017): [t1, t2, v] is a rotation.
  const double sg = v[2] >= 0.0 ? 1.0 : -1.0;
  const double aa = -1.0 / (sg + v[2]);
  const double bb = v[0] * v[1] * aa;
  const double t1[3] = {1.0 + sg * v[0] * v[0] * aa, sg * bb, -sg * v[0]};
  const double t2[3] = {bb, sg + v[1] * v[1] * aa, -v[1]};
  const double U[9] = {t1[0], t2[0], v[0], t1[1], t2[1], v[1], t1[2], t2[2], v[2]};
  // Quaternion (w, x, y, z), w >= 0 (Shepperd's branches).
  double q[4];
  const double tr = U[0] + U[4] + U[8];
  if (tr > 0.0) {
    const double sq = sqrt(tr + 1.0) * 2.0;
    q[0] = 0.25 * sq;
    q[1] = (U[7] - U[5]) / sq;
    q[2] = (U[2] - U[6]) / sq;
    q[3] = (U[3] - U[1]) / sq;
  } else if (U[0] > U[4] && U[0] > U[8]) {
    const double sq = sqrt(1.0 + U[0] - U[4] - U[8]) * 2.0;
    q[0] = (U[7] - U[5]) / sq;
    q[1] = 0.25 * sq;
    q[2] = (U[1] + U[3]) / sq;
    q[3] = (U[2] + U[6]) / sq;
  } else if (U[4] > U[8]) {
    const double sq = sqrt(1.0 + U[4] - U[0] - U[8]) * 2.0;
    q[0] = (U[2] - U[6]) / sq;
    q[1] = (U[1] + U[3]) / sq;
    q[2] = 0.25 * sq;
    q[3] = (U[5] + U[7]) / sq;
  } else {
    const double sq = sqrt(1.0 + U[8] - U[0] - U[4]) * 2.0;
    q[0] = (U[3] - U[1]) / sq;
    q[1] = (U[2] + U[6]) / sq;
    q[2] = (U[5] + U[7]) / sq;
    q[3] = 0.25 * sq;
  }
  const double qn = sqrt(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
  const double qs = (q[0] >= 0.0 ? 1.0 : -1.0) / qn;
  // Scales: s_perp from the reference projection Jacobian, s_par from angle and error.
  double ur, wr, xc[3];
  project_pt(cams, r, X, ur, wr, xc);
  const double z = xc[2];
  const double* R = cams.R[r];
  double Jc[6];
  for (int b = 0; b < 3; ++b) {
    const double j0 = cams.fx[r] / z, j2 = -cams.fx[r] * xc[0] / (z * z);
    const double k1 = cams.fy[r] / z, k2 = -cams.fy[r] * xc[1] / (z * z);
    Jc[b] = j0 * R[b] + j2 * R[6 + b];
    Jc[3 + b] = k1 * R[3 + b] + k2 * R[6 + b];
  }
  const double g00 = Jc[0] * Jc[0] + Jc[1] * Jc[1] + Jc[2] * Jc[2];
  const double g01 = Jc[0] * Jc[3] + Jc[1] * Jc[4] + Jc[2] * Jc[5];
  const double g11 = Jc[3] * Jc[3] + Jc[4] * Jc[4] + Jc[5] * Jc[5];
  const double s_perp = rsqrt(sqrt(g00 * g11 - g01 * g01));  // det(J J^T)^(-1/4)
  const double s_par = fmin(s_perp * (1.0 + err_all[i]) / sin(ang_all[i]), c.s_par_cap * s_perp);
  // Colour: median over the supporting views of the exposure-corrected bilinear samples.
  double smp[3][kMaxNb + 1];
  int ns = 0;
  for (int s2 = -1; s2 < k; ++s2) {
    const int vv = s2 < 0 ? r : nb_view[(size_t)i * k + s2];
    if (vv < 0 || vv >= cams.n_views) continue;
    double u, w, xcv[3], col[3];
    project_pt(cams, vv, X, u, w, xcv);
    if (!(xcv[2] > 0.0) || !bilinear(cams, obs, vv, u, w, col)) continue;
    const double g = gain_bias[2 * vv], b = gain_bias[2 * vv + 1];
    for (int ch = 0; ch < 3; ++ch) smp[ch][ns] = (col[ch] - b) / g;
    ++ns;
  }
  double colr[3] = {0.5, 0.5, 0.5};
  if (ns > 0)
    for (int ch = 0; ch < 3; ++ch) colr[ch] = median_of(smp[ch], ns);
  const double alpha = c.alpha_lo + (c.alpha_hi - c.alpha_lo) * (double)kappa_all[i];
  const double Y0 = 0.28209479177387814;
  index[at] = (int32_t)i;
  for (int a = 0; a < 3; ++a) {
    means[3 * at + a] = (float)X[a];
    normals[3 * at + a] = (float)v[a];
  }
  log_scales[3 * at] = (float)log(s_perp);
  log_scales[3 * at + 1] = (float)log(s_perp);
  log_scales[3 * at + 2] = (float)log(s_par);
  for (int a = 0; a < 4; ++a) quats[4 * at + a] = (float)(q[a] * qs);
  logits[at] = (float)log(alpha / (1.0 - alpha));
  for (int ch = 0; ch < 3; ++ch) sh[at * sh_k * 3 + ch] = (float)((colr[ch] - 0.5) / Y0);
}

// The SH coefficients beyond the DC term of the `kept` seeds, side by side.
__global__ void __launch_bounds__(kSeedThreads) zero_sh_kernel(const uint32_t* __restrict__ kept,
                                                               int row, float* __restrict__ sh) {
  chain_wait();
  const int64_t n = (int64_t)*kept * row;
  for (int64_t e = (int64_t)blockIdx.x * kSeedThreads + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * kSeedThreads)
    if (e % row >= 3) sh[e] = 0.0f;
}

// Voxel thinning: after sorting by voxel key, the first entry of each run picks the run's best
// seed (highest confidence as float, then lowest reference index) and marks it kept.
__global__ void __launch_bounds__(kSeedThreads) voxel_best_kernel(
    int s, const unsigned long long* __restrict__ skey, const uint32_t* __restrict__ perm,
    const uint32_t* __restrict__ vidx, const float* __restrict__ kappa_all,
    uint32_t* __restrict__ keep) {
  chain_wait();
  const int j = blockIdx.x * kSeedThreads + threadIdx.x;
  if (j >= s || (j > 0 && skey[j - 1] == skey[j])) return;
  int best = perm[j];
  for (int q = j + 1; q < s && skey[q] == skey[j]; ++q) {
    const int cand = perm[q];
    const float kc = kappa_all[vidx[cand]], kb = kappa_all[vidx[best]];
    if (kc > kb || (kc == kb && vidx[cand] < vidx[best])) best = cand;
  }
  keep[best] = 1u;
}

unsigned blocks_for(int64_t n) { return (unsigned)((n + kSeedThreads - 1) / kSeedThreads); }

}  // namespace

cudaError_t launch_triangulate(const SeedCams& cams, const SeedConsts& c, int64_t m, int k,
                               const int32_t* ref_view, const double* ref_xy,
                               const int32_t* nb_view, const double* nb_xy, const float* nb_conf,
                               uint32_t* valid, double* X, int32_t* best, double* err,
                               double* angle, float* kappa, cudaStream_t stream) {
  if (m == 0) return cudaSuccess;
  const cudaError_t e = launch_chained(triangulate_kernel, dim3(blocks_for(m)),
                                       dim3(kSeedThreads), stream, cams, c, m, k, ref_view,
                                       ref_xy, nb_view, nb_xy, nb_conf, valid, X, best, err,
                                       angle, kappa);
  RGS_LAUNCHED();
  return e;
}

namespace {

// Stable sort of the s points by cell of edge h: the permutation (sorted position -> compact slot)
// in *perm. Cells within a box of up to 32 bits take one sort of as many bits (a room in 5 cm
// cells: 21 bits, 3 passes); else the low words are sorted, then the gathered high words (8
// passes).
cudaError_t sort_by_cell(const SeedScratch& w, int s, const double* X, double h,
                         const CellPack& pack, uint32_t** perm, cudaStream_t stream) {
  const dim3 grid(blocks_for(s)), block(kSeedThreads);
  cudaError_t e = launch_chained(cell_keys_kernel, grid, block, stream, s,
                                 (const uint32_t*)w.vidx, X, h, pack, w.lo, w.hi, w.slot);
  RGS_LAUNCHED();
  if (e != cudaSuccess) return e;
  const int bits = pack.on ? pack.bits[0] + pack.bits[1] + pack.bits[2] : 32;
  bool alt = false;
  if (bits > 0)
    e = launch_radix_sort(w.lo, w.slot, w.t0, w.t1, s, nullptr, 0, bits, w.hist, w.block_sums,
                          &alt, stream, kSortItemsSmall);
  uint32_t* p1 = alt ? w.t1 : w.slot;
  *perm = p1;
  if (pack.on || e != cudaSuccess) return e;
  uint32_t* spare = alt ? w.slot : w.t1;
  uint32_t* high = alt ? w.lo : w.t0;  // the buffer not holding p1's keys
  e = launch_chained(gather_u32_kernel, grid, block, stream, s, (const uint32_t*)w.hi,
                     (const uint32_t*)p1, high);
  RGS_LAUNCHED();
  if (e != cudaSuccess) return e;
  e = launch_radix_sort(high, p1, w.hi, spare, s, nullptr, 0, 31, w.hist, w.block_sums, &alt,
                        stream, kSortItemsSmall);
  *perm = alt ? spare : p1;
  return e;
}

}  // namespace

cudaError_t launch_accept_points(const SeedScratch& w, int64_t m, int n_views,
                                 const uint32_t* valid, const int32_t* ref_view, const double* X,
                                 double plane_radius, double voxel, cudaStream_t stream) {
  cudaError_t e = cudaMemsetAsync(w.counts, 0, w.reset_bytes, stream);
  if (e != cudaSuccess) return e;
  const dim3 grid(blocks_for(m)), block(kSeedThreads);
  e = launch_chained(seed_flags_kernel, grid, block, stream, m, n_views, valid, ref_view, w.flags);
  RGS_LAUNCHED();
  if (e == cudaSuccess)
    e = launch_exclusive_scan_single_pass(w.flags, w.pos, m, &w.counts->accepted, w.lb[0], stream);
  if (e == cudaSuccess) {
    e = launch_chained(compact_points_kernel, grid, block, stream, m, (const uint32_t*)w.flags,
                       (const uint32_t*)w.pos, X, plane_radius, voxel, w.vidx, w.counts->box);
    RGS_LAUNCHED();
  }
  return e;
}

cudaError_t launch_seeds(const SeedScratch& w, const SeedCams& cams, const SeedConsts& c,
                         const CellPack (&pack)[2], int s, int k, int sh_k,
                         const int32_t* ref_view, const int32_t* nb_view, const double* X,
                         const double* err, const double* angle, const float* kappa,
                         const float* obs, const float* gain_bias, int32_t* index, float* means,
                         float* log_scales, float* quats, float* logits, float* sh,
                         float* normals, cudaStream_t stream) {
  if (s == 0) return cudaSuccess;
  const dim3 grid(blocks_for(s)), block(kSeedThreads);
  uint32_t* perm = nullptr;
  cudaError_t e = cudaSuccess;
  const uint32_t *keep = nullptr, *place = nullptr, *kept = &w.counts->accepted;
  if (c.voxel > 0.0) {
    e = cudaMemsetAsync(w.flags, 0, sizeof(uint32_t) * (size_t)s, stream);
    if (e == cudaSuccess) e = sort_by_cell(w, s, X, c.voxel, pack[1], &perm, stream);
    if (e == cudaSuccess) {
      e = launch_chained(sorted_cells_kernel, grid, block, stream, s, (const uint32_t*)perm,
                         (const uint32_t*)w.vidx, X, c.voxel, w.skey, (double*)nullptr,
                         (float4*)nullptr);
      RGS_LAUNCHED();
    }
    if (e == cudaSuccess) {
      e = launch_chained(voxel_best_kernel, grid, block, stream, s,
                         (const unsigned long long*)w.skey, (const uint32_t*)perm,
                         (const uint32_t*)w.vidx, kappa, w.flags);
      RGS_LAUNCHED();
    }
    if (e == cudaSuccess)
      e = launch_exclusive_scan_single_pass(w.flags, w.pos, s, &w.counts->kept, w.lb[1], stream);
    keep = w.flags;
    place = w.pos;
    kept = &w.counts->kept;
  }
  if (e == cudaSuccess) e = sort_by_cell(w, s, X, c.plane_radius, pack[0], &perm, stream);
  if (e == cudaSuccess) {
    e = launch_chained(sorted_cells_kernel, grid, block, stream, s, (const uint32_t*)perm,
                       (const uint32_t*)w.vidx, X, c.plane_radius, w.skey, w.sX, w.local);
    RGS_LAUNCHED();
  }
  if (e == cudaSuccess) {
    const unsigned blocks =
        (unsigned)(((int64_t)s * 32 + kMomentThreads - 1) / kMomentThreads);
    e = launch_chained(moments_kernel, dim3(blocks), dim3(kMomentThreads), stream, s,
                       c.plane_radius, (const uint32_t*)perm, keep,
                       (const unsigned long long*)w.skey, (const double*)w.sX,
                       (const float4*)w.local, w.mom);
    RGS_LAUNCHED();
  }
  if (e == cudaSuccess) {
    e = launch_chained(seed_kernel, grid, block, stream, cams, c, s, k, sh_k,
                       (const uint32_t*)w.vidx, keep, place, ref_view, nb_view, X, err, angle,
                       kappa, (const double*)w.mom, obs, gain_bias, index, means, log_scales,
                       quats, logits, sh, normals);
    RGS_LAUNCHED();
  }
  if (e == cudaSuccess && sh_k > 1) {
    const int64_t need = ((int64_t)s * 3 * sh_k + kSeedThreads - 1) / kSeedThreads;
    e = launch_chained(zero_sh_kernel, dim3((unsigned)std::min<int64_t>(need, 16 * 152)), block,
                       stream, kept, 3 * sh_k, sh);
    RGS_LAUNCHED();
  }
  return e;
}

}  // namespace rgs

// Densities of refined modes where the order of the modes hangs on them.
//
// A mode's density comes out of its refinement as a sum of FP32 weights over rows
// rounded to FP32 in scaled coordinates, good to about 1e-7 (more, far from the
// origin).  Modes closer than that to another one in density are evaluated again
// at their FP64 positions, from the caller's coordinates, with differences,
// weights and sums in FP64; all others keep what they have, which orders them
// rightly.
#pragma once

#include "fms_internal.cuh"

namespace fms {

// What an FP64 density is evaluated over; X null: nothing is evaluated again.
struct DensityRows {
  const float* X;   // the caller's rows of d values
  int64_t n;
  double scale;     // positions are given in units of 1 / scale
  int unit;         // 1: over the rows' directions (cosine metric)
};

// Whether the densities sa, sb at pa, pb are closer than their error allows to tell
// apart: 4e-6 for the FP32 weights and sums (a few 1e-7 each), and 2e-7 |p| for the
// rounding of the scaled rows (2^-25 |p| a coordinate moves a log-weight by 2 ln 2
// times the distance times that).
__device__ __forceinline__ bool near_tie(double sa, const double* pa, double sb, const double* pb,
                                         int d) {
  const double gap = fabs(sa - sb), top = fmax(sa, sb);
  if (!(gap <= 0.05 * top)) return false;
  double na = 0.0, nb = 0.0;
  for (int k = 0; k < d; ++k) {
    na += pa[k] * pa[k];
    nb += pb[k] * pb[k];
  }
  return gap <= top * fmin(0.05, 4e-6 + 2e-7 * (sqrt(na) + sqrt(nb)));
}

constexpr int kDensityWarps = 8;   // warps of a block that evaluates densities

struct DensitySmem {
  double y[64];
  float yf[64];
  double red[kDensityWarps][65];
};

// sum_j w_j = exp2(-scale^2 ||x_j - y||^2) over all rows by the whole block, y = sm.y in
// the caller's units; SHIFT: and sum_j w_j (x_j - y), in red[0][1 + k].  Rows whose
// exponent is beyond 100 in FP32 are left out (n 2^-99 of weights, one of which is about
// 1).  A lane takes a row for its weight, then the lanes take the coordinates of the
// rows that count; fixed order of sums.
template <bool SHIFT>
__device__ inline double density_pass(const DensityRows& D, int d, DensitySmem& sm) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const double s2 = D.scale * D.scale;
  const float sf = (float)D.scale;
  double sum = 0.0, s[2] = {0.0, 0.0};
  for (int64_t j0 = (int64_t)w * 32; j0 < D.n; j0 += 32 * kDensityWarps) {
    const int64_t j = j0 + lane;
    const float* r = D.X + j * d;
    double wt = 0.0, f = 1.0;
    bool in = j < D.n;
    if (in) {
      float inv = 1.0f, t = 0.0f;
      if (D.unit) {
        float nn = 0.0f;
        for (int k = 0; k < d; ++k) nn = fmaf(r[k], r[k], nn);
        inv = nn > 1e-30f && nn < 1e30f ? 1.0f / sqrtf(nn) : NAN;   // (NaN: FP64 decides)
      }
      for (int k = 0; k < d; ++k) {
        const float e = (r[k] * inv - sm.yf[k]) * sf;
        t = fmaf(e, e, t);
      }
      in = !(t > 100.0f);
    }
    if (in) {
      double q = 0.0;
      if (D.unit) {
        double nn = 0.0;
        for (int k = 0; k < d; ++k) nn += (double)r[k] * (double)r[k];
        f = 1.0 / sqrt(nn);
      }
      for (int k = 0; k < d; ++k) {
        const double e = (double)r[k] * f - sm.y[k];
        q += e * e;
      }
      wt = exp2(-q * s2);
      sum += wt;
    }
    if (!SHIFT) continue;
    unsigned left = __ballot_sync(kFull, in);
    while (left) {
      const int u = __ffs(left) - 1;
      left &= left - 1;
      const double wu = __shfl_sync(kFull, wt, u), fu = __shfl_sync(kFull, f, u);
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const int k = lane + 32 * v;
        if (k < d) s[v] += wu * ((double)D.X[(j0 + u) * d + k] * fu - sm.y[k]);
      }
    }
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
  if (lane == 0) sm.red[w][0] = sum;
  if (SHIFT) {
#pragma unroll
    for (int v = 0; v < 2; ++v) sm.red[w][1 + lane + 32 * v] = s[v];
  }
  __syncthreads();
  for (int k = threadIdx.x; k <= (SHIFT ? d : 0); k += blockDim.x) {
    double v = sm.red[0][k];
    for (int u = 1; u < kDensityWarps; ++u) v += sm.red[u][k];
    sm.red[0][k] = v;
  }
  __syncthreads();
  sum = sm.red[0][0];
  return sum;
}

// The density of the mode at pos (in units of 1 / scale) by a block of 32 kDensityWarps
// threads; every thread gets it.  One more update first: the refinement ran on rows
// rounded in scaled coordinates, and its last 2^-25 |p| would decide between modes of
// equal density (single points far from the origin).  Bound by the FP64 pipe (~30 + 5 d
// operations a row that counts, 2 an SM and clock) and run for near ties only.
__device__ inline double mode_density(const DensityRows& D, int d, const double* pos,
                                      DensitySmem& sm) {
  const double inv_scale = 1.0 / D.scale;
  __syncthreads();
  for (int k = threadIdx.x; k < d; k += blockDim.x) {
    sm.y[k] = pos[k] * inv_scale;
    sm.yf[k] = (float)sm.y[k];
  }
  __syncthreads();
  const double W = density_pass<true>(D, d, sm);
  double nn = 0.0;
  if (D.unit)
    for (int k = 0; k < d; ++k) {
      const double v = sm.y[k] + sm.red[0][1 + k] / W;
      nn += v * v;
    }
  const double f = D.unit ? 1.0 / sqrt(nn) : 1.0;
  if (!(W > 0.0) || !isfinite(f)) return W;   // (the same for every thread)
  __syncthreads();
  for (int k = threadIdx.x; k < d; k += blockDim.x) {
    sm.y[k] = (sm.y[k] + sm.red[0][1 + k] / W) * f;
    sm.yf[k] = (float)sm.y[k];
  }
  __syncthreads();
  return density_pass<false>(D, d, sm);
}

// Order of two modes: density descending, ties by lexicographic coordinates.
__device__ __forceinline__ bool mode_before(double sa, const double* a, double sb, const double* b,
                                            int d) {
  if (sa != sb) return sa > sb;
  for (int k = 0; k < d; ++k)
    if (a[k] != b[k]) return a[k] < b[k];
  return false;
}

}  // namespace fms

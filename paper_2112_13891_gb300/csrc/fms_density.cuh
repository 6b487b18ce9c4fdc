// Densities of refined modes where the order of the modes hangs on them.
//
// A mode's density comes out of its refinement as a sum of FP32 weights over rows
// rounded to FP32 in scaled coordinates, good to some 1e-7 (less, far from the origin).
// Modes closer than that to another one in density are evaluated again at their FP64
// positions, from the caller's coordinates, with differences, weights and sums in FP64;
// all others keep what they have, which orders them rightly.
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

// Error of a density s = sum of weights at p, relative: 2e-7 for its FP32 sums, and the
// rows' own errors (5e-7 of FP32 weights; the rounding of scaled coordinates to 2^-25 |x|
// moves a log-weight by 2 ln 2 times the distance times that), which average out over
// the rows, of which s is no more than the number that count.
__device__ __forceinline__ float density_error(double s, float norm) {
  return 2e-7f + (7.5e-7f + 5e-8f * norm) * rsqrtf(fmaxf((float)s, 1.0f));
}
// Whether two densities are too close to tell apart (compared in FP32, whose rounding the
// errors cover).
__device__ __forceinline__ bool near_tie(float sa, float ea, float sb, float eb) {
  return fabsf(sa - sb) <= fmaxf(sa, sb) * fminf(0.05f, ea + eb);
}
__device__ __forceinline__ float mode_norm(const double* p, int d) {
  double s = 0.0;
#pragma unroll 8
  for (int k = 0; k < d; ++k) s += p[k] * p[k];
  return sqrtf((float)s);
}

constexpr int kDensityWarps = 8;    // warps of a block that evaluates densities
constexpr int kOrderStage = 1024;   // modes whose scores fit in shared memory
constexpr int kTieCap = 16;         // tied modes whose rows are split over the blocks

// Scratch of the split evaluations of `blocks` blocks.
inline size_t tie_scratch_bytes(int blocks, int d) {
  return (size_t)blocks * kTieCap * (d + 1) * 8;
}

struct OrderSmem {
  double score[kOrderStage];
  float rough[kOrderStage], err[kOrderStage];   // the score, its error
  double y[64];
  float yf[64];
  double red[kDensityWarps][65];
  unsigned char flag[kOrderStage];   // the mode is in a near tie
  int queue[kDensityWarps][64];
  int tied[kTieCap];
  int ntied, last;
};

// sum_j w_j = exp2(-scale^2 ||x_j - p / scale||^2) and sum_j w_j (x_j - p / scale) over
// rows [j0, j1) by the whole block, into sm.red[0][0 .. d].  A row counts if its exponent
// in FP32 is below `bits`; a warp queues such rows and takes 32 at a time, a lane a row
// for the weights, then a coordinate (an FP64 instruction keeps the SM's pipe for 16
// clocks however few of its lanes take part); fixed order of sums.
__device__ inline void density_sums(const DensityRows& D, int64_t j0, int64_t j1, int d,
                                    const double* pos, float bits, OrderSmem& sm) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const double s2 = D.scale * D.scale, inv_scale = 1.0 / D.scale;
  const float sf = (float)D.scale;
  __syncthreads();
  for (int k = threadIdx.x; k < 64; k += blockDim.x) {
    sm.y[k] = k < d ? pos[k] * inv_scale : 0.0;
    sm.yf[k] = (float)sm.y[k];
  }
  __syncthreads();
  double sum = 0.0, s[2] = {0.0, 0.0};
  int* queue = sm.queue[w];
  int queued = 0;
  auto take = [&](int cnt) {   // the first cnt <= 32 queued rows
    double wt = 0.0, f = 1.0;
    int64_t j = 0;
    if (lane < cnt) {
      j = j0 + queue[lane];
      const float* r = D.X + j * d;
      double q = 0.0;
      if (D.unit) {
        double nn = 0.0;
#pragma unroll 4
        for (int k = 0; k < d; ++k) nn += (double)r[k] * (double)r[k];
        f = 1.0 / sqrt(nn);
      }
#pragma unroll 4
      for (int k = 0; k < d; ++k) {
        const double e = (double)r[k] * f - sm.y[k];
        q += e * e;
      }
      wt = exp2(-q * s2);
      sum += wt;
    }
    for (int u = 0; u < cnt; ++u) {
      const double wu = __shfl_sync(kFull, wt, u), fu = __shfl_sync(kFull, f, u);
      const int64_t ju = __shfl_sync(kFull, j, u);
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const int k = lane + 32 * v;
        if (k < d) s[v] += wu * ((double)D.X[ju * d + k] * fu - sm.y[k]);
      }
    }
    __syncwarp();
  };
  for (int64_t jb = j0 + w * 32; jb < j1; jb += 32 * kDensityWarps) {
    const int64_t j = jb + lane;
    const float* r = D.X + j * d;
    bool in = j < j1;
    if (in) {
      float inv = 1.0f, t = 0.0f;
      if (D.unit) {
        float nn = 0.0f;
#pragma unroll 8
        for (int k = 0; k < d; ++k) nn = fmaf(r[k], r[k], nn);
        inv = nn > 1e-30f && nn < 1e30f ? 1.0f / sqrtf(nn) : NAN;   // (NaN: FP64 decides)
      }
      for (int k0 = 0; k0 < d; k0 += 8) {   // (eight loads in flight)
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = k0 + u < d ? __ldg(r + k0 + u) : 0.0f;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const float e = (v[u] * inv - sm.yf[k0 + u]) * sf;   // (yf: zero from d on)
          t = fmaf(e, e, t);
        }
      }
      in = !(t > bits);
    }
    const unsigned m = __ballot_sync(kFull, in);
    if (in) queue[queued + __popc(m & ((1u << lane) - 1u))] = (int)(j - j0);
    queued += __popc(m);
    __syncwarp();
    if (queued >= 32) {
      take(32);
      queued -= 32;
      const int rest = queue[32 + lane];
      __syncwarp();
      if (lane < queued) queue[lane] = rest;
      __syncwarp();
    }
  }
  take(queued);
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
  if (lane == 0) sm.red[w][0] = sum;
#pragma unroll
  for (int v = 0; v < 2; ++v)
    if (lane + 32 * v < 64) sm.red[w][1 + lane + 32 * v] = s[v];
  __syncthreads();
  for (int k = threadIdx.x; k <= d; k += blockDim.x) {
    double v = sm.red[0][k];
    for (int u = 1; u < kDensityWarps; ++u) v += sm.red[u][k];
    sm.red[0][k] = v;
  }
  __syncthreads();
}

// Rows left out below this exponent weigh 2^-37 of the mode's density together.
__device__ __forceinline__ float density_bits(double score, int64_t n) {
  return fminf(fmaxf(39.0f + log2f((float)n) - log2f((float)score), 40.0f), 1000.0f);
}

// The density at the mode from the sums (W, S) at a position next to it: the refinement
// ran on rows rounded in scaled coordinates, and what that leaves (2^-25 |p|) must not
// decide between single points of equal density.  With e = S / W the step to the mode,
// W(p + e) = W (1 + a |e|^2) to second order in e for a = ln 2 scale^2, but for a term of
// (e . (x - p))^2, as small again for points closer than 1 / scale.  Rounded to 36 bits:
// whole densities are whole.
__device__ __forceinline__ double mode_density(const double* sums, int d, double scale) {
  const double W = sums[0];
  double e2 = 0.0;
  for (int k = 0; k < d; ++k) e2 += sums[1 + k] * sums[1 + k];
  const double v = W * (1.0 + 0.69314718055994531 * scale * scale * e2 / (W * W));
  if (!(v > 0.0) || !isfinite(v)) return W;
  int e;
  const double m = frexp(v, &e);
  return ldexp(rint(ldexp(m, 36)), e - 36);
}

// The near ties' part of order_densities, for the modes that sm.flag marks (out of line:
// without any, a call's time is that of fetching the rest).
static __device__ __noinline__ bool share_ties(const DensityRows& D, const double* __restrict__ pos,
                                        double* dens, const int32_t* __restrict__ acc, int M,
                                        int d, int DP, double* scratch, int32_t* ticket, int bi,
                                        int nb, OrderSmem& sm) {
  if (threadIdx.x < 32) {   // the tied modes, in order
    int n = 0;
    for (int i0 = 0; i0 < M; i0 += 32) {
      const int i = i0 + (int)threadIdx.x;
      const unsigned m = __ballot_sync(kFull, i < M && sm.flag[i]);
      const int at = n + __popc(m & ((1u << threadIdx.x) - 1u));
      if (((m >> threadIdx.x) & 1u) && at < kTieCap) sm.tied[at] = i;
      n += __popc(m);
    }
    if (threadIdx.x == 0) sm.ntied = n;
  }
  __syncthreads();
  const int T = sm.ntied;
  const bool split = T <= kTieCap && nb > 1;
  if (split) {
    const int64_t per = (D.n + nb - 1) / nb;
    const int64_t j0 = bi * per, j1 = j0 + per < D.n ? j0 + per : D.n;
    for (int u = 0; u < T; ++u) {
      const int i = sm.tied[u], a = acc ? acc[i] : i;
      density_sums(D, j0, j1, d, pos + (int64_t)a * DP, density_bits(sm.score[i], D.n), sm);
      double* o = scratch + ((int64_t)bi * kTieCap + u) * (d + 1);
      for (int k = threadIdx.x; k <= d; k += blockDim.x) o[k] = sm.red[0][k];
    }
  } else {
    int at = 0;
    for (int i = 0; i < M; ++i) {
      if (!sm.flag[i] || at++ % nb != bi) continue;   // (the same for the whole block)
      const int a = acc ? acc[i] : i;
      density_sums(D, 0, D.n, d, pos + (int64_t)a * DP, density_bits(sm.score[i], D.n), sm);
      if (threadIdx.x == 0) dens[a] = mode_density(sm.red[0], d, D.scale);
    }
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    sm.last = atomicAdd(ticket, 1) == nb - 1;
    if (sm.last) *ticket = 0;
  }
  __syncthreads();
  if (!sm.last) return false;
  __threadfence();
  if (split) {
    for (int u = 0; u < T; ++u) {
      for (int k = threadIdx.x; k <= d; k += blockDim.x) {
        double v = 0.0;
        for (int b = 0; b < nb; ++b)
          v += __ldcg(scratch + ((int64_t)b * kTieCap + u) * (d + 1) + k);
        sm.red[0][k] = v;
      }
      __syncthreads();
      if (threadIdx.x == 0) sm.score[sm.tied[u]] = mode_density(sm.red[0], d, D.scale);
      __syncthreads();
    }
  } else {
    for (int i = threadIdx.x; i < M; i += blockDim.x)
      if (sm.flag[i]) sm.score[i] = __ldcg(dens + (acc ? acc[i] : i));
  }
  __syncthreads();
  return true;
}

// The modes' densities for the final order, by blocks bi = 0 .. nb - 1 (32 kDensityWarps
// threads each) of one set of modes acc[i] (null: i), M <= kOrderStage: sm.score[i], the
// near ties' from FP64.  Every block looks for near ties among all modes; where there are
// none, all return true at once (*tied = false).  Else the blocks share the rows of up to
// kTieCap tied modes, or the tied modes, and only the last to finish returns true
// (*ticket counts them; no waiting; 0 again afterwards).
__device__ inline bool order_densities(const DensityRows& D, const double* __restrict__ pos,
                                       const double* __restrict__ score, double* dens,
                                       const int32_t* __restrict__ acc, int M, int d, int DP,
                                       double* scratch, int32_t* ticket, int bi, int nb,
                                       OrderSmem& sm, bool* tied) {
  *tied = false;
  for (int j = threadIdx.x; j < M; j += blockDim.x) {
    const int a = acc ? acc[j] : j;
    sm.score[j] = score[a];
    sm.rough[j] = (float)score[a];
    if (D.X) sm.err[j] = density_error(score[a], mode_norm(pos + (int64_t)a * DP, d));
  }
  if (threadIdx.x == 0) sm.ntied = 0;
  __syncthreads();
  if (!D.X) return true;
  int mine = 0;
  for (int i = threadIdx.x; i < M; i += blockDim.x) {
    const float si = sm.rough[i], ei = sm.err[i];
    bool t = false;
    for (int j = 0; j < M; ++j) t = t || (j != i && near_tie(si, ei, sm.rough[j], sm.err[j]));
    sm.flag[i] = t ? 1 : 0;
    mine += t ? 1 : 0;
  }
  if (!__syncthreads_or(mine)) return true;
  *tied = true;
  return share_ties(D, pos, dens, acc, M, d, DP, scratch, ticket, bi, nb, sm);
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

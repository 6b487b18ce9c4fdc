// The probe of fms_route.cuh: one cluster of eight blocks a sampled set.
//
// A cell's radius is about the distance M from a sampled point to the nearest other one
// (the cells have as many pivots as the sample has points); a cell whose centre lies at
// distance a from a seed is seen within the cutoff and the cell's reach.  From a sampled
// point x of the cell, a^2 = |x - y|^2 - M^2 / 2 (x is M / sqrt 2 from the centre, at right
// angles to y - centre where there are many dimensions).  The cutoff follows from the
// sample's weights, as the walk takes it from W.  A set of more clusters than points in the
// sample has a large M and comes out as one without clusters.
//
// Bound by latency: 3 us at d = 3, 6 at d = 32.
#include <cooperative_groups.h>

#include "fms_cells.cuh"
#include "fms_route.cuh"

namespace fms {
namespace {

constexpr int kBlocks = 8;
constexpr int kNear = kProbePoints / kBlocks, kSeedsPer = kProbeSeeds / kBlocks;
constexpr int kRowsPer = kNear + kSeedsPer;   // rows a block compares with all points

__device__ __forceinline__ int64_t strided(int i, int of, int64_t n) {
  return ((2 * (int64_t)i + 1) * n) / (2 * (int64_t)of);
}

template <typename T>
__global__ void __cluster_dims__(kBlocks, 1, 1) __launch_bounds__(kProbePoints)
    probe_kernel(ProbeArgs a) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) float probe_smem[];
  const int d4 = (a.d + 3) & ~3, ld = d4 + 4;   // (rows 16 bytes apart modulo 128: no conflicts)
  float* pts = probe_smem;                      // [kProbePoints][ld]
  float* seeds = pts + kProbePoints * ld;       // [kSeedsPer][ld]
  __shared__ __align__(16) float near[kProbePoints];          // of the first block: all points'
  __shared__ float red[kRowsPer][kProbePoints / 32];
  __shared__ float median;
  __shared__ int seen[kBlocks], sum[32];
  cg::cluster_group cl = cg::this_cluster();
  const int b = blockIdx.x / kBlocks, rank = blockIdx.x % kBlocks, t = threadIdx.x;
  const int lane = t & 31, w = t >> 5;
  const ProbeSet s = a.set[b];
  const T *X = static_cast<const T*>(s.X), *Y = static_cast<const T*>(s.Y);
  const float scale = (float)a.scale;
  // a thread loads its point (eight values in flight) and an element or two of the seeds
  const float in = a.unit ? 1.0f : scale;
  const T* x = X + strided(t, kProbePoints, s.n) * a.ld;
  float sv[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int e = t + u * kProbePoints, r = e / d4, k = e - r * d4;
    sv[u] = r < kSeedsPer && k < a.d
                ? (float)Y[strided(rank * kSeedsPer + r, kProbeSeeds, s.m) * a.ld + k]
                : 0.0f;
  }
  for (int k0 = 0; k0 < d4; k0 += 8) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = k0 + u < a.d ? (float)x[k0 + u] : 0.0f;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (k0 + u < d4) pts[t * ld + k0 + u] = v[u] * in;
  }
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int e = t + u * kProbePoints, r = e / d4, k = e - r * d4;
    if (r < kSeedsPer) seeds[r * ld + k] = sv[u] * in;
  }
  __syncthreads();
  if (a.unit) {
    for (int r = t; r < kProbePoints + kSeedsPer; r += blockDim.x) {
      float nn = 0.0f;
      for (int k = 0; k < a.d; ++k) nn += pts[r * ld + k] * pts[r * ld + k];
      const float f = scale / sqrtf(nn);
      for (int k = 0; k < a.d; ++k) pts[r * ld + k] *= f;
    }
    __syncthreads();
  }
  if (t == 0) median = INFINITY;   // (rows that are not finite have none)
  // squared distances of the block's rows (its share of the points, then its seeds) to
  // point t, four rows at a time
  float e2[kSeedsPer];
#pragma unroll
  for (int g = 0; g < kRowsPer; g += 4) {
    const float* row = g < kNear ? pts + (rank * kNear + g) * ld : seeds + (g - kNear) * ld;
    float q[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int k = 0; k < d4; k += 4) {
      const float4 x = *reinterpret_cast<const float4*>(pts + t * ld + k);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 y = *reinterpret_cast<const float4*>(row + u * ld + k);
        float e = x.x - y.x;
        q[u] = fmaf(e, e, q[u]);
        e = x.y - y.y;
        q[u] = fmaf(e, e, q[u]);
        e = x.z - y.z;
        q[u] = fmaf(e, e, q[u]);
        e = x.w - y.w;
        q[u] = fmaf(e, e, q[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      float v = q[u];
      if (g < kNear) {
        if (t == rank * kNear + g + u) v = INFINITY;
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) v = fminf(v, __shfl_xor_sync(kFull, v, o));
      } else {
        e2[g - kNear + u] = v;
        v = ex2_ftz(-v);
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
      }
      if (lane == 0) red[g + u][w] = v;
    }
  }
  __syncthreads();
  if (t < kNear) {
    float v = red[t][0];
    for (int u = 1; u < kProbePoints / 32; ++u) v = fminf(v, red[t][u]);
    *cl.map_shared_rank(&near[rank * kNear + t], 0) = v;
  }
  cl.sync();
  if (rank == 0) {   // the median of the distances to the nearest other point
    const float v = near[t];
    int below = 0;
#pragma unroll 4
    for (int u = 0; u < kProbePoints; u += 4) {
      const float4 o = *reinterpret_cast<const float4*>(near + u);
      below += (o.x < v || (o.x == v && u < t) ? 1 : 0) + (o.y < v || (o.y == v && u + 1 < t) ? 1 : 0) +
               (o.z < v || (o.z == v && u + 2 < t) ? 1 : 0) + (o.w < v || (o.w == v && u + 3 < t) ? 1 : 0);
    }
    if (below == kProbePoints / 2) {
      for (int c = 0; c < kBlocks; ++c) *cl.map_shared_rank(&median, c) = v;
    }
  }
  cl.sync();
  const float M = sqrtf(median);
  const float log2n = log2f((float)s.n);
  int vis = 0;
#pragma unroll
  for (int q = 0; q < kSeedsPer; ++q) {
    float W = 0.0f;
    for (int u = 0; u < kProbePoints / 32; ++u) W += red[kNear + q][u];
    W = fmaxf(W * ((float)s.n / kProbePoints), 1.0f);
    const float at = sqrtf(fmaxf(e2[q] - 0.5f * M * M, 0.0f));
    float lim;
    if (a.kind == kProbeTile) {
      lim = sqrtf(cells::zero_bits<float>()) + 2.0f * M;
    } else {
      lim = M;
      if (a.kind == kProbeExtent)   // 3.5 deviations towards the seed, and the angle's part
        lim = fminf(M, 2.475f * M * rsqrtf((float)a.d) + 0.5f * M * M / fmaxf(at, 1e-9f));
      lim += sqrtf(fmaxf(cells::guard_bits<float>() + log2n - log2f(W), 1.0f));
    }
    vis += at <= lim ? 1 : 0;
  }
  vis = block_sum(vis, sum);
  if (t == 0) *cl.map_shared_rank(&seen[rank], 0) = vis;
  cl.sync();
  if (rank == 0 && t == 0) {
    int v = 0;
    for (int c = 0; c < kBlocks; ++c) v += seen[c];
    const float share = (float)v / (kProbePoints * kProbeSeeds);
    a.share[b] = share;
    if (a.walk) a.walk[b] = share <= kWalkShare ? 1 : 0;
  }
}

}  // namespace

template <typename T>
cudaError_t launch_probe(const ProbeArgs& a, cudaStream_t st) {
  if (a.sets < 1 || a.sets > kProbeSets || a.d > 64) return cudaErrorInvalidValue;
  const int bytes = (kProbePoints + kSeedsPer) * (((a.d + 3) & ~3) + 4) * 4;   // 72 KB at d = 64
  if (bytes > 40 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(
        probe_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 80 * 1024);
    if (e != cudaSuccess) return e;
  }
  probe_kernel<T><<<kBlocks * a.sets, kProbePoints, bytes, st>>>(a);
  return cudaGetLastError();
}
template cudaError_t launch_probe<float>(const ProbeArgs&, cudaStream_t);
template cudaError_t launch_probe<double>(const ProbeArgs&, cudaStream_t);

}  // namespace fms

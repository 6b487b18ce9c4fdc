// The probe of fms_route.cuh: one block a sampled set.
//
// A cell's radius is about the distance M from a sampled point to the nearest other one
// (half of the cells start from as many strided points); a cell whose centre lies at
// distance a from a seed is seen within the cutoff and the cell's reach.  From a sampled
// point x of the cell, a^2 = |x - y|^2 - M^2 / 2 (x is M / sqrt 2 from the centre, at right
// angles to y - centre where there are many dimensions).  The cutoff follows from the
// sample's weights, as the walk takes it from W.  A set of more clusters than points in the
// sample has a large M and comes out as one without clusters.
//
// One SM, bound by its shared memory (five 16-byte loads for 16 squared differences) and
// latency.  (Eight blocks in a cluster took 14 to 21 us, barriers and remote writes.)
#include "fms_cells.cuh"
#include "fms_route.cuh"

namespace fms {
namespace {

constexpr int kNear = 16;                           // points whose nearest other one is found
constexpr int kLoaded = kProbePoints + kProbeSeeds;
constexpr int kRows = kNear + kProbeSeeds;          // compared with all points
constexpr int kSplit = 1024 / kProbePoints;         // threads of a point
constexpr int kMine = kRows / kSplit;               // rows of a thread
constexpr int kWarps = kProbePoints / 32;           // warps of a part
static_assert(kRows % (4 * kSplit) == 0, "rows of a thread");

__device__ __forceinline__ int64_t strided(int i, int of, int64_t n) {
  return ((2 * (int64_t)i + 1) * n) / (2 * (int64_t)of);
}

template <typename T>
__global__ void __launch_bounds__(1024) probe_kernel(ProbeArgs a) {
  extern __shared__ __align__(16) float probe_smem[];
  const int d4 = (a.d + 3) & ~3, ld = d4 + 4;   // (16 bytes between rows: few conflicts)
  float* rows = probe_smem;                     // [kLoaded][ld]: the points, then the seeds
  __shared__ float red[kRows][kWarps];          // a row's parts: least distance or weights
  __shared__ float median;
  __shared__ int sum[32];
  const ProbeSet s = a.set[blockIdx.x];
  const T *X = static_cast<const T*>(s.X), *Y = static_cast<const T*>(s.Y);
  const int lane = threadIdx.x & 31;
  const float in = a.unit ? 1.0f : (float)a.scale;
  // rows over groups of 8 threads, four values of a thread in flight
  for (int r = threadIdx.x / 8; r < kLoaded; r += 128) {
    const T* x = r < kProbePoints ? X + strided(r, kProbePoints, s.n) * a.ld
                                  : Y + strided(r - kProbePoints, kProbeSeeds, s.m) * a.ld;
    for (int k0 = threadIdx.x % 8; k0 < d4; k0 += 32) {
      float v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = k0 + 8 * u < a.d ? (float)x[k0 + 8 * u] : 0.0f;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k0 + 8 * u < d4) rows[r * ld + k0 + 8 * u] = v[u] * in;
    }
  }
  if (threadIdx.x == 0) median = INFINITY;   // (rows that are not finite have none)
  __syncthreads();
  if (a.unit) {
    for (int r = threadIdx.x; r < kLoaded; r += blockDim.x) {
      float nn = 0.0f;
      for (int k = 0; k < a.d; ++k) nn += rows[r * ld + k] * rows[r * ld + k];
      const float f = (float)a.scale / sqrtf(nn);
      for (int k = 0; k < a.d; ++k) rows[r * ld + k] *= f;
    }
    __syncthreads();
  }
  // squared distances from point t to the thread's rows (every fourth point, then the
  // seeds), four at a time
  constexpr int kEvery = kProbePoints / kNear;
  const int t = threadIdx.x % kProbePoints, part = threadIdx.x / kProbePoints, w = t >> 5;
  float q[kMine];
#pragma unroll
  for (int g = 0; g < kMine; g += 4) {
    const int r0 = part * kMine + g, stride = r0 < kNear ? kEvery * ld : ld;
    const float* row = rows + (r0 < kNear ? r0 * kEvery : kProbePoints + r0 - kNear) * ld;
    float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 2
    for (int k = 0; k < d4; k += 4) {
      const float4 x = *reinterpret_cast<const float4*>(rows + t * ld + k);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 y = *reinterpret_cast<const float4*>(row + u * stride + k);
        float e = x.x - y.x;
        c[u] = fmaf(e, e, c[u]);
        e = x.y - y.y;
        c[u] = fmaf(e, e, c[u]);
        e = x.z - y.z;
        c[u] = fmaf(e, e, c[u]);
        e = x.w - y.w;
        c[u] = fmaf(e, e, c[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = part * kMine + g + u;
      q[g + u] = c[u];
      float v = r < kNear ? (r * kEvery == t ? INFINITY : c[u]) : ex2_ftz(-c[u]);
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) {
        const float z = __shfl_xor_sync(kFull, v, o);
        v = r < kNear ? fminf(v, z) : v + z;
      }
      if (lane == 0) red[r][w] = v;
    }
  }
  __syncthreads();
  if (threadIdx.x < 32) {   // the median of the distances to the nearest point
    float v = red[lane % kNear][0];
    for (int u = 1; u < kWarps; ++u) v = fminf(v, red[lane % kNear][u]);
    int below = 0;
    for (int u = 0; u < kNear; ++u) {
      const float o = __shfl_sync(kFull, v, u);
      below += o < v || (o == v && u < lane) ? 1 : 0;
    }
    if (lane < kNear && below == kNear / 2) median = v;
  }
  __syncthreads();
  const float M = sqrtf(median), log2n = log2f((float)s.n);
  int vis = 0;
#pragma unroll
  for (int g = 0; g < kMine; ++g) {
    const int r = part * kMine + g;
    if (r < kNear) continue;
    float W = 0.0f;
    for (int u = 0; u < kWarps; ++u) W += red[r][u];
    W = fmaxf(W * ((float)s.n / kProbePoints), 1.0f);
    const float at = sqrtf(fmaxf(q[g] - 0.5f * M * M, 0.0f));
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
  if (threadIdx.x == 0) {
    const float share = (float)vis / (kProbePoints * kProbeSeeds);
    a.share[blockIdx.x] = share;
    if (a.walk) a.walk[blockIdx.x] = share <= a.limit ? 1 : 0;
  }
}

}  // namespace

template <typename T>
cudaError_t launch_probe(const ProbeArgs& a, cudaStream_t st) {
  if (a.sets < 1 || a.sets > kProbeSets || a.d > 64) return cudaErrorInvalidValue;
  const int bytes = kLoaded * (((a.d + 3) & ~3) + 4) * 4;   // 43.5 KB at d = 64
  probe_kernel<T><<<a.sets, 1024, bytes, st>>>(a);
  return cudaGetLastError();
}
template cudaError_t launch_probe<float>(const ProbeArgs&, cudaStream_t);
template cudaError_t launch_probe<double>(const ProbeArgs&, cudaStream_t);

}  // namespace fms

// A group of 32 seeds (one per lane) and the team of warps that splits its
// visible tiles: row loads, shared memory, sums over the team.
#pragma once

#include "fms_cells.cuh"

namespace fms {

using cells::Groups;
using cells::View;

template <int DPAD>
__device__ __forceinline__ void load_row(const float* __restrict__ p, float (&v)[DPAD]) {
#pragma unroll
  for (int q = 0; q < DPAD / 4; ++q) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(p) + q);
    v[4 * q] = t.x;
    v[4 * q + 1] = t.y;
    v[4 * q + 2] = t.z;
    v[4 * q + 3] = t.w;
  }
}

template <int DPAD>
__device__ __forceinline__ void load_row(const double* __restrict__ p, double (&v)[DPAD]) {
#pragma unroll
  for (int q = 0; q < DPAD / 2; ++q) {
    const double2 t = __ldg(reinterpret_cast<const double2*>(p) + q);
    v[2 * q] = t.x;
    v[2 * q + 1] = t.y;
  }
}

// a row already in shared memory: plain vector loads
template <int DPAD>
__device__ __forceinline__ void smem_row(const float* p, float (&v)[DPAD]) {
#pragma unroll
  for (int q = 0; q < DPAD / 4; ++q) {
    const float4 t = reinterpret_cast<const float4*>(p)[q];
    v[4 * q] = t.x;
    v[4 * q + 1] = t.y;
    v[4 * q + 2] = t.z;
    v[4 * q + 3] = t.w;
  }
}
template <int DPAD>
__device__ __forceinline__ void smem_row(const double* p, double (&v)[DPAD]) {
#pragma unroll
  for (int q = 0; q < DPAD / 2; ++q) {
    const double2 t = reinterpret_cast<const double2*>(p)[q];
    v[2 * q] = t.x;
    v[2 * q + 1] = t.y;
  }
}

template <typename T, int DP>
__device__ __forceinline__ void store_row(T* p, const T (&v)[DP]) {
  constexpr int E = 16 / (int)sizeof(T);
#pragma unroll
  for (int q = 0; q < DP / E; ++q) {
    float4 t;
    T* u = reinterpret_cast<T*>(&t);
#pragma unroll
    for (int e = 0; e < E; ++e) u[e] = v[q * E + e];
    reinterpret_cast<float4*>(p)[q] = t;
  }
}

// the element type's exp2, fma and min (FP32: the MUFU exp2 with flush to zero)
__device__ __forceinline__ float uex2(float x) { return ex2_ftz(x); }
__device__ __forceinline__ double uex2(double x) { return exp2(x); }
__device__ __forceinline__ float ufma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double ufma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float umin(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ double umin(double a, double b) { return fmin(a, b); }

// Shared memory of a team of W warps: each warp's tile ring and its share of the
// sums exchanged at the end of a pass; for the groups of seeds (GROUP) one list of
// row ranges and the group's rows, else a list for each warp.
constexpr int kListCap = cells::kMaxCells;

template <typename T, int DP>
struct GroupSmem {
  T row[32][DP];          // the active seeds
  T rc[32], delta[32];    // their cutoff radius and distance to the nearest centre
  unsigned mask[kListCap / 32], near[16];
};

template <typename T, int ROW, int SUMS>
constexpr int team_warp_smem() {
  return 2 * cells::kTileRows * ROW * (int)sizeof(T) + SUMS * 32 * (int)sizeof(T);
}
template <typename T, int DP, int SUMS>   // a team that walks cells
constexpr int group_team_smem(int W) {
  return W * team_warp_smem<T, DP, SUMS>() + SUMS * 32 * (int)sizeof(T) + kListCap * 8 +
         (int)sizeof(GroupSmem<T, DP>);
}
// Few unsorted points are kept in shared memory by every team for all its updates,
// in the place of the rings: an update of 1,500 points by 16 warps is three tiles a
// warp, whose copies from L2 it would wait for.
constexpr int kResidentBytes = 48 * 1024;
template <typename T, int DP>
inline bool team_resident(int P, int64_t n) {
  return P == 0 && n * DP * (int64_t)sizeof(T) <= kResidentBytes;
}
template <typename T, int DP, int SUMS>
inline int resident_team_smem(int W, int64_t n) {
  return (int)(n * DP * sizeof(T)) + (W + 1) * SUMS * 32 * (int)sizeof(T) + kListCap * 8 +
         (int)sizeof(GroupSmem<T, DP>);
}
template <typename T, int ROW, int SUMS>   // a team with a list per warp
constexpr int list_team_smem(int W) {
  return W * (team_warp_smem<T, ROW, SUMS>() + kListCap * 8) + SUMS * 32 * (int)sizeof(T);
}

template <typename T, int ROW, int SUMS, bool GROUP = true>
struct TeamSmem {
  T* ring;      // this warp's two tiles
  int2* list;   // the team's list (GROUP), or this warp's
  T* sums;      // [W + 1][SUMS][32], the whole team's (the last: totals)
  GroupSmem<T, ROW>* group;
  T* all;       // every point (few unsorted ones), else null
  // n_all > 0: the points at `rows` are resident (copied here; ends with a barrier)
  __device__ TeamSmem(unsigned char* base, int w, int W, const T* rows = nullptr, int n_all = 0) {
    constexpr int ring_e = 2 * cells::kTileRows * ROW;
    ring = reinterpret_cast<T*>(base) + (n_all > 0 ? 0 : (size_t)w * ring_e);
    all = n_all > 0 ? ring : nullptr;
    unsigned char* p = base + (n_all > 0 ? (size_t)n_all * ROW : (size_t)W * ring_e) * sizeof(T);
    sums = reinterpret_cast<T*>(p);
    p += (size_t)(W + 1) * SUMS * 32 * sizeof(T);
    list = reinterpret_cast<int2*>(p) + (GROUP ? 0 : w * kListCap);
    group = reinterpret_cast<GroupSmem<T, ROW>*>(p + kListCap * 8);
    if (n_all > 0) {
      const int n16 = n_all * (ROW * (int)sizeof(T) / 16);
      for (int i = threadIdx.x; i < n16; i += blockDim.x)
        reinterpret_cast<float4*>(all)[i] = __ldg(reinterpret_cast<const float4*>(rows) + i);
      __syncthreads();
    }
  }
  // the team's tiles: of the listed cells of X, or of the resident points
  template <typename F>
  __device__ __forceinline__ void walk(const T* X, int n, int nl, int w, int W, int lane,
                                       F&& tile_fn) const {
    if (all) cells::walk_resident<ROW>(all, n, w, W, tile_fn);
    else cells::walk_tiles<ROW>(X, list, nl, w, W, ring, lane, tile_fn);
  }
};

// warps a block may have: 16 where the registers allow
template <typename T, int DP>
constexpr int most_warps() {
  return sizeof(T) == 4 && DP <= 8 ? 16 : 8;
}
// rows evaluated together (independent chains)
template <typename T, int DP>
constexpr int row_unroll() {
  return DP <= 4 ? 8 : (DP <= 8 ? 4 : 1);
}

// The team's list of the cells of set b that can hold a point within the distance
// rc of an active lane's seed y, as (first row, rows); returns its length.  First
// the ball around the active seeds against each cell's ball, then the cells left,
// one per lane, against every active seed: in many dimensions the ball around the
// seeds is as wide as their cluster, and only the second test keeps its neighbours
// out.  At least one lane is active; every thread of the team calls.  Without cells
// (P = 0) the list is every row, and *reach and *ball are not set.
template <typename T, int DP, int SUMS>
__device__ __forceinline__ int visible_cells(const View<T>& v, int b, int n, const T (&y)[DP],
                                             bool act, T rc, T* reach,
                                             T (*ball)[DP], const TeamSmem<T, DP, SUMS>& sm,
                                             int w, int W, int lane) {
  if (v.P == 0) {
    if (sm.all) return 0;   // (walk takes the resident points)
    if (threadIdx.x == 0) sm.list[0] = make_int2(0, n);
    __syncthreads();
    return 1;
  }
  const unsigned live = __ballot_sync(kFull, act);
  const int src = __ffs(live) - 1, nact = __popc(live);
  T c[DP];
  {
    T yb[DP];
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      const T u = __shfl_sync(kFull, y[k], src);
      yb[k] = act ? y[k] : u;
    }
    const T rho = cells::group_ball<T, DP>(yb, c);
    const T rc0 = __shfl_sync(kFull, rc, src);
    *reach = rho + cells::warp_max(act ? rc : rc0);
  }
  if (ball) {
#pragma unroll
    for (int k = 0; k < DP; ++k) (*ball)[k] = c[k];
  }
  GroupSmem<T, DP>& g = *sm.group;
  const int32_t* st = v.start + (int64_t)b * (v.P + 1);
  const int at = __popc(live & ((1u << lane) - 1u));
  if (w == 0 && act) {
    store_row<T, DP>(g.row[at], y);
    g.rc[at] = rc;
  }
  // the ball test, each warp its share of the cells, and the nearest cell
  unsigned best = 0xffffffffu;
  for (int i = w; i < v.P / 32; i += W) {
    const int p = i * 32 + lane;
    const T* z = v.ctr + ((int64_t)b * v.P + p) * DP;
    T x[DP], d2 = T(0);
    load_row<DP>(z, x);
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      const T f = x[k] - c[k];
      d2 += f * f;
    }
    // 1e-4 covers the rounding of the distances and of their sum
    const T lim = (*reach + v.rad[(int64_t)b * v.P + p]) * T(1.0001);
    const bool some = st[p + 1] > st[p];
    const unsigned m = __ballot_sync(kFull, some && !(d2 > lim * lim));
    if (lane == 0) g.mask[i] = m;
    if constexpr (sizeof(T) == 4)
      if (some) best = min(best, (__float_as_uint(d2) & ~255u) | (unsigned)p);
  }
  bool by_extent = false;
  if constexpr (sizeof(T) == 4) by_extent = v.ext != nullptr;
  if (by_extent) {
    best = __reduce_min_sync(kFull, best);
    if (lane == 0) g.near[w] = best;
  }
  __syncthreads();
  int q = 0;
  if constexpr (sizeof(T) == 4) {
    if (by_extent) {
      for (int u = 0; u < W; ++u) best = min(best, g.near[u]);
      q = (int)(best & 255u);
      if (w == 0 && act) {
        const float* z = v.ctr + (int64_t)q * DP;
        float s = 0.0f;
#pragma unroll
        for (int k = 0; k < DP; ++k) s += (z[k] - y[k]) * (z[k] - y[k]);
        g.delta[at] = sqrtf(s);
      }
      __syncthreads();
    }
  }
  // every seed against the cells that are left
  for (int i = w; i < v.P / 32; i += W) {
    const unsigned m = g.mask[i];
    if (!m) continue;
    const int p = i * 32 + lane;
    bool see = false;
    if ((m >> lane) & 1u) {
      T x[DP];
      load_row<DP>(v.ctr + ((int64_t)b * v.P + p) * DP, x);
      const T rad = v.rad[(int64_t)b * v.P + p];
      float2 ext = make_float2(0.f, 0.f);
      if (by_extent) ext = __ldg(v.ext + q * v.P + p);
      for (int u = 0; u < nact && !see; ++u) {
        T d2 = T(0), r[DP];
        smem_row<DP>(g.row[u], r);
#pragma unroll
        for (int k = 0; k < DP; ++k) d2 += (x[k] - r[k]) * (x[k] - r[k]);
        T far_ = rad;
        if constexpr (sizeof(T) == 4)
          if (by_extent) far_ = cells::reach_towards(rad, ext, sqrtf(d2), g.delta[u]);
        const T lim = (g.rc[u] + far_) * T(1.0001);
        see = !(d2 > lim * lim);
      }
    }
    const unsigned keep = __ballot_sync(kFull, see);
    __syncwarp();
    if (lane == 0) g.mask[i] = keep;
  }
  __syncthreads();
  int nl = 0;
  for (int i = 0; i < v.P / 32; ++i) {
    const unsigned m = g.mask[i];
    if (i % W == w && ((m >> lane) & 1u)) {
      const int a = st[i * 32 + lane];
      sm.list[nl + __popc(m & ((1u << lane) - 1u))] = make_int2(a, st[i * 32 + lane + 1] - a);
    }
    nl += __popc(m);
  }
  __syncthreads();
  return nl;
}

// PH > 1 (few seeds, nothing sorted): a group is 32 / PH seeds, lane l holds seed
// l % (32 / PH) and takes rows l / (32 / PH), + PH, ... of a tile, so PH times as many
// blocks share the work.  row_fn(row, inside) for each of the lane's rows; a row
// outside the tile repeats its last one and must count nothing.
template <int ROW, int PH, int UNROLL, typename T, typename F>
__device__ __forceinline__ void tile_rows(const T* rows, int nr, int lane, F&& row_fn) {
  if constexpr (PH == 1) {
#pragma unroll UNROLL
    for (int q = 0; q < nr; ++q) row_fn(rows + q * ROW, true);
  } else {
    const int ph = lane / (32 / PH);
    if (nr == cells::kTileRows) {
#pragma unroll UNROLL
      for (int q = 0; q < cells::kTileRows / PH; ++q) row_fn(rows + (q * PH + ph) * ROW, true);
    } else {
      for (int q = 0; q < nr; q += PH)
        row_fn(rows + min(q + ph, nr - 1) * ROW, q + ph < nr);
    }
  }
}
// ... and their sums over the PH lanes of a seed.
template <int PH, typename T, int N>
__device__ __forceinline__ void phase_sum(T (&v)[N]) {
#pragma unroll
  for (int k = 0; k < N; ++k)
#pragma unroll
    for (int o = 16; o >= 32 / PH && PH > 1; o >>= 1) v[k] += __shfl_xor_sync(kFull, v[k], o);
}
// PH for `seeds` seeds of all sets: enough groups for the GPU's SMs.
template <typename T, int DP>
inline int team_phases(int P, int64_t seeds, int sms) {
  if (P > 0 || sizeof(T) != 4 || DP > 16) return 1;
  return (seeds + 31) / 32 >= sms ? 1 : 4;
}

// Sums over the team in warp order; every warp gets the result.  Lanes l and
// l + GS hold the same values; a thread adds one value's W parts (every warp adding
// all of them would read W^2 rows of shared memory).  The values are already in the
// warps' parts of `sums`:
template <int GS, typename T, int N>
__device__ __forceinline__ void team_total(T (&v)[N], T* sums, int stride, int W, int lane) {
  T* total = sums + W * stride * 32;
  __syncthreads();
  for (int i = threadIdx.x; i < N * GS; i += 32 * W) {
    const int at = i / GS * 32 + i % GS;
    T s = sums[at];
    for (int u = 1; u < W; ++u) s += sums[u * stride * 32 + at];
    total[at] = s;
  }
  __syncthreads();
  // (rewritten only after the next call's first barrier)
#pragma unroll
  for (int k = 0; k < N; ++k) v[k] = total[k * 32 + lane % GS];
}

// ... or in v:
template <int GS, typename T, int N>
__device__ __forceinline__ void team_sum(T (&v)[N], T* sums, int stride, int w, int W, int lane) {
  if (W == 1) return;
  if (lane < GS) {
#pragma unroll
    for (int k = 0; k < N; ++k) sums[(w * stride + k) * 32 + lane] = v[k];
  }
  team_total<GS>(v, sums, stride, W, lane);
}

__device__ __forceinline__ bool group_rows(const Groups& g, int b, int gi, int rows, int* row0,
                                           int* cnt, int size = 32) {
  if (g.table) {
    const int2 e = __ldg(g.table + (int64_t)b * g.per_set + gi);
    *row0 = e.x;
    *cnt = e.y;
  } else {
    *row0 = gi * size;
    *cnt = min(size, rows - gi * size);
  }
  return *cnt > 0;
}


// Warps of a team: enough of them for about 32 warps per SM over all groups, as
// many as shared memory holds.
inline int team_warps(int64_t groups, int sms, int warp_smem, int most = 8) {
  int W = 1;
  while (W < most && groups * W < (int64_t)sms * 32 && 2 * W * warp_smem <= 200 * 1024) W *= 2;
  return W;
}

// Lets a kernel use the device's 227 KB of shared memory a block, less kTeamStatic for
// its static arrays: one limit for every launch of the kernel, whatever its size, since
// the attribute belongs to the kernel (another thread's launch may come in between).
// The default of 48 KB counts the static arrays as well.
constexpr int kTeamStatic = 256;
template <typename K>
inline cudaError_t team_attr(K kernel, int bytes) {
  if (bytes + kTeamStatic <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              227 * 1024 - kTeamStatic);
}

}  // namespace fms

// Sorting of rows into cells (fms_cells.cuh): nearest pivot, then a stable
// counting sort over blocks of kChunkRows rows.  Every step gives the same
// result on each run (maxima, counts and ranks only).
#include "fms_cells.cuh"

namespace fms {
namespace cells {

// First row and rows of set b: offs [B + 1] or, null, sets of `each` rows.
__device__ __forceinline__ int64_t set_rows(const int64_t* __restrict__ offs, int b, int64_t each,
                                            int* n) {
  if (!offs) {
    *n = (int)each;
    return (int64_t)b * each;
  }
  const int64_t o = offs[b];
  *n = (int)(offs[b + 1] - o);
  return o;
}

// Blocks run over (set, run of R rows): `per` runs to a set of `each` rows, or set_of_run.
template <int R>
__device__ __forceinline__ int block_set(const int64_t* __restrict__ offs, int B, int per,
                                         int* run) {
  if (offs) return set_of_run<R>(offs, B, blockIdx.x, run);
  *run = blockIdx.x % per;
  return blockIdx.x / per;
}

// The counters of set b's first chunk of kChunkRows rows are row chunk0 of counts
// [chunks][P].
__device__ __forceinline__ int64_t chunk0(const int64_t* __restrict__ offs, int b, int per) {
  return offs ? offs[b] / kChunkRows + b : (int64_t)b * per;
}

// Row of pivot p: the middle of the p-th of P equal runs of the set's rows.
__device__ __forceinline__ int64_t pivot_row(int p, int P, int64_t n) {
  return ((2 * (int64_t)p + 1) * n) / (2 * (int64_t)P);
}

// Loads pivot rows p0 .. p1 of a set (strided rows) into shared memory.
template <typename T, int DP>
__device__ __forceinline__ void load_pivots(const T* __restrict__ set, int64_t n, int P, T* pv) {
  for (int e = threadIdx.x; e < P * DP; e += blockDim.x)
    pv[e] = set[pivot_row(e / DP, P, n) * DP + e % DP];
}

// Nearest of the pivots [p0, p1) in shared memory for two rows at a time (ties: the
// lower pivot); b0, b1, i0, i1 carry the best so far.  Half the squared distance
// less the row's own part, |c|^2 / 2 - x.c, decides (half[p] = |c_p|^2 / 2; any
// choice is a valid cell), which is DP multiply-adds a pair against the 2 DP of the
// differences.  Bound by FP32 issue and the pivots' broadcast loads.
template <typename T, int DP>
__device__ __forceinline__ void nearest(const T (&x0)[DP], const T (&x1)[DP], const T* pv,
                                        const T* half, int p0, int p1, T& b0, T& b1, int& i0,
                                        int& i1) {
#pragma unroll 2
  for (int p = p0; p < p1; ++p) {
    T d0 = half[p], d1 = d0;
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      const T q = pv[p * DP + k];
      d0 -= x0[k] * q;
      d1 -= x1[k] * q;
    }
    if (p == 0 || d0 < b0) {
      b0 = d0;
      i0 = p;
    }
    if (p == 0 || d1 < b1) {
      b1 = d1;
      i1 = p;
    }
  }
}

// Moves the n pivots to the first one as origin (kept in org: products of coordinates
// far from zero would cancel) and sets half[p] = |c_p|^2 / 2.  Ends with a barrier.
template <typename T, int DP>
__device__ __forceinline__ void center_pivots(T* pv, T* org, T* half, int n) {
  for (int k = threadIdx.x; k < DP; k += blockDim.x) org[k] = pv[k];
  __syncthreads();
  for (int p = threadIdx.x; p < n; p += blockDim.x) {
    T s = T(0);
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      const T v = pv[p * DP + k] - org[k];
      pv[p * DP + k] = v;
      s += v * v;
    }
    half[p] = T(0.5) * s;
  }
  __syncthreads();
}

template <typename T, int DP>
__device__ __forceinline__ void row_values(const T* p, T (&x)[DP]) {
#pragma unroll
  for (int q = 0; q < DP * (int)sizeof(T) / 16; ++q) {
    const float4 t = reinterpret_cast<const float4*>(p)[q];
    const T* u = reinterpret_cast<const T*>(&t);
#pragma unroll
    for (int e = 0; e < 16 / (int)sizeof(T); ++e) x[q * (16 / (int)sizeof(T)) + e] = u[e];
  }
}

// First pass over the points: the nearest of the P0 strided pivots, and each
// pivot's farthest row as (squared distance bits, row).
// two rows a thread at a time (wide rows: fewer threads, for their registers)
template <typename T, int DP>
constexpr int assign_threads() {
  return DP * sizeof(T) > 128 ? kChunkRows / 4 : kChunkRows / 2;
}

constexpr int kPivotRows = 512;   // (smaller blocks: 200,000 rows over 152 SMs leave less idle)

template <typename T, int DP>
__global__ void __launch_bounds__(256)
    pivot_kernel(const T* __restrict__ src, const int64_t* __restrict__ offs, int B, int each,
                 int P0, int per, unsigned char* __restrict__ id,
                 unsigned long long* __restrict__ far_, Gate gate) {
  wait_for_previous();
  if (!gate.open()) return;
  extern __shared__ __align__(16) unsigned char cell_smem[];
  __shared__ T org[DP];
  T* pv = reinterpret_cast<T*>(cell_smem);                                        // [P0][DP]
  T* half = pv + P0 * DP;                                                         // [P0]
  unsigned long long* fs = reinterpret_cast<unsigned long long*>(half + P0);      // [P0]
  int blk, nrows;
  const int b = block_set<kPivotRows>(offs, B, per, &blk);
  const int64_t row0 = set_rows(offs, b, each, &nrows);
  if ((int64_t)blk * kPivotRows >= nrows) return;
  const T* set = src + row0 * DP;
  load_pivots<T, DP>(set, nrows, P0, pv);
  for (int p = threadIdx.x; p < P0; p += blockDim.x) fs[p] = 0ull;
  __syncthreads();
  center_pivots<T, DP>(pv, org, half, P0);
  const int r_end = min((int64_t)nrows, ((int64_t)blk + 1) * kPivotRows);
  for (int r0 = blk * kPivotRows + threadIdx.x; r0 < r_end; r0 += 2 * blockDim.x) {
    const int r1 = r0 + (int)blockDim.x < r_end ? r0 + (int)blockDim.x : r0;
    T x0[DP], x1[DP], b0 = T(0), b1 = T(0);
    row_values<T, DP>(set + (int64_t)r0 * DP, x0);
    row_values<T, DP>(set + (int64_t)r1 * DP, x1);
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      x0[k] -= org[k];
      x1[k] -= org[k];
    }
    int i0 = 0, i1 = 0;
    nearest<T, DP>(x0, x1, pv, half, 0, P0, b0, b1, i0, i1);
    b0 = b1 = T(0);
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      const T e0 = x0[k] - pv[i0 * DP + k], e1 = x1[k] - pv[i1 * DP + k];
      b0 += e0 * e0;
      b1 += e1 * e1;
    }
    id[row0 + r0] = (unsigned char)i0;
    id[row0 + r1] = (unsigned char)i1;
    auto key = [](T v, int r) {
      return ((unsigned long long)(__float_as_uint((float)v) & 0x7fffffffu) << 32) | (unsigned)r;
    };
    const unsigned long long k0 = key(b0, r0), k1 = key(b1, r1);
    if (fs[i0] < k0) atomicMax(&fs[i0], k0);
    if (fs[i1] < k1) atomicMax(&fs[i1], k1);
  }
  __syncthreads();
  for (int p = threadIdx.x; p < P0; p += blockDim.x)
    if (fs[p]) atomicMax(&far_[(int64_t)b * P0 + p], fs[p]);
}

// The pivots of a set (one block): the P0 strided ones, then the farthest row of
// every cell whose radius is over twice the lowest eighth's (a cluster that no
// strided pivot hit hangs on to cells of other ones and would make their balls span
// both; in many dimensions a few such clusters reach most cells, hence not the
// median).  Writes them to ctr and their number to npiv.
template <typename T, int DP>
__global__ void __launch_bounds__(kMaxCells)
    select_kernel(const T* __restrict__ src, const int64_t* __restrict__ offs, int each, int P,
                  const unsigned long long* __restrict__ far_, T* __restrict__ ctr,
                  int32_t* __restrict__ npiv, Gate gate) {
  wait_for_previous();
  if (!gate.open()) return;
  __shared__ float r2s[kMaxCells / 2];
  __shared__ float small;
  __shared__ int sel[kMaxCells], red[64];
  const int b = blockIdx.x, P0 = P / 2, p = threadIdx.x;
  int nrows;
  const T* set = src + set_rows(offs, b, each, &nrows) * DP;
  unsigned long long k = 0;
  float r2 = 0.0f;
  if (p < P0) {
    k = far_[(int64_t)b * P0 + p];
    r2 = __uint_as_float((unsigned)(k >> 32));
    r2s[p] = r2;
    sel[p] = (int)pivot_row(p, P0, nrows);
  }
  if (p == 0) small = INFINITY;
  __syncthreads();
  if (p < P0) {
    int rank = 0;
    for (int q = 0; q < P0; ++q) rank += (r2s[q] < r2 || (r2s[q] == r2 && q < p)) ? 1 : 0;
    if (rank == P0 / 8) small = r2;
  }
  __syncthreads();
  const int take = p < P0 && r2 > 4.0f * small ? 1 : 0;
  int K = 0;
  const int at = block_exclusive_scan(take, &K, red);
  if (take) sel[P0 + at] = (int)(unsigned)k;
  __syncthreads();
  T* out = ctr + (int64_t)b * P * DP;
  for (int e = threadIdx.x; e < P * DP; e += blockDim.x)   // (the rest: empty cells)
    out[e] = e < (P0 + K) * DP ? set[(int64_t)sel[e / DP] * DP + e % DP] : T(0);
  if (p == 0) npiv[b] = P0 + K;
}

// The cell of every row, and the rows of every (block, cell) in counts [chunks][P].
// EXTEND (the points): id holds the nearest strided pivot and only the added ones are
// tried; else (the seeds) all of them.
template <typename T, int DP, bool EXTEND>
__global__ void __launch_bounds__(assign_threads<T, DP>())
    assign_kernel(const T* __restrict__ src, const int64_t* __restrict__ offs, int B, int each,
                  int per, int P, unsigned char* __restrict__ id,
                  int32_t* __restrict__ counts, const T* __restrict__ ctr,
                  const int32_t* __restrict__ npiv, Gate gate) {
  wait_for_previous();
  if (!gate.open()) return;
  extern __shared__ __align__(16) unsigned char cell_smem[];
  __shared__ T org[DP];
  T* pv = reinterpret_cast<T*>(cell_smem);                 // [P][DP]
  T* half = pv + (size_t)P * DP;                           // [P]
  int* hist = reinterpret_cast<int*>(half + P);            // [P]
  const int P0 = P / 2;
  int blk, nrows;
  const int b = block_set<kChunkRows>(offs, B, per, &blk);
  const int64_t row0 = set_rows(offs, b, each, &nrows);
  if ((int64_t)blk * kChunkRows >= nrows) return;
  const T* set = src + row0 * DP;
  for (int p = threadIdx.x; p < P; p += blockDim.x) hist[p] = 0;
  const int np = npiv[b];
  for (int e = threadIdx.x; e < np * DP; e += blockDim.x) pv[e] = ctr[(int64_t)b * P * DP + e];
  __syncthreads();
  center_pivots<T, DP>(pv, org, half, np);
  const int r_end = min((int64_t)nrows, ((int64_t)blk + 1) * kChunkRows);
  for (int r0 = blk * kChunkRows + threadIdx.x; r0 < r_end; r0 += 2 * blockDim.x) {
    const int r1 = r0 + (int)blockDim.x < r_end ? r0 + (int)blockDim.x : r0;
    T x0[DP], x1[DP], b0 = T(0), b1 = T(0);
    row_values<T, DP>(set + (int64_t)r0 * DP, x0);
    row_values<T, DP>(set + (int64_t)r1 * DP, x1);
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      x0[k] -= org[k];
      x1[k] -= org[k];
    }
    int i0 = 0, i1 = 0;
    if (EXTEND) {
      i0 = id[row0 + r0];
      i1 = id[row0 + r1];
      b0 = half[i0];
      b1 = half[i1];
#pragma unroll
      for (int k = 0; k < DP; ++k) {
        b0 -= x0[k] * pv[i0 * DP + k];
        b1 -= x1[k] * pv[i1 * DP + k];
      }
      nearest<T, DP>(x0, x1, pv, half, P0, np, b0, b1, i0, i1);
    } else {
      nearest<T, DP>(x0, x1, pv, half, 0, np, b0, b1, i0, i1);
    }
    id[row0 + r0] = (unsigned char)i0;
    atomicAdd(&hist[i0], 1);
    if (r1 != r0) {
      id[row0 + r1] = (unsigned char)i1;
      atomicAdd(&hist[i1], 1);
    }
  }
  __syncthreads();
  int32_t* out = counts + (chunk0(offs, b, per) + blk) * P;
  for (int p = threadIdx.x; p < P; p += blockDim.x) out[p] = hist[p];
}

// Mean and radius of every cell (one block each): its rows are contiguous by now.
constexpr int kBoundWarps = 8;

template <typename T, int DP>
__global__ void __launch_bounds__(32 * kBoundWarps)
    bound_kernel(const T* __restrict__ rows, const int64_t* __restrict__ offs, int each, int P,
                 const int32_t* __restrict__ start, T* __restrict__ ctr, T* __restrict__ rad,
                 Gate gate) {
  wait_for_previous();
  if (!gate.open()) return;
  __shared__ T red[kBoundWarps][DP];
  __shared__ T mean[DP];
  const int b = blockIdx.x / P, p = blockIdx.x % P, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int a = start[(int64_t)b * (P + 1) + p], e = start[(int64_t)b * (P + 1) + p + 1];
  if (e <= a) {
    if (threadIdx.x == 0) rad[(int64_t)b * P + p] = T(0);
    return;
  }
  int nrows;
  const T* set = rows + set_rows(offs, b, each, &nrows) * DP;
  T s[DP];
#pragma unroll
  for (int k = 0; k < DP; ++k) s[k] = T(0);
  for (int r = a + threadIdx.x; r < e; r += blockDim.x) {
    T x[DP];
    row_values<T, DP>(set + (int64_t)r * DP, x);
#pragma unroll
    for (int k = 0; k < DP; ++k) s[k] += x[k];
  }
#pragma unroll
  for (int k = 0; k < DP; ++k) {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) s[k] += __shfl_xor_sync(kFull, s[k], o);
    if (lane == 0) red[w][k] = s[k];
  }
  __syncthreads();
  for (int k = threadIdx.x; k < DP; k += blockDim.x) {
    T v = red[0][k];
    for (int u = 1; u < kBoundWarps; ++u) v += red[u][k];
    v /= T(e - a);
    mean[k] = v;
    ctr[((int64_t)b * P + p) * DP + k] = v;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < DP; ++k) s[k] = mean[k];
  T far_ = T(0);
  for (int r = a + threadIdx.x; r < e; r += blockDim.x) {
    T x[DP], d2 = T(0);
    row_values<T, DP>(set + (int64_t)r * DP, x);
#pragma unroll
    for (int k = 0; k < DP; ++k) d2 += (x[k] - s[k]) * (x[k] - s[k]);
    far_ = (d2 > far_ || !(d2 == d2)) ? d2 : far_;   // NaN wins
  }
  far_ = warp_max(far_);
  __syncthreads();
  if (lane == 0) red[w][0] = far_;
  __syncthreads();
  if (w == 0) {
    far_ = warp_max(red[lane % kBoundWarps][0]);
    if (lane == 0) rad[(int64_t)b * P + p] = csqrt(far_);
  }
}

// From kScanChunks chunks a set on, one pass turns the counters of a set's chunks into
// those of the chunks before, and keeps the cells' totals: 32 cells a block, a lane each,
// every warp a run of chunks.  (Every block of the scatter adding up all of them grows
// with the square of n: 10^7 rows of d = 9 took 7.5 ms more.)
__global__ void __launch_bounds__(1024)
    scan_kernel(const int64_t* __restrict__ offs, int each, int per, int P,
                int32_t* __restrict__ counts, int32_t* __restrict__ cell_rows, Gate gate) {
  wait_for_previous();
  if (!gate.open()) return;
  __shared__ int part[32][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int b = blockIdx.x / (P / 32), p = blockIdx.x % (P / 32) * 32 + lane;
  int nrows;
  set_rows(offs, b, each, &nrows);
  const int nblk = (int)(((int64_t)nrows + kChunkRows - 1) / kChunkRows);
  const int run = (nblk + 31) / 32, q0 = min(nblk, w * run), q1 = min(nblk, q0 + run);
  int32_t* c = counts + chunk0(offs, b, per) * P + p;
  int s = 0;
#pragma unroll 8
  for (int q = q0; q < q1; ++q) s += c[(int64_t)q * P];
  part[w][lane] = s;
  __syncthreads();
  int at = 0, all = 0;
  for (int u = 0; u < 32; ++u) {
    const int v = part[u][lane];
    if (u < w) at += v;
    all += v;
  }
  if (w == 0) cell_rows[(int64_t)b * P + p] = all;
#pragma unroll 8
  for (int q = q0; q < q1; ++q) {
    const int v = c[(int64_t)q * P];
    c[(int64_t)q * P] = at;
    at += v;
  }
}

// Each block finds where its rows of every cell go (rows of earlier cells, then of the
// same cell in earlier blocks), ranks its rows in order warp by warp, and copies them.
// Latency bound; without the scan (cell_rows null) every block reads blocks x P counters
// from L2.
template <typename T, int DP>
__global__ void __launch_bounds__(256)
    scatter_kernel(const T* __restrict__ src, const int64_t* __restrict__ offs, int B, int each,
                   int per, int P, const unsigned char* __restrict__ id,
                   const int32_t* __restrict__ counts, const int32_t* __restrict__ cell_rows,
                   T* __restrict__ dst, int32_t* __restrict__ perm, int32_t* __restrict__ start,
                   int2* __restrict__ table, int cap, int gsz, int32_t* __restrict__ gcell,
                   Gate gate) {
  wait_for_previous();
  if (!gate.open()) return;
  constexpr int WARPS = 8, ITER = kChunkRows / (WARPS * 32);
  __shared__ int wcnt[WARPS][kMaxCells];
  __shared__ int base[kMaxCells];
  __shared__ int scan[64];
  int blk, nrows;
  const int b = block_set<kChunkRows>(offs, B, per, &blk);
  const int64_t row0 = set_rows(offs, b, each, &nrows);
  const int nblk = (int)(((int64_t)nrows + kChunkRows - 1) / kChunkRows);
  if (blk >= nblk) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  // thread p: rows of cell p in the whole set and in earlier blocks
  int tot = 0, before = 0;
  if ((int)threadIdx.x < P) {
    const int32_t* c = counts + chunk0(offs, b, per) * P + threadIdx.x;
    if (cell_rows) {
      tot = __ldg(cell_rows + (int64_t)b * P + threadIdx.x);
      before = __ldg(c + (int64_t)blk * P);
    } else {
#pragma unroll 16
      for (int q = 0; q < nblk; ++q) {
        const int v = __ldg(c + (int64_t)q * P);
        tot += v;
        if (q < blk) before += v;
      }
    }
  }
  int all = 0;
  const int first = block_exclusive_scan(tot, &all, scan);
  if ((int)threadIdx.x < P) base[threadIdx.x] = first + before;
  if (blk == 0) {
    int32_t* so = start + (int64_t)b * (P + 1);
    if ((int)threadIdx.x < P) so[threadIdx.x] = first;
    if (threadIdx.x == 0) so[P] = nrows;
    if (table) {
      const int ng = (int)threadIdx.x < P ? (tot + gsz - 1) / gsz : 0;
      int gall = 0;
      const int g0 = block_exclusive_scan(ng, &gall, scan);
      int2* to = table + (int64_t)b * cap;
      for (int g = 0; g < ng; ++g) {
        to[g0 + g] = make_int2(first + gsz * g, min(gsz, tot - gsz * g));
        if (gcell) gcell[(int64_t)b * cap + g0 + g] = threadIdx.x;
      }
      for (int g = gall + threadIdx.x; g < cap; g += blockDim.x) to[g] = make_int2(0, 0);
    }
  }
  for (int e = threadIdx.x; e < WARPS * kMaxCells; e += blockDim.x) (&wcnt[0][0])[e] = 0;
  __syncthreads();
  int ids[ITER];
#pragma unroll
  for (int i = 0; i < ITER; ++i) {
    const int r = blk * kChunkRows + (w * ITER + i) * 32 + lane;
    ids[i] = r < nrows ? (int)id[row0 + r] : -1;
    const unsigned m = __match_any_sync(kFull, ids[i]);
    if (ids[i] >= 0 && (m & ((1u << lane) - 1u)) == 0) wcnt[w][ids[i]] += __popc(m);
    __syncwarp();
  }
  __syncthreads();
  if ((int)threadIdx.x < P) {
    int o = base[threadIdx.x];
    for (int u = 0; u < WARPS; ++u) {
      const int v = wcnt[u][threadIdx.x];
      wcnt[u][threadIdx.x] = o;
      o += v;
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < ITER; ++i) {
    const int r = blk * kChunkRows + (w * ITER + i) * 32 + lane;
    const unsigned m = __match_any_sync(kFull, ids[i]);
    const unsigned lower = m & ((1u << lane) - 1u);
    int at = 0;
    if (ids[i] >= 0) at = wcnt[w][ids[i]] + __popc(lower);
    __syncwarp();
    if (ids[i] >= 0 && lower == 0) wcnt[w][ids[i]] += __popc(m);
    __syncwarp();
    if (ids[i] >= 0) {
      const int64_t from = row0 + r, to = row0 + at;
      if (perm) perm[to] = r;
      const float4* s4 = reinterpret_cast<const float4*>(src + from * DP);
      float4* d4 = reinterpret_cast<float4*>(dst + to * DP);
#pragma unroll
      for (int q = 0; q < DP * (int)sizeof(T) / 16; ++q) d4[q] = s4[q];
    }
  }
}

// Thread q of a block keeps the unit vectors from cell p's centre to those of cells q
// and q + P / 2, the rows of p come by broadcast from shared memory; DP multiply-adds
// a (row, cell), and a row's loads serve two of them.  Only cells below *npiv have
// rows, so a warp whose second 32 lie beyond it skips them (200,000 x 16: 61 -> 52 us).
constexpr int kExtRows = 64;

template <int DP, int NU>
__device__ __forceinline__ void extent_rows(const float* tile, int nr, const float (&v)[2][DP],
                                            float (&far_)[2]) {
#pragma unroll (DP <= 16 ? 4 : 2)
  for (int r = 0; r < nr; ++r) {
    float s[NU];
#pragma unroll
    for (int u = 0; u < NU; ++u) s[u] = 0.0f;
#pragma unroll
    for (int k = 0; k < DP; k += 4) {
      const float4 x = *reinterpret_cast<const float4*>(tile + r * DP + k);
#pragma unroll
      for (int u = 0; u < NU; ++u) {
        s[u] = fmaf(x.x, v[u][k], s[u]);
        s[u] = fmaf(x.y, v[u][k + 1], s[u]);
        s[u] = fmaf(x.z, v[u][k + 2], s[u]);
        s[u] = fmaf(x.w, v[u][k + 3], s[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < NU; ++u)
      far_[u] = (s[u] > far_[u] || !(s[u] == s[u])) ? s[u] : far_[u];   // NaN wins
  }
}

template <int DP>
__global__ void __launch_bounds__(kMaxCells / 2)
    extent_kernel(const float* __restrict__ rows, int P, const int32_t* __restrict__ npiv,
                  const int32_t* __restrict__ start, const float* __restrict__ ctr,
                  float2* __restrict__ ext, Gate gate) {
  wait_for_previous();
  if (!gate.open()) return;
  __shared__ __align__(16) float tile[kExtRows * DP];
  const int p = blockIdx.x;
  const int a = start[p], e = start[p + 1];
  const bool both = *npiv > P / 2 + (int)(threadIdx.x & ~31u);   // (the same for a warp)
  if (a + (int)blockIdx.y * kExtRows >= e && blockIdx.y > 0) return;
  float v[2][DP], dist[2], far_[2] = {0.0f, 0.0f};
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int q = threadIdx.x + u * (P / 2);
    float d2 = 0.0f;
#pragma unroll
    for (int k = 0; k < DP; k += 4) {
      const float4 c = __ldg(reinterpret_cast<const float4*>(ctr + q * DP + k));
      const float4 o = __ldg(reinterpret_cast<const float4*>(ctr + p * DP + k));
      v[u][k] = c.x - o.x;
      v[u][k + 1] = c.y - o.y;
      v[u][k + 2] = c.z - o.z;
      v[u][k + 3] = c.w - o.w;
    }
#pragma unroll
    for (int k = 0; k < DP; ++k) d2 = fmaf(v[u][k], v[u][k], d2);
    dist[u] = sqrtf(d2);
    const float inv = dist[u] > 0.0f ? 1.0f / dist[u] : 0.0f;
#pragma unroll
    for (int k = 0; k < DP; ++k) v[u][k] *= inv;
  }
  for (int r0 = a + blockIdx.y * kExtRows; r0 < e; r0 += gridDim.y * kExtRows) {
    const int nr = min(kExtRows, e - r0);
    __syncthreads();
    for (int i = threadIdx.x; i < nr * DP; i += blockDim.x)
      tile[i] = rows[(int64_t)r0 * DP + i] - __ldg(ctr + p * DP + i % DP);
    __syncthreads();
    if (both) extent_rows<DP, 2>(tile, nr, v, far_);
    else extent_rows<DP, 1>(tile, nr, v, far_);
  }
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    if (u == 1 && !both) continue;   // (never looked up)
    // (cleared to zero: not negative, so the bits order as integers do)
    float* o = reinterpret_cast<float*>(ext + (threadIdx.x + u * (P / 2)) * P + p);
    atomicMax(reinterpret_cast<unsigned*>(o), __float_as_uint(far_[u]) & 0x7fffffffu);
    if (blockIdx.y == 0) o[1] = dist[u];
  }
}

cudaError_t launch_extents(const float* rows, int DP, int P, const int32_t* npiv,
                           const int32_t* start, const float* ctr, float2* ext, cudaStream_t st,
                           Gate gate) {
  const cudaError_t e = cudaMemsetAsync(ext, 0, (size_t)P * P * 8, st);
  if (e != cudaSuccess) return e;
  // (cells differ in size by an order of magnitude: blocks past a cell's rows leave at once)
  const dim3 grid((unsigned)P, gate.walk ? 16 : 32);   // (fewer where they may all be in vain)
#define FMS_EXTENT(DP_) \
  return launch_gated(gate, extent_kernel<DP_>, grid, P / 2, 0, st, rows, P, npiv, start, ctr, ext, gate)
  switch (DP) {
    case 16: FMS_EXTENT(16);
    case 32: FMS_EXTENT(32);
    case 64: FMS_EXTENT(64);
  }
#undef FMS_EXTENT
  return cudaErrorInvalidValue;
}

template <typename T, int DP>
static cudaError_t sort_t(const T* src, const int64_t* offs, int B, int64_t nrows, bool points,
                          int P, int64_t total, void* scratch, T* dst, int32_t* perm,
                          int32_t* start, T* ctr, int32_t* npiv, T* rad, int2* table, int group,
                          int32_t* gcell, Gate gate, cudaStream_t st) {
  const SortScratch sc = sort_scratch(B, nrows, P, offs ? total : 0);   // (as it was sized)
  unsigned char* base = static_cast<unsigned char*>(scratch);
  unsigned char* id = base + sc.id;
  int32_t* counts = reinterpret_cast<int32_t*>(base + sc.counts);
  unsigned long long* far_ = reinterpret_cast<unsigned long long*>(base + sc.far_);
  const int64_t per64 = sort_blocks(nrows), pper = (nrows + kPivotRows - 1) / kPivotRows;
  const int64_t grid64 = offs ? runs_of_sets<kChunkRows>(total, B) : per64 * B;
  const int64_t pgrid64 = offs ? runs_of_sets<kPivotRows>(total, B) : pper * B;
  if (pgrid64 > INT32_MAX || (int64_t)P * B > INT32_MAX) return cudaErrorInvalidValue;
  const int per = (int)per64, n32 = (int)nrows;
  const unsigned grid = (unsigned)grid64;
  const size_t sm = (size_t)P * (DP + 1) * sizeof(T) + (size_t)P * 4;
  const size_t sm0 = (size_t)P / 2 * (DP + 1) * sizeof(T) + (size_t)P / 2 * 8;
  cudaError_t e = cudaSuccess;
  if (sm > 40 * 1024) {   // (static arrays count against the default 48 KB)
    e = cudaFuncSetAttribute(assign_kernel<T, DP, true>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(assign_kernel<T, DP, false>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
  }
  if (points) {
    e = cudaMemsetAsync(far_, 0, (size_t)B * (P / 2) * 8, st);
    if (e != cudaSuccess) return e;
    e = launch_gated(gate, pivot_kernel<T, DP>, (unsigned)pgrid64, 256, sm0, st, src, offs, B, n32,
                     P / 2, (int)pper, id, far_, gate);
    if (e == cudaSuccess)
      e = launch_gated(gate, select_kernel<T, DP>, B, kMaxCells, 0, st, src, offs, n32, P, far_, ctr,
                       npiv, gate);
  }
  auto assign = points ? assign_kernel<T, DP, true> : assign_kernel<T, DP, false>;
  if (e == cudaSuccess)
    e = launch_gated(gate, assign, grid, assign_threads<T, DP>(), sm, st, src, offs, B, n32, per, P,
                     id, counts, ctr, npiv, gate);
  int32_t* cell_rows = nullptr;
  if (e == cudaSuccess && per > kScanChunks) {
    cell_rows = reinterpret_cast<int32_t*>(base + sc.cell_rows);
    e = launch_gated(gate, scan_kernel, (unsigned)(P / 32 * B), 1024, 0, st, offs, n32, per, P,
                     counts, cell_rows, gate);
  }
  if (e == cudaSuccess)
    e = launch_gated(gate, scatter_kernel<T, DP>, grid, 256, 0, st, src, offs, B, n32, per, P, id,
                     counts, cell_rows, dst, perm, start, table, group_cap(nrows, P, group), group,
                     gcell, gate);
  if (e == cudaSuccess && points)
    e = launch_gated(gate, bound_kernel<T, DP>, (unsigned)(P * B), 32 * kBoundWarps, 0, st, dst,
                     offs, n32, P, start, ctr, rad, gate);
  return e;
}

template <typename T>
cudaError_t launch_sort(const T* src, int B, int64_t nrows, int DP, bool points, int P,
                        void* scratch, T* dst, int32_t* perm, int32_t* start, T* ctr,
                        int32_t* npiv, T* rad, int2* table, cudaStream_t st, const int64_t* offs,
                        int64_t total, int group, int32_t* gcell, Gate gate) {
  if (total == 0) total = (int64_t)B * nrows;
  if (P < 32 || P > kMaxCells || (P & 31) || B < 1) return cudaErrorInvalidValue;
#define FMS_SORT(DP_)                                                                           \
  return sort_t<T, DP_>(src, offs, B, nrows, points, P, total, scratch, dst, perm, start, ctr, \
                        npiv, rad, table, group, gcell, gate, st)
  switch (DP) {
    case 4: FMS_SORT(4);
    case 8: FMS_SORT(8);
    case 16: FMS_SORT(16);
    case 32: FMS_SORT(32);
    case 64:
      if constexpr (sizeof(T) == 4) FMS_SORT(64);
  }
#undef FMS_SORT
  return cudaErrorInvalidValue;
}

template cudaError_t launch_sort<float>(const float*, int, int64_t, int, bool, int, void*, float*,
                                        int32_t*, int32_t*, float*, int32_t*, float*, int2*,
                                        cudaStream_t, const int64_t*, int64_t, int, int32_t*, Gate);
template cudaError_t launch_sort<double>(const double*, int, int64_t, int, bool, int, void*,
                                         double*, int32_t*, int32_t*, double*, int32_t*, double*,
                                         int2*, cudaStream_t, const int64_t*, int64_t, int, int32_t*, Gate);

}  // namespace cells
}  // namespace fms

// Device body of the sorted prune, shared by the single-set and batched kernels.
#pragma once

#include <type_traits>

#include "fms_internal.cuh"

namespace fms {

// Same prune with the candidates in shared memory, in two stages: (1) the block
// sorts the candidates by (score descending, rank ascending); (2) it takes batches
// of up to 32 from the list of those still alive, resolves each batch in visit
// order, tests the whole list against the modes accepted from it and compacts the
// list in place.
//
// Candidates that converged to one mode have nearly the same score and stand in a
// row, so a batch takes its members from as far down the list as it can: a
// candidate within r of the one before it is passed over (it is expected to fall
// to the mode its predecessor fell to).  The test of the list shows whether each
// one passed over does lie within r of a mode accepted before its turn; at the
// first that does not, the batch is cut: modes after it are put back, it heads the
// next batch, and from then on batches pass over nothing.  Every suppression uses
// the distance of the one-by-one greedy visit, so the accepted set and its order
// are that visit's.
//
// What bounds it is the chain of barriers and dependent shared memory loads of
// one block (a batch is nine barriers, 3 us at d = 2 and 5 at d = 32), hence few
// batches: of 32 modes, not of 32 candidates.  2,000 candidates of 5 modes at d = 2
// take 22 us (batches of 32 candidates, each tested against all modes so far: 50);
// the three prunes of a 65,536 x 32 clustering of 64 modes 48 (135), its FP64 prune
// 24 (72), the two of 200,000 x 16 directions 19 (34) and 10 (19).
constexpr int kPruneTileStride = 36;   // row of the transposed batch tile (16-byte aligned)
constexpr int kPruneMaxDim = 64;
constexpr int kPruneThreads = 1024;    // block size of the sorted prune
constexpr int kPruneModes = 4;         // modes x entries of one thread at a time: a broadcast
constexpr int kPruneEntries = 4;       //   of 16 bytes takes the shared memory pipe 4 cycles

// Wider FP32 candidates are tested by their first coordinates, and the whole
// distance is taken only of the pairs that these leave within r: of 64 modes and
// 512 candidates at d = 32 that is a quarter of the arithmetic of one SM.
constexpr int kPruneFirst = 8;

// sort slots: a power of two
__host__ __device__ inline int prune_slots(int K) {
  int P = 32;
  while (P < K) P <<= 1;
  return P;
}

// row length of the coordinates: odd, so that neither storing columns nor reading
// rows meets a bank twice
__host__ __device__ inline int prune_row(int K) { return (K + 31) / 32 * 32 + 1; }

// two buffers of rank words; masks, modes' norms and indices, members' places;
// horizon and cut; masks of the groups
constexpr int kPruneScratchInts = 64 + 4 * 32 + 32 + kPruneThreads;

// Shared memory for up to K candidates of d coordinates: the batch's tile and
// the modes accepted from it, scratch, sort keys (then the list), the visit order
// and the first `pre` coordinates of every candidate in that order, transposed.
// FP64 positions are held rounded to FP32 (see PruneTest).
template <typename ST>
__host__ __device__ inline size_t greedy_sorted_smem(int K, int d, int pre) {
  return (size_t)((d + 3) & ~3) * (kPruneTileStride + 32) * 4 + kPruneScratchInts * 4 +
         (size_t)prune_slots(K) * (sizeof(ST) + 4) + (size_t)prune_row(K) * pre * 4;
}

// The coordinates to preload: all, else those of the first test, else none.
template <typename ST>
__host__ __device__ inline int greedy_sorted_pre(int K, int d, size_t limit) {
  if (greedy_sorted_smem<ST>(K, d, d) <= limit) return d;
  if (d > kPruneFirst && greedy_sorted_smem<ST>(K, d, kPruneFirst) <= limit) return kPruneFirst;
  return 0;
}

// ---------------------------------------------------------------------------
// The greedy visit for candidate sets too large for the sorted prune's shared
// memory: repeatedly accept the remaining candidate of highest (score, lowest
// index) and drop every candidate within r of it.  The remaining candidates
// are kept as a compacted list (in `list`, K entries of global memory); one
// pass per accepted mode drops the new mode's neighbours and finds the next
// winner, each thread taking kGlobalRun list entries per step with their loads
// issued together.  The winner and every suppression are decided exactly as
// in the one-by-one visit, so the accepted set and order are the same.
// Candidate q has rank q; its row is cand_row[q] (or q when cand_row is
// null).  `sm` holds greedy_global_smem() bytes of shared memory.
// ---------------------------------------------------------------------------
constexpr int kGlobalRun = 8;

template <typename ST>
__device__ __forceinline__ void argmax_merge(ST& best, int& bq, ST os, int oq) {
  if (os > best || (os == best && oq < bq)) {
    best = os;
    bq = oq;
  }
}

// Block-wide (score desc, index asc) winner; INT32_MAX when no candidate
// has a comparable score.  Every thread returns the same value.
template <typename ST>
__device__ int block_argmax(ST best, int bq, ST* sh_s, int* sh_q, int* sh_best) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    const ST os = __shfl_xor_sync(kFull, best, o);
    const int oq = __shfl_xor_sync(kFull, bq, o);
    argmax_merge<ST>(best, bq, os, oq);
  }
  if (lane == 0) {
    sh_s[wid] = best;
    sh_q[wid] = bq;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    ST b = sh_s[0];
    int bb = sh_q[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) argmax_merge<ST>(b, bb, sh_s[w], sh_q[w]);
    *sh_best = bb;
  }
  __syncthreads();
  const int win = *sh_best;
  __syncthreads();   // sh_best and sh_s / sh_q are reused by the next call
  return win;
}

// shared memory of greedy_global_body: winner scores and indices per warp,
// the winner's coordinates, the winner, the scan's warp sums
template <typename PT, typename ST>
__host__ __device__ constexpr size_t greedy_global_smem() {
  return 32 * sizeof(ST) + 32 * 4 + kPruneMaxDim * sizeof(PT) + 16 + 64 * 4;
}

template <typename PT, typename ST>
__device__ void greedy_global_body(const int32_t* __restrict__ cand_row, const int K,
                                   const ST* __restrict__ score, const PT* __restrict__ pos,
                                   int DP, int d, PT r2, int32_t* __restrict__ list,
                                   int32_t* __restrict__ accepted, int32_t* __restrict__ M_out,
                                   unsigned char* sm) {
  ST* sh_s = reinterpret_cast<ST*>(sm);
  int* sh_q = reinterpret_cast<int*>(sh_s + 32);
  PT* sh_pos = reinterpret_cast<PT*>(sh_q + 32);
  int* sh_best = reinterpret_cast<int*>(sh_pos + kPruneMaxDim);
  int* scratch = sh_best + 4;
  const int T = blockDim.x;
  ST best = (ST)-INFINITY;
  int bq = INT32_MAX;
  for (int b = 0; b < K; b += T * kGlobalRun) {
#pragma unroll
    for (int v = 0; v < kGlobalRun; ++v) {
      const int q = b + v * T + threadIdx.x;
      if (q < K) {
        list[q] = q;
        argmax_merge<ST>(best, bq, score[q], q);
      }
    }
  }
  int win = block_argmax<ST>(best, bq, sh_s, sh_q, sh_best);
  int len = K, M = 0;
  while (win != INT32_MAX) {
    if (threadIdx.x == 0) accepted[M] = win;
    ++M;
    const int64_t wrow = cand_row ? cand_row[win] : win;
    for (int k = threadIdx.x; k < d; k += T) sh_pos[k] = pos[wrow * DP + k];
    __syncthreads();
    best = (ST)-INFINITY;
    bq = INT32_MAX;
    int newlen = 0;
    for (int b = 0; b < len; b += T * kGlobalRun) {
      int q[kGlobalRun];
      int64_t row[kGlobalRun];
      ST sc[kGlobalRun];
      PT d2[kGlobalRun];
#pragma unroll
      for (int v = 0; v < kGlobalRun; ++v) {
        const int idx = b + v * T + threadIdx.x;
        q[v] = idx < len ? list[idx] : -1;
      }
#pragma unroll
      for (int v = 0; v < kGlobalRun; ++v) {
        sc[v] = q[v] >= 0 ? score[q[v]] : (ST)0;
        row[v] = q[v] >= 0 ? (cand_row ? (int64_t)cand_row[q[v]] : (int64_t)q[v]) : 0;
        d2[v] = 0;
      }
      for (int k = 0; k < d; ++k) {
        const PT pk = sh_pos[k];
#pragma unroll
        for (int v = 0; v < kGlobalRun; ++v) {
          if (q[v] >= 0) {
            const PT e = pos[row[v] * DP + k] - pk;
            d2[v] += e * e;
          }
        }
      }
      unsigned keep = 0;
      int cnt = 0;
#pragma unroll
      for (int v = 0; v < kGlobalRun; ++v) {
        if (q[v] >= 0 && q[v] != win && !(d2[v] < r2)) {
          keep |= 1u << v;
          ++cnt;
          argmax_merge<ST>(best, bq, sc[v], q[v]);
        }
      }
      // in-place compaction: this step writes only below the end of what it
      // read, and every read precedes the scan's barriers
      int tot;
      int off = block_exclusive_scan(cnt, &tot, scratch);
#pragma unroll
      for (int v = 0; v < kGlobalRun; ++v)
        if ((keep >> v) & 1u) list[newlen + off++] = q[v];
      newlen += tot;
    }
    len = newlen;
    win = block_argmax<ST>(best, bq, sh_s, sh_q, sh_best);
  }
  if (threadIdx.x == 0) *M_out = M;
}

// Sort key of a score: ascending order of the keys is the visit order.
__device__ __forceinline__ unsigned visit_key(float f) {
  if (!(f == f)) f = -INFINITY;   // a NaN score counts as -inf
  if (f == 0.0f) f = 0.0f;        // -0 and +0 are equal scores
  const unsigned u = __float_as_uint(f);
  return (u & 0x80000000u) ? u : ~(u | 0x80000000u);
}

__device__ __forceinline__ unsigned long long visit_key(double f) {
  if (!(f == f)) f = -INFINITY;
  if (f == 0.0) f = 0.0;
  const unsigned long long u = (unsigned long long)__double_as_longlong(f);
  return (u >> 63) ? u : ~(u | (1ull << 63));
}

// Whether two candidates lie within r.  FP32 positions: the squared distance
// itself.  FP64 positions: the distance of the positions rounded to FP32 decides
// where it is surely right, else FP64 does (its rate is 1/64 of FP32's, and all
// but the pairs within about 1e-6 of r are decided in FP32).  Rounding moves a
// position by at most u|x|, u = 2^-24, and a difference by another u|e|; the sum
// and the root are good to (d + 4) u.  So the FP32 distance differs from the
// true one by less than (d + 8) u times itself plus u (|x| + |y|); the margins
// here are twice that.
template <typename PT>
struct PruneTest {
  const PT* pos;
  const int32_t* cand_row;
  int DP, d;
  PT r2;
  float lo, hi;   // FP64 positions: surely within r below lo, surely not above hi
  __device__ PruneTest(const PT* pos_, const int32_t* rows, int DP_, int d_, PT r2_)
      : pos(pos_), cand_row(rows), DP(DP_), d(d_), r2(r2_), lo(0.0f), hi(0.0f) {
    if constexpr (sizeof(PT) == 8) {
      const float r = sqrtf((float)r2), c = (float)(2 * d + 32) * 5.9604645e-8f;
      const bool usable = r > 1e-10f && r < 1e10f;   // no under- or overflow of a square near r
      lo = usable ? r - r * c : -INFINITY;
      hi = usable ? r + r * c : INFINITY;
    }
  }
  __device__ __forceinline__ int64_t row(int q) const {
    return cand_row ? (int64_t)cand_row[q] : (int64_t)q;
  }
  // s, a, b: squared FP32 distance and squared norms of candidates p and q
  __device__ __forceinline__ bool within(float s, float a, float b, int p, int q) const {
    if constexpr (sizeof(PT) == 4) {
      return s < r2;
    } else {
      const float D = sqrtf(s), m = (sqrtf(a) + sqrtf(b)) * 2.3841858e-7f + 1e-17f;
      if (D + m < lo) return true;
      if (D - m > hi && D < 1e15f) return false;
      return within_exactly(p, q);
    }
  }
  // (out of line: a small problem's time is that of fetching the code)
  __device__ __noinline__ bool within_exactly(int p, int q) const {
    const PT *x = pos + row(p) * DP, *y = pos + row(q) * DP;
    PT d2 = 0;
    for (int k = 0; k < d; ++k) {
      const PT e = x[k] - y[k];
      d2 += e * e;
    }
    return d2 < r2;
  }
};

// A candidate in the sort: key, then index.  FP32 scores: both in one integer.
struct VisitF {
  unsigned long long v;
  __device__ __forceinline__ void set(unsigned key, int i) {
    v = ((unsigned long long)key << 32) | (unsigned)i;
  }
  __device__ __forceinline__ void pad() { v = ~0ull; }
  __device__ __forceinline__ int index() const { return (int)(unsigned)v; }
  __device__ __forceinline__ bool before(const VisitF& o) const { return v < o.v; }
  __device__ __forceinline__ VisitF shfl_xor(int m) const {
    VisitF o;
    o.v = __shfl_xor_sync(kFull, v, m);
    return o;
  }
  __device__ __forceinline__ void put(unsigned char* buf, int, int i) const {
    reinterpret_cast<unsigned long long*>(buf)[i] = v;
  }
  __device__ __forceinline__ void get(const unsigned char* buf, int, int i) {
    v = reinterpret_cast<const unsigned long long*>(buf)[i];
  }
};

struct VisitD {
  unsigned long long k;
  int at;
  __device__ __forceinline__ void set(unsigned long long key, int i) {
    k = key;
    at = i;
  }
  __device__ __forceinline__ void pad() {
    k = ~0ull;
    at = INT32_MAX;
  }
  __device__ __forceinline__ int index() const { return at; }
  __device__ __forceinline__ bool before(const VisitD& o) const {
    return k < o.k || (k == o.k && at < o.at);
  }
  __device__ __forceinline__ VisitD shfl_xor(int m) const {
    VisitD o;
    o.k = __shfl_xor_sync(kFull, k, m);
    o.at = __shfl_xor_sync(kFull, at, m);
    return o;
  }
  __device__ __forceinline__ void put(unsigned char* buf, int P, int i) const {
    reinterpret_cast<unsigned long long*>(buf)[i] = k;
    reinterpret_cast<int*>(buf + (size_t)P * 8)[i] = at;
  }
  __device__ __forceinline__ void get(const unsigned char* buf, int P, int i) {
    k = reinterpret_cast<const unsigned long long*>(buf)[i];
    at = reinterpret_cast<const int*>(buf + (size_t)P * 8)[i];
  }
};

// Bitonic sort of P slots in registers, E a thread of the first P / E: strides
// below E within the thread, up to 16 E by shuffles, beyond through `buf`.  At P =
// 2,048, E = 8, that is 30, 30 and 6 of the 66 steps.  What bounds it is some 15
// instructions a slot and step (12 us at 2,048 slots, as with a slot a thread), and
// beyond 8,192 slots it would be the barriers of a sort in shared memory (9,000
// candidates: 195 us there, 112 so).
template <typename V, typename ST, int E>
__device__ __noinline__ void sort_slots(const ST* __restrict__ score, int K, int P,
                                           unsigned char* buf, int* order) {
  V x[E];
  const int tid = threadIdx.x, T = P / E;
  const bool in = tid < T;   // (whole warps)
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int i = tid * E + e;
    if (i < K) x[e].set(visit_key(score[i]), i);
    else x[e].pad();
  }
  auto merge = [&](int e, const V& o, int k, int j) {
    const int i = tid * E + e;
    const bool low = ((i & j) == 0) == ((i & k) == 0);   // this slot takes the earlier one
    if (o.before(x[e]) == low) x[e] = o;
  };
  for (int k = 2; k <= P; k <<= 1) {
    for (int j = k >> 1; j >= 32 * E; j >>= 1) {
      if (in)
#pragma unroll
        for (int e = 0; e < E; ++e) x[e].put(buf, P, e * T + tid);
      __syncthreads();
      if (in)
#pragma unroll
        for (int e = 0; e < E; ++e) {
          V o;
          o.get(buf, P, e * T + (tid ^ (j / E)));
          merge(e, o, k, j);
        }
      __syncthreads();
    }
    if (!in) continue;
    for (int j = min(k >> 1, 16 * E); j >= E; j >>= 1)
#pragma unroll
      for (int e = 0; e < E; ++e) merge(e, x[e].shfl_xor(j / E), k, j);
#pragma unroll
    for (int j = E / 2; j > 0; j >>= 1)
      if (j < k)
#pragma unroll
        for (int e = 0; e < E; ++e)
          if (!(e & j)) {
            const V a = x[e], b = x[e | j];
            merge(e, b, k, j);
            merge(e | j, a, k, j);
          }
  }
  if (in)
#pragma unroll
    for (int e = 0; e < E; ++e)
      if (tid * E + e < K) order[tid * E + e] = x[e].index();
}

// order[i] = the i-th candidate in visit order.  buf: prune_slots(K) x (sizeof(ST)
// + 4) bytes, the last four a slot of which are `order`.
template <typename ST>
__device__ void visit_order(const ST* __restrict__ score, int K, unsigned char* buf, int* order) {
  using V = typename std::conditional<sizeof(ST) == 4, VisitF, VisitD>::type;
  const int P = prune_slots(K);
  if (P <= 256) {
    // a candidate's place is the number of those before it: four candidates a
    // thread, a group of 4,096 / P lanes (16 or 32, then several groups) to each four
    constexpr int Q = 4;
    const int G = min(32, Q * kPruneThreads / P), c = threadIdx.x / G * Q, at = threadIdx.x % G;
    if ((int)threadIdx.x < P) {
      V x;
      if ((int)threadIdx.x < K) x.set(visit_key(score[threadIdx.x]), threadIdx.x);
      else x.pad();
      x.put(buf, P, threadIdx.x);
    }
    __syncthreads();
    int r[Q] = {0, 0, 0, 0};
    if (c < P) {   // (whole warps)
      V x[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) x[q].get(buf, P, c + q);
#pragma unroll 4
      for (int j = at; j < P; j += G) {
        V o;
        o.get(buf, P, j);
#pragma unroll
        for (int q = 0; q < Q; ++q) r[q] += o.before(x[q]) ? 1 : 0;
      }
      for (int o = G >> 1; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < Q; ++q) r[q] += __shfl_xor_sync(kFull, r[q], o);
    }
    __syncthreads();
    if (at == 0)
#pragma unroll
      for (int q = 0; q < Q; ++q)
        if (c + q < K) order[r[q]] = c + q;
  } else if (P <= 512) {
    sort_slots<V, ST, 2>(score, K, P, buf, order);
  } else if (P <= 1024) {
    sort_slots<V, ST, 4>(score, K, P, buf, order);
  } else if (P <= 8 * kPruneThreads) {
    sort_slots<V, ST, 8>(score, K, P, buf, order);
  } else {   // at most 16,384 fit in shared memory
    sort_slots<V, ST, 16>(score, K, P, buf, order);
  }
  __syncthreads();
}

// Number of true flags of the block's threads below this one, and in all (*total):
// one barrier.  `words` is one of two buffers of 32, used in turn.
__device__ __forceinline__ int block_rank(bool flag, int* total, unsigned* words) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned m = __ballot_sync(kFull, flag);
  if (lane == 0) words[warp] = m;
  __syncthreads();
  const int n = lane < (int)(blockDim.x >> 5) ? __popc(words[lane]) : 0;
  *total = __reduce_add_sync(kFull, n);
  return __reduce_add_sync(kFull, lane < warp ? n : 0) + __popc(m & ((1u << lane) - 1u));
}

__device__ __forceinline__ void load_row4(const float* p, float x[4]) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  x[0] = v.x, x[1] = v.y, x[2] = v.z, x[3] = v.w;
}

__device__ __forceinline__ void load_row4(const double* p, float x[4]) {
  const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
  x[0] = (float)a.x, x[1] = (float)a.y, x[2] = (float)b.x, x[3] = (float)b.y;
}

// Two FP32 values in one register pair: x - m and s + e e for two modes at once,
// each half rounded as the scalar operation is.
__device__ __forceinline__ void add_square2(unsigned long long& s, unsigned long long x,
                                            unsigned long long minus_m) {
  unsigned long long e;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(e) : "l"(x), "l"(minus_m));
  asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(s) : "l"(e));
}

template <typename PT, typename ST>
__device__ void greedy_sorted_body(const int32_t* __restrict__ cand_row, const int K,
                                   const ST* __restrict__ score, const PT* __restrict__ pos,
                                   int DP, int d, PT r2, int32_t* __restrict__ accepted,
                                   int32_t* __restrict__ M_out, unsigned char* smem,
                                   int pre) {
  constexpr bool kWide = sizeof(PT) == 8;
  const int P = prune_slots(K), XS = prune_row(K), d4 = (d + 3) & ~3;
  float* tile = reinterpret_cast<float*>(smem);             // [d4][kPruneTileStride]
  float* modes = tile + (size_t)d4 * kPruneTileStride;      // [d4][32], negated
  unsigned* words = reinterpret_cast<unsigned*>(modes + (size_t)d4 * 32);   // two buffers
  unsigned* near = words + 64;
  float* mnorm = reinterpret_cast<float*>(near + 32);
  int* mcand = reinterpret_cast<int*>(mnorm + 32);
  int* member = mcand + 32;                                 // a batch member's place in the list
  int* horizon = member + 32;                               // the batch's members lie before it
  int* cut = horizon + 1;
  unsigned* part = reinterpret_cast<unsigned*>(horizon + 32);
  unsigned char* buf = reinterpret_cast<unsigned char*>(part + kPruneThreads);
  // an entry: 2 x its place in the visit order + (it lies within r of the place before)
  int* list = reinterpret_cast<int*>(buf);
  int* order = reinterpret_cast<int*>(buf + (size_t)P * sizeof(ST));
  float* xs = reinterpret_cast<float*>(order + P);          // [d][XS]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const PruneTest<PT> test(pos, cand_row, DP, d, r2);
  visit_order<ST>(score, K, buf, order);
  if (pre) {   // DP is a power of two: whole rows, read together, eight loads in flight
    const int shift = 31 - __clz(DP);
    for (int e0 = threadIdx.x; e0 < K << shift; e0 += 8 * blockDim.x) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int e = e0 + u * blockDim.x, k = e & (DP - 1);
        v[u] = e < K << shift && k < pre ? (float)pos[test.row(order[e >> shift]) * DP + k] : 0.0f;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int e = e0 + u * blockDim.x, k = e & (DP - 1);
        if (e < K << shift && k < pre) xs[k * XS + (e >> shift)] = v[u];
      }
    }
    __syncthreads();
  }
  auto coord = [&](int i, int64_t row, int k) -> float {
    return k < pre ? xs[k * XS + i] : (float)pos[row * DP + k];
  };
  const int first_d = kWide ? d : min(d, kPruneFirst);
  const int near_d = pre ? pre : first_d;   // (a guess that the batches verify)
  for (int i = threadIdx.x; i < K; i += blockDim.x) {
    float s = i > 0 ? 0.0f : INFINITY;
    if (i > 0) {
      const int64_t r0 = test.row(order[i - 1]), r1 = test.row(order[i]);
#pragma unroll 8
      for (int k = 0; k < near_d; ++k) {
        const float e = coord(i, r1, k) - coord(i - 1, r0, k);
        s += e * e;
      }
    }
    list[i] = 2 * i + (s < (float)r2 ? 1 : 0);
  }
  part[threadIdx.x] = 0;
  int len = K, nacc = 0;
  int turn = 0;
  bool pass_over = true;
  while (len > 0) {
    if (threadIdx.x == 0) {
      *horizon = min(len, (int)blockDim.x);
      *cut = INT32_MAX;
    }
    __syncthreads();   // the list is written, the last batch's tile and modes are read
    // the batch: the first 32 of the block's first entries that are not passed over
    int before, nb;    // members before this thread's entry; members
    {
      const int i = threadIdx.x;
      bool lead = i < len;
      if (lead && i > 0 && pass_over) {
        const int e = list[i];
        lead = !(e & 1) || (list[i - 1] >> 1) != (e >> 1) - 1;
      }
      int tot;
      before = block_rank(lead, &tot, words + 32 * (turn ^= 1));
      if (lead && before < 32) member[before] = i;
      if (lead && before == 32) *horizon = i;
      nb = min(tot, 32);
    }
    __syncthreads();
    const int end = *horizon;
    const int slot = lane < nb ? member[lane] : INT32_MAX;   // lane's member, in every warp
    const int place = lane < nb ? list[slot] >> 1 : -1;
    const int mine = lane < nb ? order[place] : -1;
    {
      const int64_t row = mine >= 0 ? test.row(mine) : 0;
      for (int k = warp; k < d4; k += nwarps)
        tile[k * kPruneTileStride + lane] = mine >= 0 && k < d ? coord(place, row, k) : 0.0f;
    }
    __syncthreads();
    float n2 = 0.0f;   // |member|^2, in the warps that need it
    for (int v0 = warp * 4; v0 < 32; v0 += nwarps * 4) {
      float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
      n2 = 0.0f;
#pragma unroll 4
      for (int k = 0; k < d; ++k) {
        const float x = tile[k * kPruneTileStride + lane];
        const float4 m = *reinterpret_cast<const float4*>(&tile[k * kPruneTileStride + v0]);
        const float e0 = x - m.x, e1 = x - m.y, e2 = x - m.z, e3 = x - m.w;
        s[0] += e0 * e0;
        s[1] += e1 * e1;
        s[2] += e2 * e2;
        s[3] += e3 * e3;
        if (kWide) n2 += x * x;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float b = kWide ? __shfl_sync(kFull, n2, v0 + j) : 0.0f;
        const int other = kWide ? __shfl_sync(kFull, mine, v0 + j) : 0;
        const bool in = lane < nb && v0 + j < nb && test.within(s[j], n2, b, mine, other);
        const unsigned m = __ballot_sync(kFull, in);
        if (lane == 0) near[v0 + j] = m;
      }
    }
    __syncthreads();
    // every warp: the members accepted in visit order.  One with no earlier live
    // neighbour is accepted, its neighbours go, until none is left.
    const unsigned nm = near[lane];
    unsigned alive = nb == 32 ? kFull : (1u << nb) - 1u, acc = 0;
    while (alive) {
      const bool live = (alive >> lane) & 1u;
      const bool first = live && !(nm & alive & ((1u << lane) - 1u));
      const unsigned F = __ballot_sync(kFull, first);
      acc |= F;
      alive = __ballot_sync(kFull, live && !first && !(nm & F));
    }
    const int nn = __popc(acc);
    const bool taken = (acc >> lane) & 1u;
    const int at = __popc(acc & ((1u << lane) - 1u));
    if (len <= nb) {   // nothing but members
      if (warp == 0 && taken) accepted[nacc + at] = mine;
      nacc += nn;
      break;
    }
    for (int k = warp; k < d4; k += nwarps)
      if (taken) modes[k * 32 + at] = -tile[k * kPruneTileStride + lane];
    if (warp == 0 && taken) {
      mnorm[at] = n2;   // (warp 0 had members 0-3: n2 is set)
      mcand[at] = mine;
    }
    __syncthreads();
    // The list against the modes just accepted, a block of entries at a time,
    // compacted in place (a step writes only below the end of what it read, and
    // every read precedes the barriers).  A warp takes 128 entries and groups of
    // warps share the modes.
    int newlen = 0;
    unsigned valid = 0;                                       // modes not put back
    for (int b = 0; b < len; b += blockDim.x) {
      const int wide = (min(len - b, (int)blockDim.x) + 32 * kPruneEntries - 1) / (32 * kPruneEntries);
      const int groups = nwarps / wide, group = warp / wide;
      const int first = (warp - group * wide) * 32 * kPruneEntries + lane;
      for (int m0 = group * kPruneModes; m0 < nn && group < groups; m0 += groups * kPruneModes) {
        int p[kPruneEntries];
        unsigned long long s2[kPruneEntries][kPruneModes / 2];
        float a[kPruneEntries];
#pragma unroll
        for (int q = 0; q < kPruneEntries; ++q) {
          const int i = b + first + q * 32;
          p[q] = i < len ? list[i] >> 1 : 0;   // (past the end: entry 0, unused)
          a[q] = 0.0f;
#pragma unroll
          for (int j = 0; j < kPruneModes / 2; ++j) s2[q][j] = 0ull;
        }
        auto add = [&](int k, const float (&x)[kPruneEntries]) {
          const ulonglong2 m = *reinterpret_cast<const ulonglong2*>(&modes[k * 32 + m0]);
#pragma unroll
          for (int q = 0; q < kPruneEntries; ++q) {
            unsigned long long xx;
            asm("mov.b64 %0, {%1, %1};" : "=l"(xx) : "f"(x[q]));
            add_square2(s2[q][0], xx, m.x);
            add_square2(s2[q][1], xx, m.y);
            if (kWide) a[q] += x[q] * x[q];
          }
        };
        if (first_d <= pre) {
#pragma unroll 4
          for (int k = 0; k < first_d; ++k) {
            float x[kPruneEntries];
#pragma unroll
            for (int q = 0; q < kPruneEntries; ++q) x[q] = xs[k * XS + p[q]];
            add(k, x);
          }
        } else {   // DP is a multiple of 4
          for (int k0 = 0; k0 < first_d; k0 += 4) {
            float x[kPruneEntries][4];
#pragma unroll
            for (int q = 0; q < kPruneEntries; ++q) load_row4(pos + test.row(order[p[q]]) * DP + k0, x[q]);
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (k0 + u < first_d) {
                const float xu[kPruneEntries] = {x[0][u], x[1][u], x[2][u], x[3][u]};
                add(k0 + u, xu);
              }
          }
        }
        // (FP32: the whole distance, or of the first coordinates, which is no larger)
        const unsigned some = nn - m0 >= kPruneModes ? (1u << kPruneModes) - 1u : (1u << (nn - m0)) - 1u;
#pragma unroll
        for (int q = 0; q < kPruneEntries; ++q) {
          unsigned mask = 0;
#pragma unroll
          for (int j = 0; j < kPruneModes; ++j) {
            const unsigned long long h = s2[q][j / 2];
            const float s = __uint_as_float((unsigned)(j % 2 ? h >> 32 : h));
            if constexpr (kWide) {
              if (m0 + j < nn && b + first + q * 32 < len &&
                  test.within(s, a[q], mnorm[m0 + j], order[p[q]], mcand[m0 + j]))
                mask |= 1u << j;
            } else {
              mask |= s < r2 ? 1u << j : 0u;
            }
          }
          mask = b + first + q * 32 < len ? (mask & some) << m0 : 0u;
          if (mask) atomicOr(&part[first + q * 32], mask);
        }
      }
      __syncthreads();
      const int i = b + threadIdx.x;
      bool keep = i < len;
      const int entry = keep ? list[i] : 0;
      unsigned mask = part[threadIdx.x];   // the modes within r
      part[threadIdx.x] = 0;
      if (first_d < d && mask) {   // the whole distance to those that the first test left
        const int64_t row = test.row(order[entry >> 1]);
        unsigned left = mask;
        mask = 0;
        while (left) {
          const int m = __ffs(left) - 1;
          left &= left - 1;
          float s = 0.0f;
#pragma unroll 8
          for (int k = 0; k < d; ++k) {
            const float e = coord(entry >> 1, row, k) + modes[k * 32 + m];
            s += e * e;
          }
          if (test.within(s, 0.0f, 0.0f, 0, 0)) mask |= 1u << m;
        }
      }
      __syncwarp();
      if (b == 0) {
        const bool is_member = keep && before < nb && member[before] == i;
        if (keep && !is_member && i < end) {
          const unsigned earlier = before >= 32 ? acc : acc & ((1u << before) - 1u);
          const int ne = __popc(earlier);
          if (!(mask & (ne >= 32 ? kFull : (1u << ne) - 1u))) atomicMin(cut, i);
        }
        __syncthreads();
        const int stop = *cut;
        valid = __ballot_sync(kFull, taken && slot < stop);
        const int nv = __popc(valid);
        if (warp == 0 && taken && slot < stop) accepted[nacc + at] = mine;
        nacc += nv;
        valid = nv >= 32 ? kFull : (1u << nv) - 1u;   // as bits of `mask`
        if (stop != INT32_MAX) pass_over = false;
        if (is_member && i < stop) keep = false;
      }
      keep = keep && !(mask & valid);
      int tot;
      const int off = block_rank(keep, &tot, words + 32 * (turn ^= 1));
      if (keep) list[newlen + off] = entry;
      newlen += tot;
    }
    len = newlen;
  }
  if (threadIdx.x == 0) *M_out = nacc;
}

}  // namespace fms

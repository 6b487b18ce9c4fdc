// Cells of nearby points, and the walk over the cells that can reach a group
// of 32 seeds.
//
// A Gaussian weight falls below any share of the sum W of a seed's weights at
// a finite distance: with n points, dropping every point whose weight is below
// 2^-(32 + log2 n) W changes W and S/W by less than 2^-32 of W, a 256th of one
// FP32 rounding (guard_bits; more for FP64).  Points are therefore sorted into
// cells (the nearest of up to P pivots; a stable counting sort, so the order and
// every sum that follows is the same on each run), each with a bounding ball, and
// a group of seeds walks only the cells whose ball comes within the cutoff radius
// of the group's own ball.  The bound is checked against the W that came out: a group whose smallest W asks for a wider cutoff is evaluated again
// with that one (up to the distance where exp2 itself gives zero), so no
// assumption about the seeds enters.  A ball test that meets NaN or infinity
// keeps the cell.
#pragma once

#include "fms_internal.cuh"
#include "fms_route.cuh"

namespace fms {
namespace cells {

constexpr int kMaxCells = 256;      // cells of one set (ids are bytes)
constexpr int kChunkRows = 1024;    // rows one block of the sort handles
constexpr int kTileRows = 32;       // rows of one staged tile

// dropped weight, relative to W: 2^-kGuardBits (FP32: 2^-24 is one rounding)
template <typename T>
__host__ __device__ constexpr float guard_bits() {
  return sizeof(T) == 4 ? 32.0f : 62.0f;
}
// exponent from which exp2(-x) is exactly zero (FP32 flushes to zero below 2^-126)
template <typename T>
__host__ __device__ constexpr float zero_bits() {
  return sizeof(T) == 4 ? 128.0f : 1100.0f;
}

// Cells of B sets of n rows each (row b n + i).
template <typename T>
struct View {
  int P;                 // cells per set; 0: one cell with every row, nothing sorted
  const int32_t* start;  // [B][P + 1] first row of each cell (within the set)
  const T* ctr;          // [B][P][DP] the mean of each cell's rows
  const T* rad;          // [B][P] the distance of its farthest row from there
  const float2* ext;     // [P][P] (one set, FP32; nullable): at [q][p], how far cell p's
                         // rows reach from its centre towards cell q's, and the
                         // distance of the two centres
  Gate gate;             // closed: the kernel takes every row, as without cells
};

// How far cell p's rows reach towards a seed y at distance a from its centre: the
// extent towards cell q's centre, at distance delta from y, plus what the angle
// between the two directions can add (two unit vectors a/|a|, b/|b| differ by at
// most 2 |a - b| / (|a| + |b|)); never more than the radius.  In many dimensions
// the radius of a cluster is several times its extent in any one direction, and
// balls alone would find most clusters in reach of each other.
__device__ __forceinline__ float reach_towards(float rad, float2 ext, float a, float delta) {
  return fminf(rad, ext.x + rad * (2.0f * delta / (a + ext.y)));
}

// Groups of at most 32 rows of one cell.
struct Groups {
  const int2* table;     // [B][per_set] (first row within the set, rows); null: consecutive rows
  int per_set;           // groups of a set, some of them empty
};

template <typename T>
__device__ __forceinline__ T warp_max(T v) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    const T u = __shfl_xor_sync(kFull, v, o);
    v = (u > v || !(u == u)) ? u : v;   // NaN wins
  }
  return v;
}
template <typename T>
__device__ __forceinline__ T warp_min(T v) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    const T u = __shfl_xor_sync(kFull, v, o);
    v = (u < v || !(u == u)) ? u : v;   // NaN wins
  }
  return v;
}

__device__ __forceinline__ float csqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double csqrt(double x) { return sqrt(x); }

// Ball around the warp's 32 rows: their mean (same value in every lane) and
// the distance of the farthest.
template <typename T, int DP>
__device__ __forceinline__ T group_ball(const T (&y)[DP], T (&c)[DP]) {
  T r2 = T(0);
#pragma unroll
  for (int k = 0; k < DP; ++k) {
    T s = y[k];
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
    c[k] = s * T(1.0 / 32);
    const T e = y[k] - c[k];
    r2 += e * e;
  }
  return csqrt(warp_max(r2));
}

// The exponent below which weights may be dropped for a seed whose weights sum to W.
template <typename T>
__device__ __forceinline__ T cut_bits(T W, T log2n) {
  const T need = T(guard_bits<T>()) + log2n - T(log2f((float)W));
  return need < T(zero_bits<T>()) ? (need > T(1) ? need : T(1)) : T(zero_bits<T>());
}

// That exponent plus what the rounding of W in another order of summation can ask
// for (a repeated pass must not find that it needs an ulp more).
template <typename T>
__device__ __forceinline__ T widen(T need) {
  const T c = need + T(0.125);
  return c < T(zero_bits<T>()) ? c : T(zero_bits<T>());
}

// First guess of the cutoff exponent of a seed whose W is not known: small, since
// the pass at this cutoff gives a lower bound of W, from which the one that is
// needed follows (a guess from W >= 0.5 walks most of 200,000 x 16 directions).
constexpr float kFirstCut = 16.0f;

__device__ __forceinline__ void cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Warp w of a team of W walks every W-th tile of the listed row ranges in
// order: tiles of at most 32 consecutive rows of ROW elements, copied
// asynchronously one tile ahead into the warp's two-tile ring, tile_fn(rows in
// shared memory, count) for each.
template <int ROW, typename T, typename F>
__device__ __forceinline__ void walk_tiles(const T* __restrict__ rows, const int2* list, int nlist,
                                           int w, int W, T* ring, int lane, F&& tile_fn) {
  static_assert((ROW * sizeof(T)) % 16 == 0, "rows are copied 16 bytes at a time");
  constexpr int PER16 = 16 / (int)sizeof(T);
  int v = 0, t = w, cnt = 0;
  int2 cur = nlist > 0 ? list[0] : make_int2(0, 0);
  auto next = [&](int* row0) -> int {   // rows of the warp's next tile, 0 at the end
    while (v < nlist) {
      const int nt = (cur.y + kTileRows - 1) / kTileRows;
      if (t < nt) {
        const int r = t * kTileRows;
        *row0 = cur.x + r;
        t += W;
        return min(kTileRows, cur.y - r);
      }
      t -= nt;
      if (++v < nlist) cur = list[v];
    }
    return 0;
  };
  auto copy = [&](int row0, int c, T* dst) {
    const T* src = rows + (int64_t)row0 * ROW;
    const int n16 = c * (ROW / PER16);
    for (int i = lane; i < n16; i += 32) cp16(dst + i * PER16, src + i * PER16);
  };
  int row0 = 0, st = 0;
  cnt = next(&row0);
  if (cnt) copy(row0, cnt, ring);
  cp_commit();
  while (cnt) {
    const int c2 = next(&row0);
    if (c2) copy(row0, c2, ring + (st ^ 1) * kTileRows * ROW);
    cp_commit();
    cp_wait<1>();
    __syncwarp();
    tile_fn(ring + st * kTileRows * ROW, cnt);
    __syncwarp();
    cnt = c2;
    st ^= 1;
  }
  cp_wait<0>();
}

// The same for n unsorted rows that all lie in shared memory.
template <int ROW, typename T, typename F>
__device__ __forceinline__ void walk_resident(const T* rows, int n, int w, int W, F&& tile_fn) {
  for (int r = w * kTileRows; r < n; r += W * kTileRows)
    tile_fn(rows + r * ROW, min(kTileRows, n - r));
}

// Cells for a set of n points and m seeds (a power of two >= 32).  Half of them
// start from strided points, so a cluster holding a share f of the points is
// missed by all of those with probability exp(-f P / 2); fewer than 64 rows to a
// strided cell would leave the groups of 32 mostly padding.
inline int choose_cells(int64_t n, int64_t m) {
  const int64_t p = (n < m ? n : m) / 64 * 2;
  int P = 32;
  while (P * 2 <= p && P < kMaxCells) P *= 2;
  return P;
}

inline int64_t sort_blocks(int64_t rows) { return (rows + kChunkRows - 1) / kChunkRows; }
constexpr int kScanChunks = 256;   // chunks of a set from which their counters are scanned
// Kernels of one sort of points (the largest set: `rows`).
inline int sort_launches(int64_t rows) { return sort_blocks(rows) > kScanChunks ? 6 : 5; }
inline int group_cap(int64_t rows, int P, int size = 32) {
  return (int)((rows + size - 1) / size) + P;
}

// Scratch of one sort of B sets of `rows` rows: cell ids, block counts, farthest rows,
// the cells' numbers of rows.
struct SortScratch {
  size_t id, counts, far_, cell_rows, total;
};
// (rows: of the largest set; total: of all sets, 0: B rows)
inline SortScratch sort_scratch(int64_t B, int64_t rows, int P, int64_t total = 0) {
  SortScratch s{};
  s.counts = align256((size_t)(total > 0 ? total : B * rows));
  const size_t chunks =
      total > 0 ? (size_t)(total / kChunkRows + B) + 1 : (size_t)(B * sort_blocks(rows));
  s.far_ = s.counts + align256(chunks * P * 4);
  s.cell_rows = s.far_ + align256((size_t)B * (P / 2) * 8);
  s.total = s.cell_rows + align256((size_t)B * P * 4);
  return s;
}

// Sets of different sizes share one grid: run g of R rows belongs to the last set b whose
// first run, offs[b] / R + b, is not beyond g.  That leaves a set the runs it needs and at
// most one more, so total / R + B blocks serve them all however the sizes are spread
// (B times the largest set's runs would be mostly empty).  Returns the set, *run its run.
template <int R>
__device__ __forceinline__ int set_of_run(const int64_t* __restrict__ offs, int B, int64_t g,
                                          int* run) {
  int lo = 0, hi = B - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(offs + mid) / R + mid <= g) lo = mid;
    else hi = mid - 1;
  }
  *run = (int)(g - (__ldg(offs + lo) / R + lo));
  return lo;
}
template <int R>
inline int64_t runs_of_sets(int64_t total, int B) {
  return total / R + B;
}

// Sorts B sets of nrows rows of DP values (set b at src + b nrows DP) into P
// cells each.  points: the rows make the pivots, and the cells' means ctr
// [B][P][DP], their number npiv [B] and radii rad [B][P] are written; else (seeds)
// ctr and npiv are read.  Writes dst
// (sorted rows), start [B][P + 1] and, where non-null, perm (sorted position -> row
// of the set) and the table of groups [B][group_cap(nrows, P)].  Sets of different
// sizes: set b has the rows [offs[b], offs[b + 1]) of `total` (offs on the device),
// nrows is the largest, and there is no table.  The groups of the table hold up to
// `group` rows, group_cell (nullable) is the cell of each.  Nothing is done where the gate
// is closed.
template <typename T>
cudaError_t launch_sort(const T* src, int B, int64_t nrows, int DP, bool points, int P,
                        void* scratch, T* dst, int32_t* perm, int32_t* start, T* ctr,
                        int32_t* npiv, T* rad, int2* table, cudaStream_t st,
                        const int64_t* offs = nullptr, int64_t total = 0, int group = 32,
                        int32_t* group_cell = nullptr, Gate gate = Gate{});

// The extents of the P cells of one sorted set towards each other's centres
// (View::ext), for d > 8.
cudaError_t launch_extents(const float* rows, int DP, int P, const int32_t* npiv,
                           const int32_t* start, const float* ctr, float2* ext, cudaStream_t st,
                           Gate gate = Gate{});

}  // namespace cells

// ---- k_step_tc.cu: tiles of one cell each (up to 128 rows)
size_t tc_tile_images(int64_t tiles, int d);
// gate closed: tiles of the unsorted rows Xu, as launch_tc_pack.
cudaError_t launch_tc_pack_table(const float* Xs, const float* Xu, int64_t n, int d, int DP,
                                 const int2* table, int tiles, unsigned char* img, Gate gate,
                                 cudaStream_t st);
// ctl and, gate closed, the list of all m seeds: (places, Cc chunks of one tile) or (m, C, Lc).
cudaError_t launch_coarse_setup(int32_t* active, int32_t m, IterCtl* ctl, int32_t C, int32_t Lc,
                                int32_t places, int32_t Cc, Gate gate, cudaStream_t st);
cudaError_t launch_tc_visible(const float* Ys, int DP, const int2* seed_table, int seed_tiles,
                              const int32_t* yperm, const cells::View<float>& cv,
                              const int2* tile_table, const int32_t* tile_cell, int tiles,
                              int32_t* list, int32_t* count, int32_t* active, int32_t* out_row,
                              cudaStream_t st, Gate gate = Gate{});

// ---- k_travel.cu: whole trajectories in one launch (rows of DP floats, scaled)

// One update of m seeds (Ys: sorted by perm), results in the caller's order and units.
cudaError_t launch_step_groups(const float* Xs, const cells::View<float>& cv, int n,
                               const float* Ys, const cells::Groups& gr, int m,
                               const int32_t* perm, int d, int DP, const float* seeds,
                               double inv_scale, float* out_seeds, float* out_wsum, int sms,
                               cudaStream_t st, Gate gate = Gate{});
// Every point a seed, DP = 4 or 8: states, hist and the densities at the last positions.
cudaError_t launch_travel_groups(const float* Xs, const cells::View<float>& cv, int n, int d, int DP,
                                 const cells::Groups& gr, const int32_t* perm, int kf,
                                 int max_iter, float tol2_s, float sphere_r, float* y, int32_t* it,
                                 int32_t* conv, int32_t* state, float* wlast, int32_t* hist,
                                 unsigned long long* evals, unsigned long long* score_evals,
                                 int sms, cudaStream_t st);
// The RUNNING seeds of [0, N) (N and target from rc where non-null) to
// convergence or the round's stop; *total: the sum of hist.
cudaError_t launch_travel_seeds(const float* Xs, const cells::View<float>& cv, int n, int d, int DP,
                                float* y, int32_t* it, int32_t* conv, int32_t* state, float* wlast,
                                int32_t* hist, int32_t* total, const RoundCtl* rc, int N,
                                int max_N, int target, int kf, int max_iter, float tol2_s,
                                float sphere_r, unsigned long long* evals, int sms,
                                cudaStream_t st);
cudaError_t launch_refine_seeds(const float* Xs, const cells::View<float>& cv, int n, int d, int DP,
                                const float* y, const int32_t* kept, const int32_t* accepted,
                                const int32_t* M_ptr, int max_M, double* ym, float* yf,
                                double* mscore, double tol2_s, int max_iter, int32_t* iters_out,
                                unsigned long long* evals, int kf, double sphere_r, int sms,
                                cudaStream_t st);

// The batched call (k_batched.cu): queue entries [0, *n_entries) of a list of (set,
// seed) pairs, taken in turn from *queue (zero on entry); set b's cells are at
// [b] of cv and its rows at p0_b.
struct SeedQueue {
  const int32_t* list;       // set b's entries from p0_b on: seed or mode slots
  const int64_t* list_off;   // [B + 1] entries before set b's
  const int64_t* n_entries;
  unsigned long long* queue;
  SetCtl* sc;
  int B;
};
cudaError_t launch_travel_queue(const float* Xs, const cells::View<float>& cv, int d, int DP,
                                const SeedQueue& q, float* y, int32_t* it, int32_t* conv,
                                int32_t* state, float* wlast, int max_iter, float tol2_s, int sms,
                                cudaStream_t st);
// W at every listed slot's position, to score[p0 + entry] or mscore[slot].
cudaError_t launch_density_queue(const float* Xs, const cells::View<float>& cv, int DP,
                                 const SeedQueue& q, const float* y, float* score, double* mscore,
                                 int sms, cudaStream_t st);
cudaError_t launch_refine_queue(const float* Xs, const cells::View<float>& cv, int d, int DP,
                                const SeedQueue& q, double* ym, float* yf, double* mscore,
                                double tol2_s, int max_iter, int32_t* iters_out, int sms,
                                cudaStream_t st);

// ---- k_unroll.cu (rows of DP values; seeds and points in sorted order)

// Updates u0 .. u0 + len - 1 of one checkpoint segment: positions before update
// u (u0 <= u <= u0 + len), and W, the weight shift and the mean squared distance of each update.
template <typename T>
struct USegment {
  const T* ck0;        // positions before update 0 (a checkpoint)
  const T* ck1;        // positions after the segment's last update (a checkpoint)
  const T* seg;        // positions before updates 1 .. last
  int64_t row_values;  // values of one set of positions
  int seg_len, u0, len;
  const T* W;          // row 0: update 0
  const T* Sh;
  const T* M2;
  __device__ const T* pos(int u) const {
    u += u0;
    return u == 0 ? ck0 : (u == seg_len ? ck1 : seg + (int64_t)(u - 1) * row_values);
  }
};

template <typename T>
cudaError_t unroll_forward_steps(const T* X, const cells::View<T>& cv, const T* Y0,
                                 const cells::Groups& gr, const UGeom& g, T c, int steps,
                                 int every, int slot0, T* pos, T* Wout, T* Sh, T* M2, cudaStream_t st);
// SD: len x [B m] x (2 DP + 4); bctr, breach: len x [B groups] x DP and x 1;
// dh_part: one per group; first: dX and dh_part are set, not added to.
template <typename T>
cudaError_t unroll_backward_segment(const T* X, const cells::View<T>& cv, const USegment<T>& sg,
                                    const cells::Groups& gx, const cells::Groups& gr,
                                    const UGeom& g, T c, T inv_h2, double inv_h3, const T* Gin,
                                    T* Gout, T* SD, T* bctr, T* breach, double* dh_part, T* dX,
                                    int first, cudaStream_t st);
// Entries of dh_part per set (groups of the seed-major pass; per_set: of 32 seeds).
template <typename T>
int unroll_seed_groups(int P, const UGeom& g, int per_set);
cudaError_t unroll_dh_sum(const double* dh_part, int B, int per_set, double* dh, cudaStream_t st);
template <typename T>
cudaError_t unroll_pack_rows(const T* src, int64_t rows, int per_set, int d, int DP,
                             const int32_t* perm, T* dst, cudaStream_t st);
template <typename T>
cudaError_t unroll_unpack_rows(const T* src, int64_t rows, int per_set, int d, int DP,
                               const int32_t* perm, T* dst, cudaStream_t st);

}  // namespace fms

// Whole trajectories in one launch.  Seeds do not depend on each other (Early
// Stopping only needs the counts of their convergence updates), so a block
// takes its seeds from their first update to convergence: no host round trip, no
// grid barrier and no active list between updates.  Points are sorted into cells
// (fms_cells.cuh) and a seed evaluates only the cells that its cutoff reaches.
//
//   step_groups    one update of many seeds: 32 seeds of one cell per group, one
//                  per lane, points staged in shared memory and broadcast
//   travel_groups  every point a seed (Alg. 1): the same groups, to convergence
//   travel_seeds   few seeds (Alg. 2): a block per seed, points over the lanes
//   refine_seeds   the refinement of merged modes, FP64 positions and sums
//   *_queue        the same for many sets (and the density at given positions): blocks
//                  take the next (set, seed) from a queue
//
// Measured on one GB300 against the kernels that took every pair, one launch an
// update: 20,011 seeds x 65,537 points x 32 (one update) 4.91 -> 0.77 ms, of which
// step_groups 0.53 (0.67 with the sums in registers, one block an SM); 200,000 x 3,
// every point a seed, 86 -> 12.4 to 23.8 ms by the input (its slowest seeds hold their
// groups; with the padding column evaluated 17.4 where it is 12.8); 2,000 x 2 (not
// sorted) 0.56 -> 0.16 ms; 65,536 x 32 with 128 to 512 seeds 2.96 -> 0.63 ms, of which
// the three travel_seeds 0.21 (0.25 with 8 warps a seed); 200,000 x 16 directions
// 1.45 -> 0.49 ms, of which the two travel_seeds 0.12 (0.14); 256 sets of 1,000 to
// 50,000 x 16 in one call (travel_queue, 4 warps a seed) 29.0 -> 5.2 ms.
#include "fms_team.cuh"

namespace fms {
namespace {

// Flat kernel: the window's exponent, widened by more than its FP32 rounding.
constexpr float kFlatCut = -kFlatT * 1.0001f;

template <int KF>
__device__ __forceinline__ float first_cut() {
  return KF == kKernelFlat ? kFlatCut : cells::kFirstCut;
}

// W and S of the group at y (acc[0], acc[1 + k]); `act` lanes decide the ball
// and the cutoff, which comes in as a guess and leaves as the one their smallest
// W asks for.  Returns the rows visited.  The first NX of the DP columns count (the
// others are zero padding): the loop is bound by instruction issue, 11 of them at
// three columns, 15 at four.
template <int DP, int KF, int PH, int SUMS, int NA>
__device__ __forceinline__ int group_pass(const float* __restrict__ Xs, const View<float>& cv, int n,
                                          const float (&y)[DP], bool act, float log2n, float& cut,
                                          const TeamSmem<float, DP, SUMS>& sm, int w, int W,
                                          int lane, float (&acc)[NA]) {
  constexpr int NX = NA - 1;
  // The sums over tiles: 33 registers of wide rows, or, once a tile, the warp's part of
  // the team's exchange, so that two blocks of 8 warps fit an SM (163 -> 128 registers).
  constexpr bool kSmemSums = DP >= 32 && PH == 1;
  auto add_to = [&](int k) -> float& {
    if constexpr (kSmemSums) return sm.sums[(w * SUMS + k) * 32 + lane];
    else return acc[k];
  };
  int rows = 0;
  for (int pass = 0;; ++pass) {
    float reach;
    const int nl = visible_cells<float, DP>(cv, 0, n, y, act, sqrtf(cut), &reach, nullptr, sm, w,
                                            W, lane);
    if (cv.P == 0) rows = lane == 0 ? n : 0;
    else
      for (int i = lane; i < nl; i += 32) rows += sm.list[i].y;
#pragma unroll
    for (int k = 0; k <= NX; ++k) add_to(k) = 0.0f;
    sm.walk(Xs, n, nl, w, W, lane, [&](const float* tile, int nr) {
      float ta[NX + 1];
#pragma unroll
      for (int k = 0; k <= NX; ++k) ta[k] = 0.0f;
      constexpr int UNROLL = DP <= 4 ? 8 : (DP <= 8 ? 4 : (DP <= 16 ? 2 : 1));
      tile_rows<DP, PH, UNROLL>(tile, nr, lane, [&](const float* row, bool in) {
        float x[DP];
        smem_row<DP>(row, x);
        x[0] -= y[0];
        float t = -x[0] * x[0];
#pragma unroll
        for (int k = 1; k < NX; ++k) {
          x[k] -= y[k];
          t = fmaf(-x[k], x[k], t);
        }
        const float wt = in ? kweight<KF>(t) : 0.0f;
        ta[0] += wt;
#pragma unroll
        for (int k = 0; k < NX; ++k) ta[1 + k] = fmaf(wt, x[k], ta[1 + k]);
      });
#pragma unroll
      for (int k = 0; k <= NX; ++k) add_to(k) += ta[k];
    });
    if constexpr (kSmemSums) {
      team_total<32>(acc, sm.sums, SUMS, W, lane);
    } else {
      phase_sum<PH>(acc);
      team_sum<32 / PH>(acc, sm.sums, SUMS, w, W, lane);
    }
    if (KF == kKernelFlat || cv.P == 0) break;
    const float need = cells::cut_bits(cells::warp_min(act ? acc[0] : INFINITY), log2n);
    if (!(need > cut) || cut >= cells::zero_bits<float>()) {
      cut = cells::widen(need);   // (W does not decrease along a trajectory)
      break;
    }
    cut = pass == 0 ? cells::widen(need) : cells::zero_bits<float>();
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) rows += __shfl_xor_sync(kFull, rows, o);
  return rows;
}

// out = seed + (S / W) / scale in the caller's order and units, as in step_finish.
template <int DP, int NX>
__global__ void __launch_bounds__(256, 2)
    step_groups(const float* __restrict__ Xs, View<float> cv, int n, const float* __restrict__ Ys,
                Groups gr, int m, const int32_t* __restrict__ perm, int d, const float* seeds,
                double inv_scale, float* out_seeds, float* __restrict__ out_wsum, Gate gate) {
  wait_for_previous();
  if (!gate.open()) return;
  extern __shared__ __align__(16) unsigned char travel_smem[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, W = blockDim.x >> 5;
  const TeamSmem<float, DP, DP + 1> sm(travel_smem, w, W);
  int row0, cnt;
  if (!group_rows(gr, 0, blockIdx.x, m, &row0, &cnt)) return;
  const int e = row0 + min(lane, cnt - 1);
  float y[DP], acc[NX + 1];
  load_row<DP>(Ys + (int64_t)e * DP, y);
  const float log2n = log2f((float)n);
  float cut = first_cut<kKernelGaussian>();
  group_pass<DP, kKernelGaussian, 1>(Xs, cv, n, y, true, log2n, cut, sm, w, W, lane, acc);
  if (w != 0 || lane >= cnt) return;
  const int64_t i = perm[e];
#pragma unroll
  for (int k = 0; k < NX; ++k)
    if (k < d)
      out_seeds[i * d + k] =
          (float)((double)seeds[i * d + k] + (double)(acc[1 + k] / acc[0]) * inv_scale);
  if (out_wsum) out_wsum[i] = acc[0];
}

// Every point a seed, slot = the point's row in the caller's order (perm; null:
// unsorted): updates until it converges, fails or has made max_iter of them, then
// the density at its last position (wlast).  hist counts the convergence updates.
template <int DP, int NX, int KF, int PH>
__global__ void __launch_bounds__(512)
    travel_groups(const float* __restrict__ Xs, View<float> cv, int n, Groups gr,
                  const int32_t* __restrict__ perm, int max_iter, float tol2_s, float sphere_r,
                  float* __restrict__ y_out, int32_t* __restrict__ it_out,
                  int32_t* __restrict__ conv, int32_t* __restrict__ state,
                  float* __restrict__ wlast, int32_t* __restrict__ hist,
                  unsigned long long* evals, unsigned long long* score_evals, int resident) {
  extern __shared__ __align__(16) unsigned char travel_smem[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, W = blockDim.x >> 5;
  constexpr int GS = 32 / PH;   // seeds of a group
  int row0, cnt;
  if (!group_rows(gr, 0, blockIdx.x, n, &row0, &cnt, GS)) return;
  const TeamSmem<float, DP, DP + 1> sm(travel_smem, w, W, Xs, resident ? n : 0);
  const int e = row0 + min(lane % GS, cnt - 1);
  float y[DP], acc[NX + 1];
  load_row<DP>(Xs + (int64_t)e * DP, y);
  const float log2n = log2f((float)n);
  float cut = first_cut<KF>(), wl = 0.0f;
  bool act = lane % GS < cnt;
  int it = 0, cu = -1, stt = kRunning;
  unsigned long long ev = 0;
  for (;;) {
    const unsigned live = __ballot_sync(kFull, act);   // the same for every warp of the team
    if (!live) break;
    const int rows = group_pass<DP, KF, PH>(Xs, cv, n, y, act, log2n, cut, sm, w, W, lane, acc);
    ev += (unsigned long long)rows * (__popc(live) / PH);
    if (!act) continue;
    wl = acc[0];
    ++it;
    bool ok = (wl > 0.0f) && isfinite(wl);
    float dl[NX], step2 = 0.0f;
#pragma unroll
    for (int k = 0; k < NX; ++k) {
      dl[k] = ok ? acc[1 + k] / wl : 0.0f;
      step2 = fmaf(dl[k], dl[k], step2);
    }
    ok = ok && isfinite(step2);
    if (ok && sphere_r > 0.0f) {
      float nn = 0.0f;
#pragma unroll
      for (int k = 0; k < NX; ++k) {
        dl[k] += y[k];
        nn = fmaf(dl[k], dl[k], nn);
      }
      const float f = sphere_r / sqrtf(nn);
      step2 = 0.0f;
#pragma unroll
      for (int k = 0; k < NX; ++k) {
        dl[k] = dl[k] * f - y[k];
        step2 = fmaf(dl[k], dl[k], step2);
      }
      ok = nn > 0.0f && isfinite(step2);
    }
    if (ok) {
#pragma unroll
      for (int k = 0; k < NX; ++k) y[k] += dl[k];
    }
    if (!ok) {
      stt = kFailed;
    } else if (step2 <= tol2_s) {
      stt = kConverged;
      cu = it;
    } else if (it >= max_iter) {
      stt = kExhausted;
    }
    act = stt == kRunning;
  }
  const bool fine = lane % GS < cnt && stt != kFailed;
  unsigned long long sev = 0;
  if (__any_sync(kFull, fine)) {
    const int rows = group_pass<DP, KF, PH>(Xs, cv, n, y, fine, log2n, cut, sm, w, W, lane, acc);
    sev = (unsigned long long)rows * (__popc(__ballot_sync(kFull, fine)) / PH);
    wl = acc[0];
  }
  if (w != 0) return;
  if (lane < cnt) {
    const int64_t s = perm ? perm[e] : e;
    store_row<float, DP>(y_out + s * DP, y);
    it_out[s] = it;
    conv[s] = cu;
    state[s] = stt;
    wlast[s] = wl;
    if (cu > 0) atomicAdd(&hist[cu], 1);
  }
  if (lane == 0) {
    atomicAdd(evals, ev);
    atomicAdd(score_evals, sev);
  }
}

// ---------------------------------------------------------------------------
// A block per seed: its NW warps split the visible rows, LP = DP / 4 lanes to a
// row (four coordinates each), so row-major rows are read as whole 128-byte
// lines.  Bound by L2 bandwidth (4 DP bytes a row and seed).
// ---------------------------------------------------------------------------
constexpr int kSeedWarps = 16;   // one set: as many warps as the seeds leave idle
constexpr int kQueueWarps = 4;   // many sets: more seeds in flight instead

template <int DP, typename ST, int NW>
struct SeedSmem {
  float y[DP];
  int2 list[cells::kMaxCells];
  unsigned mask[cells::kMaxCells / 32 > NW ? cells::kMaxCells / 32 : NW], near[NW];
  ST red[NW][DP + 1];
  ST tot[DP + 1];
  ST part[NW][5][32];   // a lane's sums
  float cut;
  int flag;
};

// tot = (W, S) at sh.y over the cells within the cutoff sh.cut; returns the
// rows visited.  Ends with a block barrier.
template <int DP, int KF, typename ST, int NW>
__device__ int seed_pass(const float* __restrict__ Xs, const View<float>& cv, int n,
                         SeedSmem<DP, ST, NW>& sh) {
  constexpr int LP = DP / 4, PPW = 32 / LP, UN = LP == 1 ? 4 : 8, CH = PPW * UN;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int nl = 0;
  if (cv.P == 0) {
    if (threadIdx.x == 0) sh.list[0] = make_int2(0, n);
    nl = 1;
    __syncthreads();
  } else {
    constexpr int U = (cells::kMaxCells / 32 + NW - 1) / NW;   // cells of a thread
    const float rc = sqrtf(sh.cut);
    float a[U], far_[U];   // distance of the cell's centre, reach of its rows from there
    int2 mine[U];
    unsigned best = 0xffffffffu;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int p = (u * NW + w) * 32 + lane;
      mine[u] = make_int2(0, 0);
      a[u] = far_[u] = 0.0f;
      if (p >= cv.P) continue;
      const float4* q = reinterpret_cast<const float4*>(cv.ctr + (int64_t)p * DP);
      float d2 = 0.0f;
#pragma unroll
      for (int k = 0; k < LP; ++k) {
        const float4 v = __ldg(q + k);
        const float4 yy = reinterpret_cast<const float4*>(sh.y)[k];
        float t = v.x - yy.x;
        d2 = fmaf(t, t, d2);
        t = v.y - yy.y;
        d2 = fmaf(t, t, d2);
        t = v.z - yy.z;
        d2 = fmaf(t, t, d2);
        t = v.w - yy.w;
        d2 = fmaf(t, t, d2);
      }
      mine[u].x = cv.start[p];
      mine[u].y = cv.start[p + 1] - mine[u].x;
      a[u] = sqrtf(d2);
      far_[u] = cv.rad[p];
      if (mine[u].y > 0) best = min(best, (__float_as_uint(a[u]) & ~255u) | (unsigned)p);
    }
    if (cv.ext) {   // (the same for the whole block)
      best = __reduce_min_sync(kFull, best);
      if (lane == 0) sh.near[w] = best;
      __syncthreads();
#pragma unroll
      for (int u = 0; u < NW; ++u) best = min(best, sh.near[u]);
      const int q = (int)(best & 255u);
      // (the cut-off bits of the distance count as set)
      const float delta = __uint_as_float(best | 255u);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (mine[u].y > 0)
          far_[u] = cells::reach_towards(far_[u], cv.ext[q * cv.P + (u * NW + w) * 32 + lane],
                                         a[u], delta);
    }
    bool see[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      see[u] = mine[u].y > 0 && !(a[u] > (rc + far_[u]) * 1.0001f);
      const unsigned mk = __ballot_sync(kFull, see[u]);
      if (lane == 0) sh.mask[u * NW + w] = mk;
    }
    __syncthreads();
#pragma unroll
    for (int g = 0; g < cells::kMaxCells / 32; ++g) {
      const unsigned m = sh.mask[g];
      if (g % NW == w && see[g / NW]) sh.list[nl + __popc(m & ((1u << lane) - 1u))] = mine[g / NW];
      nl += __popc(m);
    }
    __syncthreads();
  }
  const int part = lane % LP, pl = lane / LP;
  const float4 y4 = reinterpret_cast<const float4*>(sh.y)[part];
  // FP32 sums of at most kFlush steps (64 or 128 rows of a lane), then added to totals of
  // type ST in shared memory: one chain over all of a lane's rows would round a sum of
  // 10^5 terms in FP32.  (Totals in registers cost 256 sets of 16-D 2.8 -> 3.1 ms.)
  constexpr int kFlush = 16;
  float aw = 0.0f;
  float4 as = make_float4(0.f, 0.f, 0.f, 0.f);
  int rows = 0, t = w, steps = 0;
  const float4* X4 = reinterpret_cast<const float4*>(Xs);
  for (int v = 0; v < nl; ++v) {
    const int2 c = sh.list[v];
    rows += c.y;
    const int nt = (c.y + CH - 1) / CH;
    for (; t < nt; t += NW) {
      float4 x[UN];
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const int r = t * CH + u * PPW + pl;
        // past the end: so far away that the weight is exactly zero
        x[u] = r < c.y ? __ldg(X4 + (int64_t)(c.x + r) * LP + part)
                       : make_float4(1e18f, 1e18f, 1e18f, 1e18f);
      }
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        x[u].x -= y4.x;
        x[u].y -= y4.y;
        x[u].z -= y4.z;
        x[u].w -= y4.w;
        float q = -x[u].x * x[u].x;
        q = fmaf(-x[u].y, x[u].y, q);
        q = fmaf(-x[u].z, x[u].z, q);
        q = fmaf(-x[u].w, x[u].w, q);
#pragma unroll
        for (int o = 1; o < LP; o <<= 1) q += __shfl_xor_sync(kFull, q, o);
        const float wt = kweight<KF>(q);
        aw += wt;
        as.x = fmaf(wt, x[u].x, as.x);
        as.y = fmaf(wt, x[u].y, as.y);
        as.z = fmaf(wt, x[u].z, as.z);
        as.w = fmaf(wt, x[u].w, as.w);
      }
      if (++steps % kFlush == 0) {
        const float a[5] = {aw, as.x, as.y, as.z, as.w};
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          ST& q = sh.part[w][k][lane];
          q = (steps > kFlush ? q : ST(0)) + (ST)a[k];
        }
        aw = 0.0f;
        as = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    t -= nt;
  }
  ST s[5] = {(ST)aw, (ST)as.x, (ST)as.y, (ST)as.z, (ST)as.w};
  if (steps >= kFlush) {
#pragma unroll
    for (int k = 0; k < 5; ++k) s[k] += sh.part[w][k][lane];
  }
#pragma unroll
  for (int k = 0; k < 5; ++k)
#pragma unroll
    for (int o = LP; o < 32; o <<= 1) s[k] += __shfl_xor_sync(kFull, s[k], o);
  if (pl == 0) {
    if (part == 0) sh.red[w][0] = s[0];
#pragma unroll
    for (int k = 0; k < 4; ++k) sh.red[w][1 + part * 4 + k] = s[1 + k];
  }
  __syncthreads();
  for (int k = threadIdx.x; k <= DP; k += blockDim.x) {
    ST a = sh.red[0][k];
#pragma unroll
    for (int u = 1; u < NW; ++u) a += sh.red[u][k];
    sh.tot[k] = a;
  }
  __syncthreads();
  return rows;
}

// Passes until the cutoff covers the W that came out (see fms_cells.cuh).
template <int DP, int KF, typename ST, int NW>
__device__ long long seed_sums(const float* __restrict__ Xs, const View<float>& cv, int n,
                               float log2n, SeedSmem<DP, ST, NW>& sh) {
  long long rows = 0;
  for (int pass = 0;; ++pass) {
    rows += seed_pass<DP, KF, ST, NW>(Xs, cv, n, sh);
    if (KF == kKernelFlat || cv.P == 0) return rows;
    const float need = cells::cut_bits((float)sh.tot[0], log2n);
    const float cut = sh.cut;
    const bool again = need > cut && cut < cells::zero_bits<float>();
    __syncthreads();   // every thread has read sh.cut
    if (threadIdx.x == 0)
      sh.cut = again && pass > 0 ? cells::zero_bits<float>() : cells::widen(need);
    __syncthreads();
    if (!again) return rows;
  }
}

// One RUNNING seed to convergence, failure, max_iter updates or the round's stop.
// seen(): seeds converged so far; stop(t): whether the convergence counts say that
// the round ends at or before update t (warp 0 calls; the counts only grow, so a
// stop can come late, never early); converged(t): counts this one.
// Returns the rows visited (10 million points and some hundred updates pass 2^31).
template <int DP, int KF, int NW, typename Seen, typename Stop, typename Conv>
__device__ long long travel_seed(const float* __restrict__ Xs, const View<float>& cv, int n, int d,
                                 int64_t s, float* y, int32_t* it, int32_t* conv, int32_t* state,
                                 float* wlast, int target, int max_iter, float tol2_s,
                                 float sphere_r, SeedSmem<DP, float, NW>& sh, Seen&& seen_,
                                 Stop&& stop_, Conv&& conv_) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const float log2n = log2f((float)n);
  __syncthreads();   // the previous seed's values are no longer read
  for (int k = threadIdx.x; k < DP; k += blockDim.x) sh.y[k] = y[s * DP + k];
  int done = it[s];
  long long rows = 0;
  // A seed that an earlier round's stop left goes on with the cutoff that it had: when it
  // noticed the stop depends on timing, and its later updates must not.
  if (threadIdx.x == 0)
    sh.cut = done > 0 && KF != kKernelFlat ? cells::widen(cells::cut_bits(wlast[s], log2n))
                                           : first_cut<KF>();
  __syncthreads();
  for (;;) {
    int seen = 0;   // (read ahead of the pass that hides it)
    if (w == 0) seen = __shfl_sync(kFull, seen_(), 0);
    rows += seed_sums<DP, KF, float, NW>(Xs, cv, n, log2n, sh);
    ++done;
    if (w == 0) {
      const float W = sh.tot[0];
      bool ok = (W > 0.0f) && isfinite(W);
      constexpr int KL = (DP + 31) / 32;
      float p[KL], dl[KL], step2 = 0.0f;
#pragma unroll
      for (int u = 0; u < KL; ++u) {
        const int k = lane + 32 * u;
        p[u] = k < DP ? sh.y[k] : 0.0f;
        dl[u] = ok && k < d ? sh.tot[1 + k] / W : 0.0f;
        step2 = fmaf(dl[u], dl[u], step2);
      }
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) step2 += __shfl_xor_sync(kFull, step2, o);
      ok = ok && isfinite(step2);
      if (ok && sphere_r > 0.0f) {
        float nn = 0.0f;
#pragma unroll
        for (int u = 0; u < KL; ++u) {
          dl[u] += p[u];
          nn = fmaf(dl[u], dl[u], nn);
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) nn += __shfl_xor_sync(kFull, nn, o);
        const float f = sphere_r / sqrtf(nn);
        step2 = 0.0f;
#pragma unroll
        for (int u = 0; u < KL; ++u) {
          const float q = dl[u] * f, g = q - p[u];
          step2 = fmaf(g, g, step2);
          dl[u] = q;   // the new position
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) step2 += __shfl_xor_sync(kFull, step2, o);
        ok = nn > 0.0f && isfinite(step2);
      } else {
#pragma unroll
        for (int u = 0; u < KL; ++u) dl[u] += p[u];
      }
      int now = kRunning;
      if (!ok) now = kFailed;
      else if (step2 <= tol2_s) now = kConverged;
      else if (done >= max_iter) now = kExhausted;
      const bool stop = now == kRunning && seen >= target && stop_(done);
#pragma unroll
      for (int u = 0; u < KL; ++u) {
        const int k = lane + 32 * u;
        if (ok && k < DP) sh.y[k] = dl[u];
      }
      if (lane == 0) {
        if (now == kConverged) {
          conv[s] = done;
          conv_(done);
        }
        if (now != kRunning || stop) {
          it[s] = done;
          state[s] = now;
          wlast[s] = W;
        }
        sh.flag = (now != kRunning || stop) ? 1 : 0;
      }
      __syncwarp();
    }
    __syncthreads();
    if (sh.flag) break;
  }
  for (int k = threadIdx.x; k < DP; k += blockDim.x) y[s * DP + k] = sh.y[k];
  return rows;
}

// The RUNNING seeds of [0, N); hist counts convergence updates, *total sums it.
template <int DP, int KF>
__global__ void __launch_bounds__(kSeedWarps * 32)
    travel_seeds(const float* __restrict__ Xs, View<float> cv, int n, int d, float* y,
                 int32_t* it, int32_t* conv, int32_t* state, float* wlast, int32_t* hist,
                 int32_t* total, const RoundCtl* __restrict__ rc, int N_arg, int target_arg,
                 int max_iter, float tol2_s, float sphere_r, unsigned long long* evals) {
  __shared__ __align__(16) SeedSmem<DP, float, kSeedWarps> sh;
  const int N = rc ? rc->N : N_arg, target = rc ? rc->target : target_arg;
  const int lane = threadIdx.x & 31;
  unsigned long long ev = 0;
  for (int s = blockIdx.x; s < N; s += gridDim.x) {
    if (state[s] != kRunning) continue;
    ev += (unsigned long long)travel_seed<DP, KF, kSeedWarps>(
        Xs, cv, n, d, s, y, it, conv, state, wlast, target, max_iter, tol2_s, sphere_r, sh,
        [&] { return *(volatile int32_t*)total; },
        [&](int t) {
          int c = 0;
          for (int b = 0; b <= t; b += 32)
            if (b + lane <= t) c += *(volatile int32_t*)(hist + b + lane);
#pragma unroll
          for (int o = 16; o >= 1; o >>= 1) c += __shfl_xor_sync(kFull, c, o);
          return c >= target;
        },
        [&](int t) {
          atomicAdd(&hist[t], 1);
          atomicAdd(total, 1);
        });
  }
  if (threadIdx.x == 0 && ev) atomicAdd(evals, ev);
}

// ---- many sets: a queue of (set, seed) entries

__device__ __forceinline__ int queue_set(const int64_t* __restrict__ off, int B, int64_t x) {
  int lo = 0, hi = B - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(off + mid) <= x) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

template <int DP>
__device__ __forceinline__ View<float> set_view(const View<float>& cv, int b) {
  View<float> v = cv;
  if (cv.P == 0) return v;
  v.start += (int64_t)b * (cv.P + 1);
  v.ctr += (int64_t)b * cv.P * DP;
  v.rad += (int64_t)b * cv.P;
  return v;
}

// The block's next entry: its set and place in the set's list; false at the end.
__device__ __forceinline__ bool next_entry(const SeedQueue& q, int* set, int* at) {
  __shared__ long long sh_e;
  __syncthreads();
  if (threadIdx.x == 0) sh_e = (long long)atomicAdd(q.queue, 1ull);
  __syncthreads();
  const int64_t e = sh_e;
  if (e >= *q.n_entries) return false;
  *set = queue_set(q.list_off, q.B, e);
  *at = (int)(e - q.list_off[*set]);
  return true;
}

template <int DP>
__global__ void __launch_bounds__(kQueueWarps * 32, 5)   // (121 registers: 4 blocks an SM)
    travel_queue(const float* __restrict__ Xs, View<float> cv, int d, SeedQueue q, float* y,
                 int32_t* it, int32_t* conv, int32_t* state, float* wlast, int max_iter,
                 float tol2_s) {
  __shared__ __align__(16) SeedSmem<DP, float, kQueueWarps> sh;
  const int lane = threadIdx.x & 31;
  int b, at;
  while (next_entry(q, &b, &at)) {
    SetCtl* c = q.sc + b;
    const int p0 = c->p0, N = c->N, target = c->target;
    const long long rows = travel_seed<DP, kKernelGaussian, kQueueWarps>(
        Xs + (int64_t)p0 * DP, set_view<DP>(cv, b), c->n, d, q.list[p0 + at], y, it, conv, state,
        wlast, target, max_iter, tol2_s, 0.0f, sh,
        [&] { return *(volatile int32_t*)&c->total; },
        [&](int t) {
          int k = 0;
          for (int i = lane; i < N; i += 32) {
            const int v = *(volatile int32_t*)(conv + p0 + i);
            k += v > 0 && v <= t ? 1 : 0;
          }
#pragma unroll
          for (int o = 16; o >= 1; o >>= 1) k += __shfl_xor_sync(kFull, k, o);
          return k >= target;
        },
        [&](int) { atomicAdd(&c->total, 1); });
    if (threadIdx.x == 0)
      atomicAdd(reinterpret_cast<unsigned long long*>(&c->evals), (unsigned long long)rows);
  }
}

template <int DP>
__global__ void __launch_bounds__(kQueueWarps * 32)
    density_queue(const float* __restrict__ Xs, View<float> cv, SeedQueue q,
                  const float* __restrict__ y, float* __restrict__ score,
                  double* __restrict__ mscore) {
  __shared__ __align__(16) SeedSmem<DP, double, kQueueWarps> sh;
  int b, at;
  while (next_entry(q, &b, &at)) {
    SetCtl* c = q.sc + b;
    const int64_t s = q.list[c->p0 + at];
    __syncthreads();
    for (int k = threadIdx.x; k < DP; k += blockDim.x) sh.y[k] = y[s * DP + k];
    if (threadIdx.x == 0) sh.cut = first_cut<kKernelGaussian>();
    __syncthreads();
    const long long rows = seed_sums<DP, kKernelGaussian, double, kQueueWarps>(
        Xs + (int64_t)c->p0 * DP, set_view<DP>(cv, b), c->n, log2f((float)c->n), sh);
    if (threadIdx.x == 0) {
      if (score) score[c->p0 + at] = (float)sh.tot[0];
      if (mscore) mscore[s] = sh.tot[0];
      atomicAdd(reinterpret_cast<unsigned long long*>(&c->evals), (unsigned long long)rows);
    }
  }
}

// The refinement of one mode from sh.y: ym <- ym + S/W - (ym - fl32(ym)) until
// ||step|| <= tol or max_iter updates; the position (and the sums over lanes) in
// FP64, the density is W of the last update.  Returns the updates made.
template <int DP, int KF, int NW>
__device__ int refine_seed(const float* __restrict__ Xs, const View<float>& cv, int n, int d,
                           double* ym, float* yf, double* mscore, double tol2_s, int max_iter,
                           double sphere_r, SeedSmem<DP, double, NW>& sh, unsigned long long& ev) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const float log2n = log2f((float)n);
  constexpr int KL = (DP + 31) / 32;
  if (threadIdx.x == 0) sh.cut = first_cut<KF>();
  __syncthreads();
  double p[KL], W = 0.0;   // warp 0: the position
#pragma unroll
  for (int u = 0; u < KL; ++u) p[u] = lane + 32 * u < DP ? (double)sh.y[lane + 32 * u] : 0.0;
  int iters = 0;
  for (; iters < max_iter;) {
    ev += (unsigned long long)seed_sums<DP, KF, double, NW>(Xs, cv, n, log2n, sh);
    ++iters;
    if (w == 0) {
      W = sh.tot[0];
      bool ok = W > 0.0 && isfinite(W);
      double q[KL], step2 = 0.0;
#pragma unroll
      for (int u = 0; u < KL; ++u) {
        const int k = lane + 32 * u;
        const double dl = ok && k < d ? sh.tot[1 + k] / W - (p[u] - (double)sh.y[k]) : 0.0;
        step2 += dl * dl;
        q[u] = p[u] + dl;
      }
      if (ok && sphere_r > 0.0) {
        double nn = 0.0;
#pragma unroll
        for (int u = 0; u < KL; ++u) nn += q[u] * q[u];
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) nn += __shfl_xor_sync(kFull, nn, o);
        const double f = sphere_r / sqrt(nn);
        step2 = 0.0;
#pragma unroll
        for (int u = 0; u < KL; ++u) {
          q[u] *= f;
          step2 += (q[u] - p[u]) * (q[u] - p[u]);
        }
        ok = nn > 0.0;
      }
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) step2 += __shfl_xor_sync(kFull, step2, o);
      ok = ok && isfinite(step2);
#pragma unroll
      for (int u = 0; u < KL; ++u) {
        const int k = lane + 32 * u;
        if (ok) p[u] = q[u];
        if (ok && k < DP) sh.y[k] = (float)q[u];
      }
      if (lane == 0) sh.flag = (!ok || step2 <= tol2_s) ? 1 : 0;
      __syncwarp();
    }
    __syncthreads();
    if (sh.flag) break;
  }
  if (w == 0) {
#pragma unroll
    for (int u = 0; u < KL; ++u) {
      const int k = lane + 32 * u;
      if (k < DP) {
        ym[k] = p[u];
        yf[k] = (float)p[u];
      }
    }
    if (lane == 0) *mscore = W;
  }
  return iters;
}

template <int DP, int KF>
__global__ void __launch_bounds__(kSeedWarps * 32)
    refine_seeds(const float* __restrict__ Xs, View<float> cv, int n, int d,
                 const float* __restrict__ y, const int32_t* __restrict__ kept,
                 const int32_t* __restrict__ accepted, const int32_t* __restrict__ M_ptr,
                 double* __restrict__ ym, float* __restrict__ yf, double* __restrict__ mscore,
                 double tol2_s, int max_iter, int32_t* iters_out, unsigned long long* evals,
                 double sphere_r) {
  __shared__ __align__(16) SeedSmem<DP, double, kSeedWarps> sh;
  const int M = *M_ptr;
  unsigned long long ev = 0;
  for (int m = blockIdx.x; m < M; m += gridDim.x) {
    const int64_t src = kept[accepted[m]];
    __syncthreads();
    for (int k = threadIdx.x; k < DP; k += blockDim.x) sh.y[k] = y[src * DP + k];
    const int iters = refine_seed<DP, KF, kSeedWarps>(Xs, cv, n, d, ym + (int64_t)m * DP,
                                                      yf + (int64_t)m * DP, mscore + m, tol2_s,
                                                      max_iter, sphere_r, sh, ev);
    if (threadIdx.x == 0) atomicMax(iters_out, iters);
  }
  if (threadIdx.x == 0 && ev) atomicAdd(evals, ev);
}

// The modes at the slots of the queue's list, from yf.
template <int DP>
__global__ void __launch_bounds__(kQueueWarps * 32)
    refine_queue(const float* __restrict__ Xs, View<float> cv, int d, SeedQueue q, double* ym,
                 float* yf, double* mscore, double tol2_s, int max_iter, int32_t* iters_out) {
  __shared__ __align__(16) SeedSmem<DP, double, kQueueWarps> sh;
  int b, at;
  while (next_entry(q, &b, &at)) {
    SetCtl* c = q.sc + b;
    const int64_t s = q.list[c->p0 + at];
    __syncthreads();
    for (int k = threadIdx.x; k < DP; k += blockDim.x) sh.y[k] = yf[s * DP + k];
    unsigned long long ev = 0;
    const int iters = refine_seed<DP, kKernelGaussian, kQueueWarps>(
        Xs + (int64_t)c->p0 * DP, set_view<DP>(cv, b), c->n, d, ym + s * DP, yf + s * DP,
        mscore + s, tol2_s, max_iter, 0.0, sh, ev);
    if (threadIdx.x == 0) {
      atomicMax(iters_out, iters);
      atomicAdd(reinterpret_cast<unsigned long long*>(&c->evals), ev);
    }
  }
}

int seed_grid(int max_seeds, int sms) {
  const int g = sms * 2;   // (resident blocks; each takes its seeds in turn)
  return max_seeds < g ? (max_seeds > 0 ? max_seeds : 1) : g;
}

}  // namespace

// RUN(padded width, columns that count) for d <= 8.
#define FMS_BY_COLUMNS(RUN)   \
  switch (d) {                \
    case 1:                   \
    case 2: RUN(4, 2)         \
    case 3: RUN(4, 3)         \
    case 4: RUN(4, 4)         \
    case 5:                   \
    case 6: RUN(8, 6)         \
    case 7:                   \
    case 8: RUN(8, 8)         \
  }

cudaError_t launch_step_groups(const float* Xs, const View<float>& cv, int n, const float* Ys,
                               const Groups& gr, int m, const int32_t* perm, int d, int DP,
                               const float* seeds, double inv_scale, float* out_seeds,
                               float* out_wsum, int sms, cudaStream_t st, Gate gate) {
#define FMS_STEP_GROUPS(DP_, NX_)                                                                \
  {                                                                                              \
    constexpr int ws = team_warp_smem<float, DP_, DP_ + 1>();                                    \
    const int W = team_warps(gr.per_set, sms, ws);                                               \
    const int smem = group_team_smem<float, DP_, DP_ + 1>(W);                                    \
    const cudaError_t e = team_attr(step_groups<DP_, NX_>, smem);                                \
    if (e != cudaSuccess) return e;                                                              \
    return launch_gated(gate, step_groups<DP_, NX_>, gr.per_set, 32 * W, smem, st, Xs, cv, n,   \
                        Ys, gr, m, perm, d, seeds, inv_scale, out_seeds, out_wsum, gate);       \
  }
  FMS_BY_COLUMNS(FMS_STEP_GROUPS)
  switch (DP) {
    case 16: FMS_STEP_GROUPS(16, 16)
    case 32: FMS_STEP_GROUPS(32, 32)
  }
#undef FMS_STEP_GROUPS
  return cudaErrorInvalidValue;
}

template <int DP, int NX, int KF, int PH>
static cudaError_t travel_groups_t(const float* Xs, const View<float>& cv, int n, Groups gr,
                                   const int32_t* perm, int max_iter, float tol2_s,
                                   float sphere_r, float* y, int32_t* it, int32_t* conv,
                                   int32_t* state, float* wlast, int32_t* hist,
                                   unsigned long long* evals, unsigned long long* score_evals,
                                   int sms, cudaStream_t st) {
  if (PH > 1) gr.per_set = (n + 32 / PH - 1) / (32 / PH);
  constexpr int ws = team_warp_smem<float, DP, DP + 1>();
  // at least 4 warps: the last groups take many updates, with few others running
  const int W0 = team_warps(gr.per_set, sms, ws, 16), W = W0 < 4 ? 4 : W0;
  const bool res = team_resident<float, DP>(cv.P, n);
  const int smem =
      res ? resident_team_smem<float, DP, DP + 1>(W, n) : group_team_smem<float, DP, DP + 1>(W);
  const cudaError_t e = team_attr(travel_groups<DP, NX, KF, PH>, smem);
  if (e != cudaSuccess) return e;
  travel_groups<DP, NX, KF, PH><<<gr.per_set, 32 * W, smem, st>>>(
      Xs, cv, n, gr, perm, max_iter, tol2_s, sphere_r, y, it, conv, state, wlast, hist, evals,
      score_evals, res ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_travel_groups(const float* Xs, const View<float>& cv, int n, int d, int DP,
                                 const Groups& gr, const int32_t* perm, int kf, int max_iter,
                                 float tol2_s, float sphere_r, float* y, int32_t* it,
                                 int32_t* conv, int32_t* state, float* wlast, int32_t* hist,
                                 unsigned long long* evals, unsigned long long* score_evals,
                                 int sms, cudaStream_t st) {
#define FMS_TRAVEL_PH(DP_, NX_, KF_, PH_)                                                       \
  travel_groups_t<DP_, NX_, KF_, PH_>(Xs, cv, n, gr, perm, max_iter, tol2_s, sphere_r, y, it,   \
                                      conv, state, wlast, hist, evals, score_evals, sms, st)
#define FMS_TRAVEL(DP_, NX_)                                                                   \
  {                                                                                            \
    if (team_phases<float, DP_>(cv.P, n, sms) == 4)                                            \
      return kf ? FMS_TRAVEL_PH(DP_, NX_, 1, 4) : FMS_TRAVEL_PH(DP_, NX_, 0, 4);               \
    return kf ? FMS_TRAVEL_PH(DP_, NX_, 1, 1) : FMS_TRAVEL_PH(DP_, NX_, 0, 1);                 \
  }
  FMS_BY_COLUMNS(FMS_TRAVEL)
#undef FMS_TRAVEL
#undef FMS_TRAVEL_PH
  return cudaErrorInvalidValue;
}

cudaError_t launch_travel_seeds(const float* Xs, const View<float>& cv, int n, int d, int DP,
                                float* y, int32_t* it, int32_t* conv, int32_t* state,
                                float* wlast, int32_t* hist, int32_t* total, const RoundCtl* rc,
                                int N, int max_N, int target, int kf, int max_iter, float tol2_s,
                                float sphere_r, unsigned long long* evals, int sms,
                                cudaStream_t st) {
  const int g = seed_grid(max_N, sms);
#define FMS_SEEDS(DP_)                                                                           \
  if (kf)                                                                                        \
    travel_seeds<DP_, 1><<<g, kSeedWarps * 32, 0, st>>>(Xs, cv, n, d, y, it, conv, state, wlast, \
                                                        hist, total, rc, N, target, max_iter,    \
                                                        tol2_s, sphere_r, evals);                \
  else                                                                                           \
    travel_seeds<DP_, 0><<<g, kSeedWarps * 32, 0, st>>>(Xs, cv, n, d, y, it, conv, state, wlast, \
                                                        hist, total, rc, N, target, max_iter,    \
                                                        tol2_s, sphere_r, evals);                \
  return cudaGetLastError();
  switch (DP) {
    case 8: FMS_SEEDS(8)
    case 16: FMS_SEEDS(16)
    case 32: FMS_SEEDS(32)
    case 64: FMS_SEEDS(64)
  }
#undef FMS_SEEDS
  return cudaErrorInvalidValue;
}

cudaError_t launch_refine_seeds(const float* Xs, const View<float>& cv, int n, int d, int DP,
                                const float* y, const int32_t* kept, const int32_t* accepted,
                                const int32_t* M_ptr, int max_M, double* ym, float* yf,
                                double* mscore, double tol2_s, int max_iter, int32_t* iters_out,
                                unsigned long long* evals, int kf, double sphere_r, int sms,
                                cudaStream_t st) {
  const int g = seed_grid(max_M, sms);
#define FMS_SEEDS(DP_)                                                                          \
  if (kf)                                                                                       \
    refine_seeds<DP_, 1><<<g, kSeedWarps * 32, 0, st>>>(Xs, cv, n, d, y, kept, accepted, M_ptr, \
                                                        ym, yf, mscore, tol2_s, max_iter,       \
                                                        iters_out, evals, sphere_r);            \
  else                                                                                          \
    refine_seeds<DP_, 0><<<g, kSeedWarps * 32, 0, st>>>(Xs, cv, n, d, y, kept, accepted, M_ptr, \
                                                        ym, yf, mscore, tol2_s, max_iter,       \
                                                        iters_out, evals, sphere_r);            \
  return cudaGetLastError();
  switch (DP) {
    case 4: FMS_SEEDS(4)
    case 8: FMS_SEEDS(8)
    case 16: FMS_SEEDS(16)
    case 32: FMS_SEEDS(32)
    case 64: FMS_SEEDS(64)
  }
#undef FMS_SEEDS
  return cudaErrorInvalidValue;
}

#define FMS_BY_WIDTH(RUN)             \
  switch (DP) {                       \
    case 4: RUN(4); break;            \
    case 8: RUN(8); break;            \
    case 16: RUN(16); break;          \
    case 32: RUN(32); break;          \
    case 64: RUN(64); break;          \
    default: return cudaErrorInvalidValue; \
  }                                   \
  return cudaGetLastError()

cudaError_t launch_travel_queue(const float* Xs, const View<float>& cv, int d, int DP,
                                const SeedQueue& q, float* y, int32_t* it, int32_t* conv,
                                int32_t* state, float* wlast, int max_iter, float tol2_s, int sms,
                                cudaStream_t st) {
#define FMS_RUN(DP_)                                                                            \
  travel_queue<DP_><<<sms * 8, kQueueWarps * 32, 0, st>>>(Xs, cv, d, q, y, it, conv, state, wlast, \
                                                          max_iter, tol2_s)
  FMS_BY_WIDTH(FMS_RUN);
#undef FMS_RUN
}

cudaError_t launch_density_queue(const float* Xs, const View<float>& cv, int DP, const SeedQueue& q,
                                 const float* y, float* score, double* mscore, int sms,
                                 cudaStream_t st) {
#define FMS_RUN(DP_) \
  density_queue<DP_><<<sms * 8, kQueueWarps * 32, 0, st>>>(Xs, cv, q, y, score, mscore)
  FMS_BY_WIDTH(FMS_RUN);
#undef FMS_RUN
}

cudaError_t launch_refine_queue(const float* Xs, const View<float>& cv, int d, int DP,
                                const SeedQueue& q, double* ym, float* yf, double* mscore,
                                double tol2_s, int max_iter, int32_t* iters_out, int sms,
                                cudaStream_t st) {
#define FMS_RUN(DP_)                                                                           \
  refine_queue<DP_><<<sms * 8, kQueueWarps * 32, 0, st>>>(Xs, cv, d, q, ym, yf, mscore, tol2_s, \
                                                          max_iter, iters_out)
  FMS_BY_WIDTH(FMS_RUN);
#undef FMS_RUN
}

}  // namespace fms

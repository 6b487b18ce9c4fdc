// Differentiable unrolled mean-shift steps: T Gaussian updates of every seed
// (for B independent sets at once) and their adjoint.
//
// Forward (Eq. 6 with the Gaussian weight), for each set and seed i:
//   W_i = sum_j w_ij,  y_i <- mu_i = sum_j w_ij x_j / W_i,
//   w_ij = exp(-||y_i - x_j||^2 / (2h^2)) = exp2(-c ||y_i - x_j||^2), c = log2(e)/(2h^2).
// Adjoint of one update, with p_ij = w_ij / W_i, g_i = dL/dmu_i and
// a_ij = g_i . (x_j - mu_i) (derived by differentiating log w_ij):
//   dL/dy_i  = (1/h^2) sum_j p_ij a_ij (x_j - mu_i)
//   dL/dx_j += p_ij [g_i - a_ij (x_j - y_i) / h^2]
//   dL/dh   += (1/h^3) sum_ij p_ij ||y_i - x_j||^2 a_ij
// The weights are recomputed tile by tile: nothing of size m x n is stored.
// Positions Y_t are checkpointed every k updates; the backward recomputes one
// segment of k updates from its checkpoint, then walks it in reverse.
//
// Points and seeds are kept sorted into cells (fms_cells.cuh), and a group of 32
// seeds of one cell walks only the point cells within its cutoff radius (where a
// sample says that cells leave too little out, 32 seeds in a row walk every point,
// in one pass an update).  Seeds
// do not depend on each other, so one launch takes a group through all T updates
// (or, in the adjoint, through a whole segment).  Kernels (FP32, or FP64 for
// checking gradients; exact differences, fixed-order sums; rows padded to DP =
// 4, 8, 16 or 32 values):
//   unroll_travel     lanes own the seeds of a group, a team of warps splits
//                     the tiles of visible points (staged in shared memory,
//                     read with broadcast loads); T updates in one launch.  A
//                     seed whose W underflows (every point farther than ~13 h)
//                     is recomputed with the weights taken relative to its
//                     nearest point, w = exp2(-c (D2 - D2min)) (the shift
//                     cancels in w / W), and the shift c D2min kept for the
//                     backward
//   unroll_bwd_seed   the same groups backwards through a segment: per update
//                     the sums of p a (x - y), p a and p a ||y - x||^2, the
//                     gradient w.r.t. the positions before it, and one row per
//                     seed [y | g | 1/W, shift, g . (y - mu)] and one ball per
//                     group for
//   unroll_bwd_point  lanes own 32 points of a cell, the seed groups of every
//                     update of the segment whose ball reaches them are
//                     streamed: sum_i p_ij [g_i - a_ij (x_j - y_i) / h^2]
// Both adjoint passes take a_ij = g_i . (x_j - y_i) + g_i . (y_i - mu_i): every
// term is a difference of nearby positions (no cancellation of coordinates).
// Sums go tile by tile (32 rows) into totals, then over the team's warps in order.
//
// Bound by FP32 issue (3 DP + 3, 5 DP + 6 and 6 DP + 6 operations per visible pair).
// 8 sets x 16,384 points and seeds x 16, 32 blobs, T = 20, k = 5: each group sees
// about 515 of the 16,384 points; forward and backward 390.4 -> 19 ms (forward
// 3.9, recomputed positions 3.8, seed-major 5.2, point-major 6.0) against kernels
// that took every pair.  3 sets x 1,500 points x 701 seeds x 3, T = 10 (nothing
// sorted): 0.99 -> 0.40 ms, of which 0.43 came from 94 launches going to 15 and 0.13
// from resident points and phases; the zero column of d <= 3 left out is the rest.
#include "fms_team.cuh"

namespace fms {


// Below this W the unshifted weights lose precision (FP32 terms under 2^-126
// flush to zero) and the seed is recomputed with a shift.
template <typename T>
__device__ __forceinline__ T unroll_min_w() {
  return sizeof(T) == 4 ? (T)1e-20f : (T)1e-280;
}

// One far seed, recomputed by a warp with the points over its lanes: pass 1 the
// nearest squared distance D2min, pass 2 the weights exp2(-c (D2 - D2min)) and
// their sums (fixed xor tree).  acc = (W, S, sum w D2); returns the shift c D2min.
template <typename T, int DP>
__device__ T rescue_seed(const T* __restrict__ Xb, int n, T c, const T (&y)[DP], T (&acc)[DP + 2],
                         int lane) {
  T dmin = T(INFINITY);
  for (int j = lane; j < n; j += 32) {
    T x[DP];
    load_row<DP>(Xb + (int64_t)j * DP, x);
    T D2 = T(0);
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      const T e = x[k] - y[k];
      D2 = ufma(e, e, D2);
    }
    dmin = umin(dmin, D2);
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) dmin = umin(dmin, __shfl_xor_sync(kFull, dmin, o));
  const T sh = c * dmin;
#pragma unroll
  for (int k = 0; k < DP + 2; ++k) acc[k] = T(0);
  for (int j = lane; j < n; j += 32) {
    T x[DP];
    load_row<DP>(Xb + (int64_t)j * DP, x);
    T dx[DP], D2 = T(0);
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      dx[k] = x[k] - y[k];
      D2 = ufma(dx[k], dx[k], D2);
    }
    const T w = uex2(ufma(-c, D2, sh));
    acc[0] += w;
    acc[DP + 1] = ufma(w, D2, acc[DP + 1]);
#pragma unroll
    for (int k = 0; k < DP; ++k) acc[1 + k] = ufma(w, dx[k], acc[1 + k]);
  }
#pragma unroll
  for (int k = 0; k < DP + 2; ++k)
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) acc[k] += __shfl_xor_sync(kFull, acc[k], o);
  return sh;
}

// ---- forward: `steps` updates of one group of seeds per block.  After update
// t the positions go to slot ceil(t / every) - slot0 of pos where t is a
// multiple of `every` or the last one; W and the shift of update t to row t - 1
// of Wout and Sh (nullable).
template <typename T, int DP, int NX, int PH>
__global__ void __launch_bounds__(32 * most_warps<T, DP>())
    unroll_travel(const T* __restrict__ X, View<T> cv, const T* __restrict__ Y0, Groups gr,
                  UGeom g, T c, int steps, int every, int slot0, T* __restrict__ pos,
                  T* __restrict__ Wout, T* __restrict__ Sh, T* __restrict__ M2, int resident) {
  extern __shared__ __align__(16) unsigned char unroll_smem[];
  constexpr int SUMS = DP + 3, GS = 32 / PH;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, W = blockDim.x >> 5;
  if (!cv.gate.open()) {
    cv.P = 0;
    gr.table = nullptr;
  }
  const int b = blockIdx.x / gr.per_set;
  int row0, cnt;
  if (!group_rows(gr, b, blockIdx.x % gr.per_set, g.m, &row0, &cnt, GS)) return;
  const T* Xb = X + (int64_t)b * g.n * DP;
  const TeamSmem<T, DP, SUMS> sm(unroll_smem, w, W, Xb, resident ? g.n : 0);
  const int64_t rowsY = (int64_t)g.B * g.m;
  const int64_t e = (int64_t)b * g.m + row0 + min(lane % GS, cnt - 1);
  T y[DP];
  load_row<DP>(Y0 + e * DP, y);
  const T log2n = T(log2f((float)g.n));
  T cut = T(cells::kFirstCut);
  for (int t = 1; t <= steps; ++t) {
    T acc[DP + 2];   // W, S, sum w ||x - y||^2
    T need = T(0);
    for (int pass = 0;; ++pass) {
      T reach;
      const int nl = visible_cells<T, DP>(cv, b, g.n, y, true, cells::csqrt(cut / c), &reach,
                                          nullptr, sm, w, W, lane);
#pragma unroll
      for (int k = 0; k < DP + 2; ++k) acc[k] = T(0);
      sm.walk(Xb, g.n, nl, w, W, lane, [&](const T* rows, int nr) {
        T ta[DP + 2];
#pragma unroll
        for (int k = 0; k < DP + 2; ++k) ta[k] = T(0);
        tile_rows<DP, PH, row_unroll<T, DP>()>(rows, nr, lane, [&](const T* row, bool in) {
          T x[DP];
          smem_row<DP>(row, x);
          T D2 = T(0);
#pragma unroll
          for (int k = 0; k < NX; ++k) {
            x[k] -= y[k];
            D2 = ufma(x[k], x[k], D2);
          }
          const T wt = in ? uex2(-c * D2) : T(0);
          ta[0] += wt;
          ta[DP + 1] = ufma(wt, D2, ta[DP + 1]);
#pragma unroll
          for (int k = 0; k < NX; ++k) ta[1 + k] = ufma(wt, x[k], ta[1 + k]);
        });
#pragma unroll
        for (int k = 0; k < DP + 2; ++k) acc[k] += ta[k];
      });
      phase_sum<PH>(acc);
      team_sum<GS>(acc, sm.sums, SUMS, w, W, lane);
      if (cv.P == 0) break;
      need = cells::cut_bits(cells::warp_min(acc[0]), log2n);
      if (!(need > cut)) break;
      cut = pass == 0 ? cells::widen(need) : T(cells::zero_bits<T>());
    }
    cut = cells::widen(need);   // (W does not decrease along a trajectory)
    T sh = T(0);
    unsigned bad = __ballot_sync(kFull, !(acc[0] >= unroll_min_w<T>()) || !isfinite(acc[0]));
    if (bad) {   // the same for every warp of the team
      for (int u = 0; u < GS; ++u) {
        if (!((bad >> u) & 1u) || u % W != w) continue;
        T ys[DP], a2[DP + 2];
#pragma unroll
        for (int k = 0; k < DP; ++k) ys[k] = __shfl_sync(kFull, y[k], u);
        const T s2 = rescue_seed<T, DP>(Xb, g.n, c, ys, a2, lane);
        if (lane == 0) {
#pragma unroll
          for (int k = 0; k < DP + 2; ++k) sm.sums[k * 32 + u] = a2[k];
          sm.sums[(DP + 2) * 32 + u] = s2;
        }
      }
      __syncthreads();
      if ((bad >> lane) & 1u) {
#pragma unroll
        for (int k = 0; k < DP + 2; ++k) acc[k] = sm.sums[k * 32 + lane % GS];
        sh = sm.sums[(DP + 2) * 32 + lane % GS];
      }
      __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < DP; ++k)
      if (k < g.d) y[k] += acc[1 + k] / acc[0];
    if (w == 0 && lane < cnt) {
      if (Wout) {
        Wout[(int64_t)(t - 1) * rowsY + e] = acc[0];
        Sh[(int64_t)(t - 1) * rowsY + e] = sh;
        M2[(int64_t)(t - 1) * rowsY + e] = acc[DP + 1] / acc[0];
      }
      if (t % every == 0 || t == steps)
        store_row<T, DP>(pos + ((int64_t)((t + every - 1) / every - slot0) * rowsY + e) * DP, y);
    }
  }
}

// ---- backward, seed-major, updates len-1 .. 0 of one segment: with
//   DY_i = sum_j p_ij a_ij (x_j - mu_i) = sum_j p a (x_j - y_i) + (y_i - mu_i) sum_j p a,
//   DH_i = sum_j p_ij a_ij ||y_i - x_j||^2 = sum_j p a (||y_i - x_j||^2 - s_i),
// g <- DY / h^2 and dh_part += DH / h^3.  The last form of DH holds for any s_i
// because sum_j p_ij a_ij = g_i . sum_j p_ij (x_j - mu_i) = 0; s_i = the mean of
// ||y_i - x_j||^2 under p (kept by the forward) makes the terms smallest, and a
// far seed's residual sum p a (FP32 rounding of a D2 of hundreds leaves ~1e-5
// instead of 0) is not multiplied by D2.  DH is summed over tiles in FP64.
template <typename T, int DP, int NX, int PH>
__global__ void __launch_bounds__(32 * most_warps<T, DP>())
    unroll_bwd_seed(const T* __restrict__ X, View<T> cv, USegment<T> sg, Groups gr, UGeom g, T c,
                    T inv_h2, double inv_h3, const T* __restrict__ Gin, T* __restrict__ Gout,
                    T* __restrict__ SD, T* __restrict__ bctr, T* __restrict__ breach,
                    double* __restrict__ dh_part, int first, int resident) {
  extern __shared__ __align__(16) unsigned char unroll_smem[];
  constexpr int SUMS = DP + 2, SDW = 2 * DP + 4, GS = 32 / PH;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, W = blockDim.x >> 5;
  if (!cv.gate.open()) {
    cv.P = 0;
    gr.table = nullptr;
  }
  __shared__ double dhs[16];
  const int b = blockIdx.x / gr.per_set, gi = blockIdx.x % gr.per_set;
  const int64_t NG = (int64_t)g.B * gr.per_set;
  int row0, cnt;
  if (!group_rows(gr, b, gi, g.m, &row0, &cnt, GS)) {
    if (threadIdx.x == 0 && first) dh_part[blockIdx.x] = 0.0;
    return;
  }
  const T* Xb = X + (int64_t)b * g.n * DP;
  const TeamSmem<T, DP, SUMS> sm(unroll_smem, w, W, Xb, resident ? g.n : 0);
  const int64_t rowsY = (int64_t)g.B * g.m;
  const int64_t e = (int64_t)b * g.m + row0 + min(lane % GS, cnt - 1);
  const T log2n = T(log2f((float)g.n));
  T gg[DP];
  load_row<DP>(Gin + e * DP, gg);
  double dh = 0.0;
  // the next update's row and values are loaded a pass ahead where registers allow
  constexpr bool kAhead = DP <= 8;
  T yn[DP], ya[DP], Wn, shn, m2n;
  auto fetch = [&](int u) {
    const int64_t ue = (int64_t)(sg.u0 + u) * rowsY + e;
    load_row<DP>(sg.pos(u) + e * DP, yn);
    Wn = sg.W[ue];
    shn = sg.Sh[ue];
    m2n = sg.M2[ue];
  };
  if (kAhead) {
    load_row<DP>(sg.pos(sg.len) + e * DP, ya);
    fetch(sg.len - 1);
  }
  for (int u = sg.len - 1; u >= 0; --u) {
    T y[DP], ym[DP], ctr[DP];
    if (!kAhead) {
      load_row<DP>(sg.pos(u + 1) + e * DP, ya);
      fetch(u);
    }
    const T Wt = Wn, sh = shn, s0 = m2n;
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      y[k] = yn[k];
      ym[k] = ya[k];
      if (kAhead) ya[k] = y[k];
    }
    if (kAhead && u > 0) fetch(u - 1);
    const T invW = T(1) / Wt;
    T gd = T(0);
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      ym[k] = y[k] - ym[k];
      gd = ufma(gg[k], ym[k], gd);
    }
    // every weight above the cutoff of its seed (exponent c D2 - sh)
    T reach;
    const int nl = visible_cells<T, DP>(cv, b, g.n, y, true,
                                        cells::csqrt((cells::cut_bits(Wt, log2n) + sh) / c),
                                        &reach, &ctr, sm, w, W, lane);
    if (w == 0) {
      if (lane < cnt) {
        T* o = SD + ((int64_t)u * rowsY + e) * SDW;
        store_row<T, DP>(o, y);
        store_row<T, DP>(o + DP, gg);
        const T tail[4] = {invW, sh, gd, T(0)};
        store_row<T, 4>(o + 2 * DP, tail);
      }
      if (lane == 0 && cv.P > 0) {
        store_row<T, DP>(bctr + ((int64_t)u * NG + blockIdx.x) * DP, ctr);
        breach[(int64_t)u * NG + blockIdx.x] = reach;
      }
    }
    T acc[DP + 1];   // sum p a, DY
    double DH = 0.0;
#pragma unroll
    for (int k = 0; k <= DP; ++k) acc[k] = T(0);
    sm.walk(Xb, g.n, nl, w, W, lane, [&](const T* rows, int nr) {
      T ta[DP + 2];
#pragma unroll
      for (int k = 0; k < DP + 2; ++k) ta[k] = T(0);
      tile_rows<DP, PH, row_unroll<T, DP>()>(rows, nr, lane, [&](const T* row, bool in) {
        T x[DP];
        smem_row<DP>(row, x);
        T D2 = T(0), a = gd;
#pragma unroll
        for (int k = 0; k < NX; ++k) {
          x[k] -= y[k];
          D2 = ufma(x[k], x[k], D2);
          a = ufma(gg[k], x[k], a);
        }
        const T pa = in ? uex2(ufma(-c, D2, sh)) * invW * a : T(0);
        ta[0] = ufma(pa, D2 - s0, ta[0]);
        ta[1] += pa;
#pragma unroll
        for (int k = 0; k < NX; ++k) ta[2 + k] = ufma(pa, x[k], ta[2 + k]);
      });
#pragma unroll
      for (int k = 0; k <= DP; ++k) acc[k] += ta[1 + k];
      DH += (double)ta[0];
    });
    phase_sum<PH>(acc);
    team_sum<GS>(acc, sm.sums, SUMS, w, W, lane);
    dh += DH;   // (this warp's tiles)
#pragma unroll
    for (int k = 0; k < DP; ++k) gg[k] = ufma(ym[k], acc[0], acc[1 + k]) * inv_h2;
  }
  if (lane % GS >= cnt) dh = 0.0;
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) dh += __shfl_xor_sync(kFull, dh, o);
  if (lane == 0) dhs[w] = dh;
  __syncthreads();
  if (w == 0) {
    if (lane < cnt) store_row<T, DP>(Gout + e * DP, gg);
    if (lane == 0) {
      double t = 0.0;
      for (int u = 0; u < W; ++u) t += dhs[u];
      t *= inv_h3;
      dh_part[blockIdx.x] = first ? t : dh_part[blockIdx.x] + t;
    }
  }
}

// ---- backward, point-major, all updates of one segment: one block per group
// of 32 points adds
//   DX_j = sum_i p_ij g_i - (1/h^2) sum_i p_ij a_ij (x_j - y_i)
// to its rows of dX.
template <typename T, int DP, int NX>
__global__ void __launch_bounds__(32 * most_warps<T, DP>())
    unroll_bwd_point(const T* __restrict__ X, Gate gate, Groups gx, Groups gr, UGeom g, int len,
                     T c, T inv_h2, const T* __restrict__ SD, const T* __restrict__ bctr,
                     const T* __restrict__ breach, T* __restrict__ dX, int first) {
  extern __shared__ __align__(16) unsigned char unroll_smem[];
  constexpr int SUMS = DP, SDW = 2 * DP + 4;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, W = blockDim.x >> 5;
  if (!gate.open()) gx.table = gr.table = nullptr;
  const TeamSmem<T, SDW, SUMS, false> sm(unroll_smem, w, W);
  const int b = blockIdx.x / gx.per_set;
  int row0, cnt;
  if (!group_rows(gx, b, blockIdx.x % gx.per_set, g.n, &row0, &cnt)) return;
  const int64_t e = (int64_t)b * g.n + row0 + min(lane, cnt - 1);
  const int64_t rowsY = (int64_t)g.B * g.m, NG = (int64_t)g.B * gr.per_set;
  T x[DP], ctr[DP], acc[DP];
  load_row<DP>(X + e * DP, x);
  const T rho = cells::group_ball<T, DP>(x, ctr);
#pragma unroll
  for (int k = 0; k < DP; ++k) acc[k] = T(0);
  for (int u = 0; u < len; ++u) {
    const T* sdb = SD + ((int64_t)u * rowsY + (int64_t)b * g.m) * SDW;
    if (!gr.table) {   // nothing sorted: every seed
      if (lane == 0) sm.list[0] = make_int2(0, g.m);
      __syncwarp();
    }
    for (int g0 = 0; gr.table ? g0 < gr.per_set : g0 == 0;) {
      // the next seed groups that reach these points, as many as the list holds
      int nl = gr.table ? 0 : 1;
      if (!gr.table) g0 = 1;
      for (; gr.table && g0 < gr.per_set && nl <= kListCap - 32; g0 += 32) {
        const int gi = g0 + lane;
        bool see = false;
        int r0 = 0, rc = 0;
        if (gi < gr.per_set && group_rows(gr, b, gi, g.m, &r0, &rc)) {
          const int64_t at = (int64_t)u * NG + (int64_t)b * gr.per_set + gi;
          T q[DP];
          load_row<DP>(bctr + at * DP, q);
          T d2 = T(0);
#pragma unroll
          for (int k = 0; k < DP; ++k) {
            const T f = q[k] - ctr[k];
            d2 += f * f;
          }
          const T lim = (rho + breach[at]) * T(1.0001);
          see = !(d2 > lim * lim);
        }
        const unsigned m = __ballot_sync(kFull, see);
        if (see) sm.list[nl + __popc(m & ((1u << lane) - 1u))] = make_int2(r0, rc);
        nl += __popc(m);
      }
      __syncwarp();
      cells::walk_tiles<SDW>(sdb, sm.list, nl, w, W, sm.ring, lane, [&](const T* rows, int nr) {
        T ta[DP];
#pragma unroll
        for (int k = 0; k < DP; ++k) ta[k] = T(0);
#pragma unroll (DP <= 4 ? 4 : 1)
        for (int q = 0; q < nr; ++q) {
          const T* sd = rows + q * SDW;
          T dx[DP], gv[DP], tail[4];
          smem_row<DP>(sd, dx);
          smem_row<DP>(sd + DP, gv);
          smem_row<4>(sd + 2 * DP, tail);
          T D2 = T(0), a = tail[2];
#pragma unroll
          for (int k = 0; k < NX; ++k) {
            dx[k] = x[k] - dx[k];
            D2 = ufma(dx[k], dx[k], D2);
            a = ufma(gv[k], dx[k], a);
          }
          const T p = uex2(ufma(-c, D2, tail[1])) * tail[0];
          const T q2 = p * a * inv_h2;
#pragma unroll
          for (int k = 0; k < NX; ++k) ta[k] = ufma(p, gv[k], ufma(-q2, dx[k], ta[k]));
        }
#pragma unroll
        for (int k = 0; k < DP; ++k) acc[k] += ta[k];
      });
    }
  }
  team_sum<32>(acc, sm.sums, SUMS, w, W, lane);
  if (w == 0 && lane < cnt) {
    T* o = dX + e * DP;
    if (!first) {
#pragma unroll
      for (int k = 0; k < DP; ++k) acc[k] += o[k];
    }
    store_row<T, DP>(o, acc);
  }
}

// dh[b] = the sum of set b's group sums in FP64, in a fixed order (one block per set).
__global__ void unroll_dh_reduce(const double* __restrict__ dh_part, int per_set,
                                 double* __restrict__ dh) {
  __shared__ double red[8];
  const double* p = dh_part + (int64_t)blockIdx.x * per_set;
  double s = 0.0;
  for (int i = threadIdx.x; i < per_set; i += blockDim.x) s += p[i];
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    dh[blockIdx.x] = t;
  }
}

// Row repacking between the caller's [rows x d] and the padded [rows x DP]; with
// perm, padded row i of a set is the caller's row perm[i] of that set.
template <typename T>
__global__ void unroll_pack(const T* __restrict__ src, int64_t rows, int per_set, int d, int DP,
                            const int32_t* __restrict__ perm, T* __restrict__ dst) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < rows * DP;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / DP;
    const int k = (int)(e % DP);
    const int64_t s = perm ? r / per_set * per_set + perm[r] : r;
    dst[e] = k < d ? src[s * d + k] : T(0);
  }
}

template <typename T>
__global__ void unroll_unpack(const T* __restrict__ src, int64_t rows, int per_set, int d, int DP,
                              const int32_t* __restrict__ perm, T* __restrict__ dst) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < rows * DP;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / DP;
    const int k = (int)(e % DP);
    if (k >= d) continue;
    const int64_t s = perm ? r / per_set * per_set + perm[r] : r;
    dst[s * d + k] = src[e];
  }
}

static int blocks_for(int64_t work, int per = 256) {
  int64_t b = (work + per - 1) / per;
  if (b < 1) b = 1;
  if (b > 8192) b = 8192;
  return (int)b;
}

template <typename T, int DP, int NX, int PH>
static cudaError_t travel_p(const T* X, const View<T>& cv, const T* Y0, Groups gr, const UGeom& g,
                            T c, int steps, int every, int slot0, T* pos, T* Wout, T* Sh, T* M2,
                            cudaStream_t st) {
  if (PH > 1) gr.per_set = (g.m + 32 / PH - 1) / (32 / PH);
  const int64_t NG = (int64_t)g.B * gr.per_set;
  constexpr int ws = team_warp_smem<T, DP, DP + 3>();
  const int W = team_warps(NG, g.sms, ws, most_warps<T, DP>());
  const bool res = team_resident<T, DP>(cv.P, g.n);
  const int smem = res ? resident_team_smem<T, DP, DP + 3>(W, g.n) : group_team_smem<T, DP, DP + 3>(W);
  const cudaError_t e = team_attr(unroll_travel<T, DP, NX, PH>, smem);
  if (e != cudaSuccess) return e;
  unroll_travel<T, DP, NX, PH><<<(unsigned)NG, 32 * W, smem, st>>>(
      X, cv, Y0, gr, g, c, steps, every, slot0, pos, Wout, Sh, M2, res ? 1 : 0);
  return cudaGetLastError();
}

template <typename T, int DP, int NX = DP>
static cudaError_t travel_t(const T* X, const View<T>& cv, const T* Y0, const Groups& gr,
                            const UGeom& g, T c, int steps, int every, int slot0, T* pos, T* Wout,
                            T* Sh, T* M2, cudaStream_t st) {
  if constexpr (sizeof(T) == 4 && DP <= 16)
    if (team_phases<T, DP>(cv.P, (int64_t)g.B * g.m, g.sms) == 4)
      return travel_p<T, DP, NX, 4>(X, cv, Y0, gr, g, c, steps, every, slot0, pos, Wout, Sh, M2, st);
  return travel_p<T, DP, NX, 1>(X, cv, Y0, gr, g, c, steps, every, slot0, pos, Wout, Sh, M2, st);
}

template <typename T>
cudaError_t unroll_forward_steps(const T* X, const View<T>& cv, const T* Y0, const Groups& gr,
                                 const UGeom& g, T c, int steps, int every, int slot0, T* pos,
                                 T* Wout, T* Sh, T* M2, cudaStream_t st) {
  if (g.d <= 3) return travel_t<T, 4, 3>(X, cv, Y0, gr, g, c, steps, every, slot0, pos, Wout, Sh, M2, st);
  switch (g.DP) {
    case 4: return travel_t<T, 4>(X, cv, Y0, gr, g, c, steps, every, slot0, pos, Wout, Sh, M2, st);
    case 8: return travel_t<T, 8>(X, cv, Y0, gr, g, c, steps, every, slot0, pos, Wout, Sh, M2, st);
    case 16: return travel_t<T, 16>(X, cv, Y0, gr, g, c, steps, every, slot0, pos, Wout, Sh, M2, st);
    case 32: return travel_t<T, 32>(X, cv, Y0, gr, g, c, steps, every, slot0, pos, Wout, Sh, M2, st);
  }
  return cudaErrorInvalidValue;
}

// the seed-major pass; *groups: its groups in all (the entries of dh_part)
template <typename T, int DP, int NX, int PH>
static cudaError_t bwd_seed_p(const T* X, const View<T>& cv, const USegment<T>& sg, Groups gr,
                              const UGeom& g, T c, T inv_h2, double inv_h3, const T* Gin, T* Gout,
                              T* SD, T* bctr, T* breach, double* dh_part, int first,
                              cudaStream_t st) {
  if (PH > 1) gr.per_set = (g.m + 32 / PH - 1) / (32 / PH);
  const int64_t NG = (int64_t)g.B * gr.per_set;
  constexpr int ws = team_warp_smem<T, DP, DP + 2>();
  const int W = team_warps(NG, g.sms, ws, most_warps<T, DP>());
  const bool res = team_resident<T, DP>(cv.P, g.n);
  const int smem = res ? resident_team_smem<T, DP, DP + 2>(W, g.n) : group_team_smem<T, DP, DP + 2>(W);
  const cudaError_t e = team_attr(unroll_bwd_seed<T, DP, NX, PH>, smem);
  if (e != cudaSuccess) return e;
  unroll_bwd_seed<T, DP, NX, PH><<<(unsigned)NG, 32 * W, smem, st>>>(
      X, cv, sg, gr, g, c, inv_h2, inv_h3, Gin, Gout, SD, bctr, breach, dh_part, first, res ? 1 : 0);
  return cudaGetLastError();
}

template <typename T, int DP, int NX = DP>
static cudaError_t bwd_t(const T* X, const View<T>& cv, const USegment<T>& sg, const Groups& gx,
                         const Groups& gr, const UGeom& g, T c, T inv_h2, double inv_h3,
                         const T* Gin, T* Gout, T* SD, T* bctr, T* breach, double* dh_part, T* dX,
                         int first, cudaStream_t st) {
  cudaError_t e = cudaErrorInvalidValue;
  bool done = false;
  if constexpr (sizeof(T) == 4 && DP <= 16)
    if (team_phases<T, DP>(cv.P, (int64_t)g.B * g.m, g.sms) == 4) {
      e = bwd_seed_p<T, DP, NX, 4>(X, cv, sg, gr, g, c, inv_h2, inv_h3, Gin, Gout, SD, bctr, breach,
                               dh_part, first, st);
      done = true;
    }
  if (!done)
    e = bwd_seed_p<T, DP, NX, 1>(X, cv, sg, gr, g, c, inv_h2, inv_h3, Gin, Gout, SD, bctr, breach,
                             dh_part, first, st);
  if (e != cudaSuccess) return e;
  const int64_t PG = (int64_t)g.B * gx.per_set;
  constexpr int wp = team_warp_smem<T, 2 * DP + 4, DP>();
  const int Wp = team_warps(PG, g.sms, wp, most_warps<T, DP>());
  const int smem_p = list_team_smem<T, 2 * DP + 4, DP>(Wp);
  e = team_attr(unroll_bwd_point<T, DP, NX>, smem_p);
  if (e != cudaSuccess) return e;
  unroll_bwd_point<T, DP, NX><<<(unsigned)PG, 32 * Wp, smem_p, st>>>(X, cv.gate, gx, gr, g, sg.len, c, inv_h2,
                                                                 SD, bctr, breach, dX, first);
  return cudaGetLastError();
}

// Groups of a set in the seed-major passes (and entries of dh_part per set).
template <typename T>
int unroll_seed_groups(int P, const UGeom& g, int per_set) {
  const int64_t seeds = (int64_t)g.B * g.m;
  int ph = 1;
  if (g.DP <= 4) ph = team_phases<T, 4>(P, seeds, g.sms);
  else if (g.DP <= 8) ph = team_phases<T, 8>(P, seeds, g.sms);
  else if (g.DP <= 16) ph = team_phases<T, 16>(P, seeds, g.sms);
  return ph == 1 ? per_set : (g.m + 32 / ph - 1) / (32 / ph);
}
template int unroll_seed_groups<float>(int, const UGeom&, int);
template int unroll_seed_groups<double>(int, const UGeom&, int);

template <typename T>
cudaError_t unroll_backward_segment(const T* X, const View<T>& cv, const USegment<T>& sg,
                                    const Groups& gx, const Groups& gr, const UGeom& g, T c,
                                    T inv_h2, double inv_h3, const T* Gin, T* Gout, T* SD, T* bctr,
                                    T* breach, double* dh_part, T* dX, int first,
                                    cudaStream_t st) {
#define FMS_BWD(...)                                                                         \
  return bwd_t<T, __VA_ARGS__>(X, cv, sg, gx, gr, g, c, inv_h2, inv_h3, Gin, Gout, SD, bctr, \
                               breach, dh_part, dX, first, st)
  if (g.d <= 3) FMS_BWD(4, 3);
  switch (g.DP) {
    case 4: FMS_BWD(4);
    case 8: FMS_BWD(8);
    case 16: FMS_BWD(16);
    case 32: FMS_BWD(32);
  }
#undef FMS_BWD
  return cudaErrorInvalidValue;
}

cudaError_t unroll_dh_sum(const double* dh_part, int B, int per_set, double* dh, cudaStream_t st) {
  unroll_dh_reduce<<<B, 256, 0, st>>>(dh_part, per_set, dh);
  return cudaGetLastError();
}

template <typename T>
cudaError_t unroll_pack_rows(const T* src, int64_t rows, int per_set, int d, int DP,
                             const int32_t* perm, T* dst, cudaStream_t st) {
  unroll_pack<T><<<blocks_for(rows * DP), 256, 0, st>>>(src, rows, per_set, d, DP, perm, dst);
  return cudaGetLastError();
}

template <typename T>
cudaError_t unroll_unpack_rows(const T* src, int64_t rows, int per_set, int d, int DP,
                               const int32_t* perm, T* dst, cudaStream_t st) {
  unroll_unpack<T><<<blocks_for(rows * DP), 256, 0, st>>>(src, rows, per_set, d, DP, perm, dst);
  return cudaGetLastError();
}

#define FMS_UNROLL_INST(T)                                                                        \
  template cudaError_t unroll_forward_steps<T>(const T*, const View<T>&, const T*, const Groups&, \
                                               const UGeom&, T, int, int, int, T*, T*, T*, T*,    \
                                               cudaStream_t);                                     \
  template cudaError_t unroll_backward_segment<T>(                                                \
      const T*, const View<T>&, const USegment<T>&, const Groups&, const Groups&, const UGeom&,   \
      T, T, double, const T*, T*, T*, T*, T*, double*, T*, int, cudaStream_t);                        \
  template cudaError_t unroll_pack_rows<T>(const T*, int64_t, int, int, int, const int32_t*, T*,  \
                                           cudaStream_t);                                         \
  template cudaError_t unroll_unpack_rows<T>(const T*, int64_t, int, int, int, const int32_t*,    \
                                             T*, cudaStream_t);
FMS_UNROLL_INST(float)
FMS_UNROLL_INST(double)
#undef FMS_UNROLL_INST

}  // namespace fms

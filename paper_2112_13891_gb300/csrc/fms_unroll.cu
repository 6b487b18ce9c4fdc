// C ABI of the differentiable unrolled mean-shift steps (see k_unroll.cu for
// the kernels and the adjoint formulas), in FP32 and, for checking gradients,
// FP64 (the *_f64 entry points).
#include <math.h>
#include <string.h>

#include "../../include/fms.h"
#include "fms_cells.cuh"

using namespace fms;

namespace {

size_t a256(size_t x) { return (x + 255) / 256 * 256; }

bool valid(int32_t B, int64_t n, int64_t m, int32_t d, int32_t T, int32_t k) {
  return B >= 1 && n >= 1 && m >= 1 && n <= INT32_MAX && m <= INT32_MAX && d >= 1 && d <= 32 &&
         T >= 1 && k >= 1 && (int64_t)B * n <= INT32_MAX && (int64_t)B * m <= INT32_MAX;
}

int sm_count() {
  int dev = 0, s = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&s, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  return s;
}

// rows padded to 4, 8, 16 or 32 floats (the kernels know the width at compile time)
int padded_width(int d) { return d <= 4 ? 4 : (d <= 8 ? 8 : (d <= 16 ? 16 : 32)); }

UGeom geom(int32_t B, int64_t n, int64_t m, int32_t d) {
  UGeom g{};
  g.B = B;
  g.n = (int)n;
  g.m = (int)m;
  g.d = d;
  g.DP = padded_width(d);
  const int sms = sm_count();
  g.sms = sms > 0 ? sms : 1;
  return g;
}

// Cells per set, 0 for none.  Sorting points and seeds takes ~40 us in each
// direction; below ~4 M pairs an update the whole pass over every pair is cheaper.
int cells_for(int32_t B, int64_t n, int64_t m) {
  if (B > 65535 || (double)B * (double)n * (double)m < 4194304.0) return 0;
  return cells::choose_cells(n, m);
}

int n_ckpt(int32_t T, int32_t k) { return (T + k - 1) / k; }

int groups_for(int64_t rows, int P) {
  return P > 0 ? cells::group_cap(rows, P) : (int)((rows + 31) / 32);
}

// updates of a segment whose seed rows are kept for one point-major pass
constexpr int kPointBatch = 8;

// Sorted copies of the points (and the scratch of sorting them and the seeds).
struct SortLayout {
  size_t Xp, Xs, perm, start, ctr, npiv, rad, table, ystart, scratch;
};

template <typename Take>
SortLayout sort_layout(const UGeom& g, int P, size_t es, Take&& take) {
  SortLayout L{};
  const size_t rows = (size_t)g.B * g.n, pad = (size_t)g.DP * es;
  L.Xs = take(rows * pad);
  if (P == 0) return L;
  L.Xp = take(rows * pad);
  L.perm = take(rows * 4);
  L.start = take((size_t)g.B * (P + 1) * 4);
  L.ctr = take((size_t)g.B * P * pad);
  L.npiv = take((size_t)g.B * 4);
  L.rad = take((size_t)g.B * P * es);
  L.table = take((size_t)g.B * cells::group_cap(g.n, P) * 8);
  L.ystart = take((size_t)g.B * (P + 1) * 4);
  const size_t a = cells::sort_scratch(g.B, g.n, P).total, b = cells::sort_scratch(g.B, g.m, P).total;
  L.scratch = take(a > b ? a : b);
  return L;
}

struct FwdLayout {
  SortLayout s;
  size_t Yp, total;
};
FwdLayout fwd_layout(const UGeom& g, int P, size_t es) {
  FwdLayout L{};
  size_t o = 0;
  auto take = [&](size_t b) {
    size_t at = o;
    o += a256(b > 0 ? b : 1);
    return at;
  };
  L.s = sort_layout(g, P, es, take);
  L.Yp = P > 0 ? take((size_t)g.B * g.m * g.DP * es) : 0;
  L.total = o;
  return L;
}

struct BwdLayout {
  SortLayout s;
  size_t seg, Ga, Gb, SD, bctr, breach, dh_part, dXp, total;
};
BwdLayout bwd_layout(const UGeom& g, int P, int32_t k, size_t es) {
  BwdLayout L{};
  size_t o = 0;
  auto take = [&](size_t b) {
    size_t at = o;
    o += a256(b > 0 ? b : 1);
    return at;
  };
  const size_t rowsY = (size_t)g.B * g.m, NG = (size_t)g.B * groups_for(g.m, P);
  const size_t pb = (size_t)(k < kPointBatch ? k : kPointBatch);
  const size_t seed_groups =
      es == 4 ? unroll_seed_groups<float>(P, g, groups_for(g.m, P))
              : unroll_seed_groups<double>(P, g, groups_for(g.m, P));
  L.s = sort_layout(g, P, es, take);
  L.seg = take((size_t)k * rowsY * g.DP * es);   // recomputed positions inside a segment
  L.Ga = take(rowsY * g.DP * es);
  L.Gb = take(rowsY * g.DP * es);
  L.SD = take(pb * rowsY * (2 * g.DP + 4) * es);
  L.bctr = take(pb * NG * g.DP * es);
  L.breach = take(pb * NG * es);
  L.dh_part = take((size_t)g.B * seed_groups * 8);
  L.dXp = take((size_t)g.B * g.n * g.DP * es);
  L.total = o;
  return L;
}

// The checkpoint buffer: positions Y_t for t = 0, k, 2k, .. and Y_T (rows of
// DP values, seeds in sorted order), then W_t, the weight shift and the mean
// squared distance of every update t < T (one value per seed each), so the
// backward recomputes only the positions between checkpoints; with cells, the
// seeds' order and groups and the probe's answer.
struct CkptLayout {
  size_t pos, W, Sh, M2, perm, table, walk, share, total;
};
CkptLayout ckpt_layout(const UGeom& g, int P, int32_t T, int32_t k, size_t es) {
  CkptLayout C{};
  const size_t rowsY = (size_t)g.B * g.m;
  C.pos = 0;
  C.W = (size_t)(n_ckpt(T, k) + 1) * rowsY * g.DP * es;
  C.Sh = C.W + (size_t)T * rowsY * es;
  C.M2 = C.Sh + (size_t)T * rowsY * es;
  C.perm = a256(C.M2 + (size_t)T * rowsY * es);
  C.table = C.perm + (P > 0 ? a256(rowsY * 4) : 0);
  C.walk = C.table + (P > 0 ? a256((size_t)g.B * cells::group_cap(g.m, P) * 8) : 0);
  C.share = C.walk + (P > 0 ? kProbeSets * 4 : 0);
  C.total = C.share + (P > 0 ? kProbeSets * 4 : 0);
  return C;
}

template <typename T>
T* at(void* base, size_t off) {
  return reinterpret_cast<T*>(static_cast<char*>(base) + off);
}

// Whether the cells leave enough out, asked of up to kProbeSets of the sets.
int probed_sets(int B) { return B < kProbeSets ? B : kProbeSets; }

template <typename E>
cudaError_t probe_sets(const E* points, const E* seeds0, const UGeom& g, double c, void* ckpt,
                       const CkptLayout& CL, cudaStream_t st) {
  ProbeArgs a{};
  a.sets = probed_sets(g.B);
  for (int i = 0; i < a.sets; ++i) {
    const int64_t b = ((2 * i + 1) * (int64_t)g.B) / (2 * a.sets);
    a.set[i] = {points + b * g.n * g.d, seeds0 + b * g.m * g.d, g.n, g.m};
  }
  a.d = a.ld = g.d;
  a.scale = sqrt(c);
  a.kind = kProbeBall;
  a.limit = kWalkShare;
  a.share = at<float>(ckpt, CL.share);
  a.walk = at<int32_t>(ckpt, CL.walk);
  return launch_probe<E>(a, st);
}

// Padded (and, with cells, sorted) copy of the points.
template <typename E>
cudaError_t sort_points(const E* points, const UGeom& g, int P, const SortLayout& L, void* ws,
                        cells::View<E>* cv, cudaStream_t st) {
  E* Xs = at<E>(ws, L.Xs);
  const int64_t rows = (int64_t)g.B * g.n;
  *cv = cells::View<E>{};
  if (P == 0) return unroll_pack_rows<E>(points, rows, g.n, g.d, g.DP, nullptr, Xs, st);
  const E* src = points;
  if (g.d != g.DP || (reinterpret_cast<uintptr_t>(points) & 15u)) {
    E* Xp = at<E>(ws, L.Xp);
    const cudaError_t e = unroll_pack_rows<E>(points, rows, g.n, g.d, g.DP, nullptr, Xp, st);
    if (e != cudaSuccess) return e;
    src = Xp;
  }
  cv->P = P;
  cv->start = at<int32_t>(ws, L.start);
  cv->ctr = at<E>(ws, L.ctr);
  cv->rad = at<E>(ws, L.rad);
  return cells::launch_sort<E>(src, g.B, g.n, g.DP, true, P, at<void>(ws, L.scratch), Xs,
                               at<int32_t>(ws, L.perm), at<int32_t>(ws, L.start),
                               at<E>(ws, L.ctr), at<int32_t>(ws, L.npiv), at<E>(ws, L.rad),
                               at<int2>(ws, L.table), st);
}

template <typename E>
fms_status forward_impl(const E* points, const E* seeds0, int32_t B, int64_t n, int64_t m,
                        int32_t d, E h, int32_t T, int32_t k, E* out_seeds, void* ckpt,
                        size_t ckpt_bytes, void* ws, size_t ws_bytes, void* stream) {
  if (!points || !seeds0 || !out_seeds || !valid(B, n, m, d, T, k) || !(h > 0) || !isfinite(h))
    return FMS_ERR_INVALID_ARG;
  if (!ws || !ckpt) return FMS_ERR_WORKSPACE;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const UGeom g = geom(B, n, m, d);
  const int P = cells_for(B, n, m);
  const FwdLayout L = fwd_layout(g, P, sizeof(E));
  const CkptLayout CL = ckpt_layout(g, P, T, k, sizeof(E));
  if (ws_bytes < L.total || ckpt_bytes < CL.total || (reinterpret_cast<uintptr_t>(ws) & 255u) ||
      (reinterpret_cast<uintptr_t>(ckpt) & 15u))
    return FMS_ERR_WORKSPACE;
  E* pos = at<E>(ckpt, CL.pos);
  int32_t* yperm = P > 0 ? at<int32_t>(ckpt, CL.perm) : nullptr;
  const int64_t rowsY = (int64_t)B * m;
  const E c = (E)(1.4426950408889634 / (2.0 * (double)h * (double)h));
  cells::View<E> cv;
  if (sort_points<E>(points, g, P, L.s, ws, &cv, st) != cudaSuccess) return FMS_ERR_CUDA;
  cells::Groups gr{nullptr, groups_for(m, P)};
  if (P > 0) {
    if (probe_sets<E>(points, seeds0, g, (double)c, ckpt, CL, st) != cudaSuccess)
      return FMS_ERR_CUDA;
    cv.gate = Gate{at<int32_t>(ckpt, CL.walk), probed_sets(B), 0, 0};
    const E* src = seeds0;
    if (d != g.DP || (reinterpret_cast<uintptr_t>(seeds0) & 15u)) {
      E* Yp = at<E>(ws, L.Yp);
      if (unroll_pack_rows<E>(seeds0, rowsY, (int)m, d, g.DP, nullptr, Yp, st) != cudaSuccess)
        return FMS_ERR_CUDA;
      src = Yp;
    }
    int2* table = at<int2>(ckpt, CL.table);
    gr.table = table;
    if (cells::launch_sort<E>(src, B, m, g.DP, false, P, at<void>(ws, L.s.scratch), pos, yperm,
                              at<int32_t>(ws, L.s.ystart), at<E>(ws, L.s.ctr),
                              at<int32_t>(ws, L.s.npiv), nullptr, table, st) != cudaSuccess)
      return FMS_ERR_CUDA;
  } else if (unroll_pack_rows<E>(seeds0, rowsY, (int)m, d, g.DP, nullptr, pos, st) !=
             cudaSuccess) {
    return FMS_ERR_CUDA;
  }
  if (unroll_forward_steps<E>(at<E>(ws, L.s.Xs), cv, pos, gr, g, c, T, k, 0, pos,
                              at<E>(ckpt, CL.W), at<E>(ckpt, CL.Sh), at<E>(ckpt, CL.M2), st) != cudaSuccess ||
      unroll_unpack_rows<E>(pos + (size_t)n_ckpt(T, k) * rowsY * g.DP, rowsY, (int)m, d, g.DP,
                            yperm, out_seeds, st) != cudaSuccess)
    return FMS_ERR_CUDA;
  return FMS_OK;
}

template <typename E>
fms_status backward_impl(const E* points, int32_t B, int64_t n, int64_t m, int32_t d, E h,
                         int32_t T, int32_t k, const void* ckpt, size_t ckpt_bytes,
                         const E* grad_out, E* grad_points, E* grad_seeds0, double* grad_h,
                         void* ws, size_t ws_bytes, void* stream) {
  if (!points || !grad_out || !grad_points || !grad_seeds0 || !grad_h ||
      !valid(B, n, m, d, T, k) || !(h > 0) || !isfinite(h))
    return FMS_ERR_INVALID_ARG;
  if (!ws || !ckpt) return FMS_ERR_WORKSPACE;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const UGeom g = geom(B, n, m, d);
  const int P = cells_for(B, n, m);
  const BwdLayout L = bwd_layout(g, P, k, sizeof(E));
  const CkptLayout CL = ckpt_layout(g, P, T, k, sizeof(E));
  if (ws_bytes < L.total || ckpt_bytes < CL.total || (reinterpret_cast<uintptr_t>(ws) & 255u) ||
      (reinterpret_cast<uintptr_t>(ckpt) & 15u))
    return FMS_ERR_WORKSPACE;
  void* ck = const_cast<void*>(ckpt);   // read only
  const E* Ck = at<E>(ck, CL.pos);
  const int32_t* yperm = P > 0 ? at<int32_t>(ck, CL.perm) : nullptr;
  const cells::Groups gr{P > 0 ? at<int2>(ck, CL.table) : nullptr, groups_for(m, P)};
  const cells::Groups gx{P > 0 ? at<int2>(ws, L.s.table) : nullptr, groups_for(n, P)};
  E* Xs = at<E>(ws, L.s.Xs);
  E* seg = at<E>(ws, L.seg);
  E* G = at<E>(ws, L.Ga);
  E* Gp = at<E>(ws, L.Gb);
  E* dXp = at<E>(ws, L.dXp);
  double* dh_part = at<double>(ws, L.dh_part);
  const int64_t rowsY = (int64_t)B * m, rowY = rowsY * g.DP;
  const double hd = (double)h;
  const E c = (E)(1.4426950408889634 / (2.0 * hd * hd));
  const E inv_h2 = (E)(1.0 / (hd * hd));
  const double inv_h3 = 1.0 / (hd * hd * hd);
  cells::View<E> cv;
  if (sort_points<E>(points, g, P, L.s, ws, &cv, st) != cudaSuccess ||
      unroll_pack_rows<E>(grad_out, rowsY, (int)m, d, g.DP, yperm, G, st) != cudaSuccess)
    return FMS_ERR_CUDA;
  if (P > 0) cv.gate = Gate{at<int32_t>(ck, CL.walk), probed_sets(B), 0, 0};
  int first = 1;
  for (int s = n_ckpt(T, k) - 1; s >= 0; --s) {
    const int t0 = s * k;
    const int len = (t0 + k <= T) ? k : T - t0;
    // positions of the segment: Y_t0 and Y_{t0+len} are checkpoints (the last
    // is Y_T for the final segment); Y_{t0+1} .. Y_{t0+len-1} are recomputed
    // into seg (W and the shifts of every update were stored by the forward)
    if (len > 1 && unroll_forward_steps<E>(Xs, cv, Ck + (size_t)s * rowY, gr, g, c, len - 1, 1, 1,
                                           seg, nullptr, nullptr, nullptr, st) != cudaSuccess)
      return FMS_ERR_CUDA;
    for (int hi = len; hi > 0;) {
      const int lo = hi > kPointBatch ? hi - kPointBatch : 0;
      USegment<E> sg{};
      sg.ck0 = Ck + (size_t)s * rowY;
      sg.ck1 = Ck + (size_t)(s + 1) * rowY;
      sg.seg = seg;
      sg.row_values = rowY;
      sg.seg_len = len;
      sg.u0 = lo;
      sg.len = hi - lo;
      sg.W = at<E>(ck, CL.W) + (size_t)t0 * rowsY;
      sg.Sh = at<E>(ck, CL.Sh) + (size_t)t0 * rowsY;
      sg.M2 = at<E>(ck, CL.M2) + (size_t)t0 * rowsY;
      if (unroll_backward_segment<E>(Xs, cv, sg, gx, gr, g, c, inv_h2, inv_h3, G, Gp,
                                     at<E>(ws, L.SD), at<E>(ws, L.bctr), at<E>(ws, L.breach),
                                     dh_part, dXp, first, st) != cudaSuccess)
        return FMS_ERR_CUDA;
      E* tmp = G;
      G = Gp;
      Gp = tmp;
      first = 0;
      hi = lo;
    }
  }
  if (unroll_unpack_rows<E>(G, rowsY, (int)m, d, g.DP, yperm, grad_seeds0, st) != cudaSuccess ||
      unroll_unpack_rows<E>(dXp, (int64_t)B * n, (int)n, d, g.DP,
                            P > 0 ? at<int32_t>(ws, L.s.perm) : nullptr, grad_points,
                            st) != cudaSuccess ||
      unroll_dh_sum(dh_part, B, unroll_seed_groups<E>(P, g, gr.per_set), grad_h, st) != cudaSuccess)
    return FMS_ERR_CUDA;
  return FMS_OK;
}

}  // namespace

extern "C" {

size_t fms_unrolled_ckpt_size(int32_t B, int64_t n, int64_t m, int32_t d, int32_t T, int32_t k) {
  if (!valid(B, n, m, d, T, k)) return 0;
  return ckpt_layout(geom(B, n, m, d), cells_for(B, n, m), T, k, 4).total;
}

size_t fms_unrolled_workspace_size(int32_t B, int64_t n, int64_t m, int32_t d, int32_t T,
                                   int32_t k) {
  if (!valid(B, n, m, d, T, k)) return 0;
  const UGeom g = geom(B, n, m, d);
  const int P = cells_for(B, n, m);
  const size_t f = fwd_layout(g, P, 4).total, b = bwd_layout(g, P, k, 4).total;
  return f > b ? f : b;
}

fms_status fms_unrolled_forward(const float* points, const float* seeds0, int32_t B, int64_t n,
                                int64_t m, int32_t d, float h, int32_t T, int32_t k,
                                float* out_seeds, void* ckpt, size_t ckpt_bytes, void* ws,
                                size_t ws_bytes, void* stream) {
  return forward_impl<float>(points, seeds0, B, n, m, d, h, T, k, out_seeds, ckpt, ckpt_bytes, ws,
                             ws_bytes, stream);
}

fms_status fms_unrolled_backward(const float* points, int32_t B, int64_t n, int64_t m, int32_t d,
                                 float h, int32_t T, int32_t k, const void* ckpt,
                                 size_t ckpt_bytes, const float* grad_out, float* grad_points,
                                 float* grad_seeds0, double* grad_h, void* ws, size_t ws_bytes,
                                 void* stream) {
  return backward_impl<float>(points, B, n, m, d, h, T, k, ckpt, ckpt_bytes, grad_out,
                              grad_points, grad_seeds0, grad_h, ws, ws_bytes, stream);
}

size_t fms_unrolled_ckpt_size_f64(int32_t B, int64_t n, int64_t m, int32_t d, int32_t T,
                                  int32_t k) {
  if (!valid(B, n, m, d, T, k)) return 0;
  return ckpt_layout(geom(B, n, m, d), cells_for(B, n, m), T, k, 8).total;
}

size_t fms_unrolled_workspace_size_f64(int32_t B, int64_t n, int64_t m, int32_t d, int32_t T,
                                       int32_t k) {
  if (!valid(B, n, m, d, T, k)) return 0;
  const UGeom g = geom(B, n, m, d);
  const int P = cells_for(B, n, m);
  const size_t f = fwd_layout(g, P, 8).total, b = bwd_layout(g, P, k, 8).total;
  return f > b ? f : b;
}

fms_status fms_unrolled_forward_f64(const double* points, const double* seeds0, int32_t B,
                                    int64_t n, int64_t m, int32_t d, double h, int32_t T,
                                    int32_t k, double* out_seeds, void* ckpt, size_t ckpt_bytes,
                                    void* ws, size_t ws_bytes, void* stream) {
  return forward_impl<double>(points, seeds0, B, n, m, d, h, T, k, out_seeds, ckpt, ckpt_bytes,
                              ws, ws_bytes, stream);
}

fms_status fms_unrolled_backward_f64(const double* points, int32_t B, int64_t n, int64_t m,
                                     int32_t d, double h, int32_t T, int32_t k, const void* ckpt,
                                     size_t ckpt_bytes, const double* grad_out,
                                     double* grad_points, double* grad_seeds0, double* grad_h,
                                     void* ws, size_t ws_bytes, void* stream) {
  return backward_impl<double>(points, B, n, m, d, h, T, k, ckpt, ckpt_bytes, grad_out,
                               grad_points, grad_seeds0, grad_h, ws, ws_bytes, stream);
}

}  // extern "C"

// Nearest-mode labels of a block's points, and rows scaled to unit length.
#pragma once

#include "fms_internal.cuh"

namespace fms {

// --- double-float arithmetic (Knuth's two-sum, Dekker / FMA two-product): ~2^-44
// relative, far below the FP32 rounding of the results; FP64 runs at a 64th of the
// FP32 rate here
struct Df {
  float h, l;
};
__device__ __forceinline__ Df df_sum(float a, float b) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ Df df_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ Df df_add(Df a, Df b) {
  Df s = df_sum(a.h, b.h);
  s.l = __fadd_rn(s.l, __fadd_rn(a.l, b.l));
  return df_sum(s.h, s.l);
}
__device__ __forceinline__ Df df_mul(Df a, Df b) {
  Df p = df_prod(a.h, b.h);
  p.l = __fadd_rn(p.l, __fmaf_rn(a.h, b.l, __fmul_rn(a.l, b.h)));
  return df_sum(p.h, p.l);
}

__device__ __forceinline__ float df_shift(float v, int shift) {
  return shift == 0 ? v : ldexpf(v, shift);
}

// scale / ||x|| for a row x[0 .. d): the squared length summed in double-float, then
// one Newton step on the FP32 reciprocal root (its 2^-22 squared is below 2^-43).
// Rows of extreme size are scaled by 2^*shift first, so no square over- or
// underflows.  Zero or non-finite rows: *ok = false.
template <typename Row>
__device__ __forceinline__ Df df_inverse_norm(Row&& x, int d, Df scale, bool* ok, int* shift) {
  float big = 0.0f;
  bool fine = true;
  for (int k = 0; k < d; ++k) {
    const float v = x(k);
    fine = fine && isfinite(v);
    big = fmaxf(big, fabsf(v));
  }
  *ok = fine && big > 0.0f;
  *shift = 0;
  if (!*ok) return {0.0f, 0.0f};
  if (!(big >= 0x1p-40f && big <= 0x1p40f)) {
    int e;
    frexpf(big, &e);
    *shift = -e;   // the largest entry comes to [1/2, 1)
  }
  Df nn = {0.0f, 0.0f};
  for (int k = 0; k < d; ++k) {
    const float v = df_shift(x(k), *shift);
    nn = df_add(nn, df_prod(v, v));
  }
  const float r0 = 1.0f / sqrtf(nn.h);
  // r = r0 + r0 (1 - nn r0^2) / 2
  Df t = df_mul(nn, df_prod(r0, r0));
  const float res = __fadd_rn(__fsub_rn(1.0f, t.h), -t.l);
  Df r = df_sum(r0, __fmul_rn(0.5f * r0, res));
  return df_mul(r, scale);
}
__device__ __forceinline__ float df_times(float x, Df f) {
  const Df p = df_prod(x, f.h);
  return __fadd_rn(p.h, __fmaf_rn(x, f.l, p.l));
}

// Labels and margins of points [j0, j1) of X (rows of d values) by a block of 256
// threads; the M modes (rows of d values) come in
// tiles of kLabelFloats / DP rows, zero padded to DP, through `sm`.  Ties go to the
// lowest mode.  Bound by FP32 issue (2 DP operations a point and mode) where modes
// are many, else by reading the points.
constexpr int kLabelFloats = 8192;

template <int DP, bool UNIT>
__device__ __forceinline__ void label_block(const float* __restrict__ X, int64_t j0, int64_t j1,
                                            int d, const float* __restrict__ modes, int M,
                                            int32_t* __restrict__ labels,
                                            float* __restrict__ margins, float* sm) {
  constexpr int TILE = kLabelFloats / DP;
  constexpr int U = DP <= 8 ? 1 : 2;   // points of a thread (narrow ones: more threads instead)
  const bool vec = (d & 3) == 0 && (reinterpret_cast<uintptr_t>(X) & 15u) == 0;
  for (int64_t jb = j0; jb < j1; jb += 256 * U) {
    float x[U][DP], b1[U], b2[U];
    int arg[U];
    int64_t j[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      j[u] = jb + u * 256 + threadIdx.x;
      b1[u] = b2[u] = INFINITY;
      arg[u] = -1;
      const float* r = X + (j[u] < j1 ? j[u] : j1 - 1) * d;
      if (vec) {
#pragma unroll
        for (int q = 0; q < DP / 4; ++q) {
          const float4 t = 4 * q < d ? __ldg(reinterpret_cast<const float4*>(r) + q)
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
          x[u][4 * q] = t.x;
          x[u][4 * q + 1] = t.y;
          x[u][4 * q + 2] = t.z;
          x[u][4 * q + 3] = t.w;
        }
      } else {
#pragma unroll
        for (int k = 0; k < DP; ++k) x[u][k] = k < d ? __ldg(r + k) : 0.0f;
      }
      if (UNIT) {
        bool ok;
        int sh;
        const Df f = df_inverse_norm([&](int k) { return __ldg(r + k); }, d, Df{1.0f, 0.0f}, &ok,
                                     &sh);
#pragma unroll
        for (int k = 0; k < DP; ++k) x[u][k] = df_times(df_shift(x[u][k], sh), f);
      }
    }
    for (int m0 = 0; m0 < M; m0 += TILE) {
      const int mt = min(TILE, M - m0);
      if (m0 > 0 || jb == j0 || M > TILE) {   // (one tile stays)
        __syncthreads();
        for (int e = threadIdx.x; e < mt * DP; e += 256) {
          const int k = e % DP;
          sm[e] = k < d ? modes[(int64_t)(m0 + e / DP) * d + k] : 0.0f;
        }
        __syncthreads();
      }
      for (int m = 0; m < mt; ++m) {
        float d2[U];
#pragma unroll
        for (int u = 0; u < U; ++u) d2[u] = 0.0f;
#pragma unroll
        for (int q = 0; q < DP / 4; ++q) {
          const float4 t = *reinterpret_cast<const float4*>(sm + m * DP + 4 * q);
#pragma unroll
          for (int u = 0; u < U; ++u) {
            float e = x[u][4 * q] - t.x;
            d2[u] = fmaf(e, e, d2[u]);
            e = x[u][4 * q + 1] - t.y;
            d2[u] = fmaf(e, e, d2[u]);
            e = x[u][4 * q + 2] - t.z;
            d2[u] = fmaf(e, e, d2[u]);
            e = x[u][4 * q + 3] - t.w;
            d2[u] = fmaf(e, e, d2[u]);
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (d2[u] < b1[u]) {
            b2[u] = b1[u];
            b1[u] = d2[u];
            arg[u] = m0 + m;
          } else if (d2[u] < b2[u]) {
            b2[u] = d2[u];
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (j[u] >= j1) continue;
      labels[j[u]] = arg[u];
      if (margins) margins[j[u]] = M > 1 ? sqrtf(b2[u]) - sqrtf(b1[u]) : INFINITY;
    }
  }
}

}  // namespace fms

// Device helpers shared by the dense factorisation kernels (qr.cu, jacobi.cu).
#pragma once

#include <float.h>

#include "common.cuh"

namespace dense {

template <class R> struct Lim;
template <> struct Lim<float> {
  static constexpr float eps = FLT_EPSILON, tiny = FLT_MIN, big = FLT_MAX;
};
template <> struct Lim<double> {
  static constexpr double eps = DBL_EPSILON, tiny = DBL_MIN, big = DBL_MAX;
};

template <class R>
__device__ __forceinline__ R wsum(R v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 1 / sqrt(x) and 1 / x to within a few units in the last place for normal x.
// FP64 divisions and square roots of the CUDA library take tens of FP64
// instructions each, and one FP64 warp instruction holds this part's FP64
// pipe for 16 cycles; a hardware approximation (about 20 bits) corrected by
// Newton steps takes about ten.  Arguments near the ends of the range (where
// the approximation flushes or an intermediate could leave the normal range)
// go to the library's functions.
__device__ __forceinline__ float rsqrt_nr(float x) {
  // the correction is added (y + y e / 2): multiplying by 1.5 - x y^2 / 2 rounds
  // next to 1, where the spacing changes, and leaves a bias of -1.7e-8
  const float y = rsqrtf(x);
  return fmaf(0.5f * y, fmaf(-x * y, y, 1.0f), y);
}
__device__ __forceinline__ double rsqrt_nr(double x) {
  if (!(x > 1e-290 && x < 1e290)) return 1.0 / sqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  double e = fma(-x * y, y, 1.0);            // third-order step: 20 -> 60 bits
  y = fma(y * e, fma(0.375, e, 0.5), y);
  e = fma(-x * y, y, 1.0);                   // rounding of the first step
  return fma(0.5 * y, e, y);
}
__device__ __forceinline__ float rcp_nr(float x) { return 1.0f / x; }
__device__ __forceinline__ double rcp_nr(double x) {
  const double ax = fabs(x);
  if (!(ax > 1e-290 && ax < 1e290)) return 1.0 / x;
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  double e = fma(-x, y, 1.0);
  y = fma(y, fma(e, e, e), y);
  e = fma(-x, y, 1.0);
  return fma(y, e, y);
}

// Compensated accumulation (Knuth's TwoSum): hi + lo += t.
template <class R>
__device__ __forceinline__ void add_comp(R& hi, R& lo, R t) {
  const R s = hi + t, bb = s - hi;
  lo += (hi - (s - bb)) + (t - bb);
  hi = s;
}
// the lanes' compensated sums added up, in every lane
template <class R>
__device__ __forceinline__ void wsum_comp(R& hi, R& lo) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const R ohi = __shfl_xor_sync(0xffffffffu, hi, o), olo = __shfl_xor_sync(0xffffffffu, lo, o);
    lo += olo;
    add_comp(hi, lo, ohi);
  }
}

// Brings a vector whose norm is 1 to single precision (entries on the lanes, N each)
// to the norm 1 that its stored entries allow: x += x (1 - |x|^2) / 2.  The sum of
// squares is compensated.  A rounding's vectors and reflections are used as
// exactly orthonormal, bond after bond, and a norm that is off scales
// everything: left as the factorisations leave them (1e-7) they were half of
// what a complex64 solve's error owed to them.
template <int N>
__device__ __forceinline__ void unit_norm(cplx<float> (&x)[N]) {
  float hi = 0, lo = 0;
#pragma unroll
  for (int u = 0; u < N; ++u) add_comp(hi, lo, abs2(x[u]));
  wsum_comp(hi, lo);
  const float k = -0.5f * ((hi - 1.0f) + lo);
#pragma unroll
  for (int u = 0; u < N; ++u) x[u] = cplx<float>(fmaf(x[u].re, k, x[u].re), fmaf(x[u].im, k, x[u].im));
}

}  // namespace dense

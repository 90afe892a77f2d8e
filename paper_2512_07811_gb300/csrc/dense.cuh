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

// 1 / sqrt(x) and 1 / x by Newton's method from an approximation that the
// hardware gives (rsqrt.approx, rcp.approx of the PTX ISA; about 20 bits in FP64).
// One FP64 warp instruction holds this part's FP64 pipe for 16 cycles and a
// dependent one takes 75, so that the accuracy is bought no further than
// needed and the chain kept short.
//
// Newton's method on f(y) = 1 / y^2 - x: with e = 1 - x y^2 the root is y (1 - e)^(-1/2) =
// y (1 + e / 2 + 3 e^2 / 8 + 5 e^3 / 16 + ...), the step y + y e / 2 keeps the first
// two terms and leaves 3 e^2 / 8: from |e| <= 2^-19 to 2^-39, then 2^-78.  The
// rounding of the last step leaves e good to 2^-53 and y to 2 units in the last
// place.  Newton's method on f(y) = 1 / y - x: e = 1 - x y, the root is y / (1 - e) =
// y (1 + e + ...), the step y + y e leaves e^2 (2^-40, then 2^-80); here e is exact but
// for its own last place: 1 unit.
// The third-order step (the same series with its third term: Householder's
// iteration of that order) goes from 2^-19 to 5 e^3 / 16 = 2^-58 at once: 2 units.
// Arguments near the ends of the range, where the approximation flushes
// subnormal values to zero, go to the library's functions.
__device__ __forceinline__ float rsqrt_nr(float x) {
  // the correction is added (y + y e / 2): multiplying by 1.5 - x y^2 / 2 rounds
  // next to 1, where the spacing changes, and leaves a bias of -1.7e-8
  const float y = rsqrtf(x);
  return fmaf(0.5f * y, fmaf(-x * y, y, 1.0f), y);
}
__device__ __forceinline__ double rsqrt_approx(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  return y;
}
__device__ __forceinline__ double rsqrt_newton(double x, double y) { return fma(0.5 * y, fma(-x * y, y, 1.0), y); }
__device__ __forceinline__ double rsqrt_third_order(double x, double y) {
  const double e = fma(-x * y, y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ double rsqrt_nr(double x) {
  if (!(x > 1e-290 && x < 1e290)) return 1.0 / sqrt(x);
  return rsqrt_newton(x, rsqrt_newton(x, rsqrt_approx(x)));
}
__device__ __forceinline__ float rcp_nr(float x) { return 1.0f / x; }
__device__ __forceinline__ double rcp_nr(double x) {
  const double ax = fabs(x);
  if (!(ax > 1e-290 && ax < 1e290)) return 1.0 / x;
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  y = fma(y, fma(-x, y, 1.0), y);
  return fma(y, fma(-x, y, 1.0), y);
}

// Compensated sums in working precision: a partial sum carries its rounding
// error (Knuth's TwoSum), so that a sum of squares over a column is good to a few
// units in the last place however many terms it has, without FP64 arithmetic
// (slow on this part).  hi + lo += t.
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
// exactly orthonormal, bond after bond, and a norm that is off (by 1.4 u, as the
// factorisations leave them) scales everything: C_eff of 16^3 complex64 solves
// with exact operators 1.8e-6 / 1.3e-6 off without / with it, at 1 % of a rounding.
// (FP64 solves do not gain: 7.5e-15 / 6.8e-15, runs scatter by 3e-15.)
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

// Exponent of a positive finite value, at least `least`, which also stands for
// zero and for what is not finite; 2^e.
__device__ __forceinline__ int exponent_of(float a, int least) {
  return a > 0 && a <= FLT_MAX ? max(ilogbf(a), least) : least;
}
__device__ __forceinline__ int exponent_of(double a, int least) {
  return a > 0 && a <= DBL_MAX ? max(ilogb(a), least) : least;
}
__device__ __forceinline__ float pow2(float, int e) { return ldexpf(1.f, e); }
__device__ __forceinline__ double pow2(double, int e) { return ldexp(1.0, e); }

}  // namespace dense

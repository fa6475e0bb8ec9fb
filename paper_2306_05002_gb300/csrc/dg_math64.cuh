// dg_math64.cuh -- FP64 building blocks of the kernels that the FP64 pipe bounds (GB300, sm_103a).
//
// GB300 executes two FP64 operations per clock and SM, so a warp instruction holds the pipe for 16
// clocks while integer and logic instructions run beside it for nothing.  Everything here therefore
// counts FP64 instructions: sign flips, comparisons of bit patterns and classifications are integer
// operations, and reciprocals and square roots are one step of a third-order iteration on the
// hardware's approximation instead of a correctly rounded division.
#pragma once

#include <cuda_runtime.h>

namespace dgpf {

__device__ __forceinline__ unsigned hi_abs(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// isfinite without an FP64 comparison.
__device__ __forceinline__ bool finite64(double x) { return hi_abs(x) < 0x7ff00000u; }

// x <= 0, false for a NaN, without an FP64 comparison.
__device__ __forceinline__ bool nonpositive64(double x) {
  const long long b = __double_as_longlong(x);
  const unsigned long long m = (unsigned long long)b & 0x7fffffffffffffffull;
  return m == 0ull || (b < 0 && m <= 0x7ff0000000000000ull);
}

// x with its sign bit flipped where mask has bit 31 set (mask: 0 or 0x80000000).
__device__ __forceinline__ double flip64(double x, int mask) {
  return __hiloint2double(__double2hiint(x) ^ mask, __double2loint(x));
}

// fmax of two values that are non-negative or NaN (a NaN gives way to the other), by their bits.
__device__ __forceinline__ double max_nonneg64(double a, double b) {
  const unsigned long long inf = 0x7ff0000000000000ull;
  const unsigned long long ua = (unsigned long long)__double_as_longlong(a) & 0x7fffffffffffffffull;
  const unsigned long long ub = (unsigned long long)__double_as_longlong(b) & 0x7fffffffffffffffull;
  const bool take_b = ua > inf || (ub <= inf && ub > ua);
  return take_b ? b : a;
}

// x >= 1e-24 for x >= 0 or NaN (false for a NaN): the cut-off of |grad psi|^2.
__device__ __forceinline__ bool has_gradient(double g2) {
  const long long b = __double_as_longlong(g2);
  return b >= __double_as_longlong(1e-24) && b <= 0x7ff0000000000000ll;
}

// x < 1e-24 for x >= 0 or NaN (false for a NaN), without an FP64 comparison: the same cut-off where a NaN
// has to stay one.
__device__ __forceinline__ bool no_gradient(double g2) {
  return (unsigned long long)__double_as_longlong(g2) < (unsigned long long)__double_as_longlong(1e-24);
}

// Exponents for which the iterations below neither overflow nor lose bits to gradual underflow:
// 2^-500 .. 2^500.  Zeros, infinities, NaNs, subnormals and everything outside go to CUDA's own
// functions (never in a physical state; the branch is not taken).
__device__ __forceinline__ bool mid_range64(double x) {
  return ((unsigned)__double2hiint(x) >> 20) - 523u <= 1000u;  // sign bit clear as well
}

__device__ __noinline__ inline double rcp64_slow(double x) { return 1.0 / x; }
__device__ __noinline__ inline double rsqrt64_slow(double x) { return rsqrt(x); }
__device__ __noinline__ inline double sqrt64_slow(double x) { return sqrt(x); }

// 1 / x.  With y the hardware approximation (PTX rcp.approx.ftz.f64) and e = 1 - x y,
// 1 / x = y (1 + e + e^2 + ...): Householder's third-order step y + y (e + e^2), 3 operations.
__device__ __forceinline__ double rcp64(double x) {
  if (!mid_range64(fabs(x))) return rcp64_slow(x);
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  double e = fma(-x, y, 1.0);
  e = fma(e, e, e);
  return fma(y, e, y);
}

// 1 / sqrt(x).  With y the hardware approximation (PTX rsqrt.approx.ftz.f64) and e = 1 - x y^2,
// 1 / sqrt(x) = y (1 - e)^(-1/2) = y (1 + e / 2 + 3 e^2 / 8 + ...), 5 operations.
__device__ __forceinline__ double rsqrt64(double x) {
  if (!mid_range64(x)) return rsqrt64_slow(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-(x * y), y, 1.0);
  return fma(y * e, fma(e, 0.375, 0.5), y);
}

// sqrt(x) = x / sqrt(x) by the same series on t = x y, 5 operations.
__device__ __forceinline__ double sqrt64(double x) {
  if (!mid_range64(x)) return sqrt64_slow(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double t = x * y;
  const double e = fma(-t, y, 1.0);
  return fma(t * e, fma(e, 0.375, 0.5), t);
}

// The correctly rounded forms: a residual step on the third-order result (Markstein: with y within
// a unit of 1 / b, fma(y, fma(-b, y, 1), y) is the rounded reciprocal, and fma(r, y, q), q = a y and
// r = a - b q, the rounded quotient).  A quotient then costs three operations after its denominator's
// five.
// The theorem's one exception is a denominator whose significand is all ones, e.g. 1 - 2^-53 (which a
// sum of partial densities can be): CUDA's division takes it.
__device__ __forceinline__ double rcp64_rn(double x) {
  if (!mid_range64(fabs(x)) || ((unsigned long long)__double_as_longlong(x) << 12) == 0xfffffffffffff000ull)
    return rcp64_slow(x);
  const double y = rcp64(x);
  return fma(y, fma(-x, y, 1.0), y);
}

__device__ __noinline__ inline double div64_slow(double a, double b) { return a / b; }

// a / b, y = rcp64_rn(b).
__device__ __forceinline__ double div64_rn(double a, double b, double y) {
  const double q = a * y;
  const bool zero = (__double_as_longlong(a) << 1) == 0;  // then q, with its sign
  if (!mid_range64(fabs(b)) || !(zero || mid_range64(fabs(a)))) return div64_slow(a, b);
  if (zero) return q;
  return fma(fma(-b, q, a), y, q);
}

// sqrt(x), correctly rounded: s = t (1 + d), t = x y and d = e / 2 + 3 e^2 / 8 (sqrt64), then the
// residual step s + (x - s^2) / (2 sqrt(x)).  Its multiplier has to be good to about a unit in the last
// place, so it is y (1 + d) / 2, not y / 2.  With u = 2^-53: the rounding of t moves s and y (1 + d) by
// u / 2, so s is within a unit of the root, x - s^2 is exact, and the multiplier is off by at most 3 u / 2
// (its own rounding included), the correction, half a unit near a boundary S + 1/2, by less than 3 u / 4 of a
// unit.  The root nearest to a boundary has x = S^2 + S + j with a small j, and j is even: for |j| >= 2 the
// distance is at least 7 / (8 S), of which the step's second order takes 1 / (8 S), which leaves more than
// 3 u / 4.  j = 0 only for 1 - 2^-53 and 1 + 2^-52 times powers of four, both rounded right.
__device__ __forceinline__ double sqrt64_rn(double x) {
  if (!mid_range64(x)) return sqrt64_slow(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double t = x * y;
  const double e = fma(-t, y, 1.0);
  const double d = e * fma(e, 0.375, 0.5);
  const double s = fma(t, d, t), r = fma(y, d, y);
  const double h = __hiloint2double(__double2hiint(r) - 0x100000, __double2loint(r));  // r / 2
  return fma(fma(-s, s, x), h, s);
}

}  // namespace dgpf

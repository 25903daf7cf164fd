// fp64_math.cuh -- reciprocal and roots with few FP64-pipe instructions.
//
// GB300 runs FP64 at 1/64 of its FP32 rate, so the FP64 kernels are bound by
// the number of FP64 instructions; a full-range division or root takes a
// dozen and more.  These start from the hardware's gross approximations
// (PTX rcp.approx.ftz.f64, rsqrt.approx.ftz.f64: relative error below 2^-19)
// and take one third-order step of the Newton-Halley iteration, which leaves
// a relative error below 2^-56 plus the roundings: below 0.6 units in the last
// place for the reciprocal, 1.7 for the quotient, 1.1 for the root and 1.2 for
// its reciprocal, for arguments and results in the normal range.  The FP32
// overloads are the plain operations.
#pragma once
#include <cuda_runtime.h>

namespace phl {

// 1/x: y (1 + e + e^2), e = 1 - x y.  Three FP64 multiply-adds.  Zero, an
// argument below the normal range and infinity give NaN; above 2^1022, where
// the result is below the normal range, it is 0.
__device__ __forceinline__ double rcp_nr(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ float rcp_nr(float x) { return 1.0f / x; }

__device__ __forceinline__ double div_nr(double a, double b) { return a * rcp_nr(b); }
__device__ __forceinline__ float div_nr(float a, float b) { return a / b; }

// true where |x| is below the normal range (integer test: no FP64 compare)
__device__ __forceinline__ bool below_normal(double x) {
  return ((unsigned)__double2hiint(x) & 0x7fffffffu) < 0x00100000u;
}

// x > 0 without an FP64 compare (those run on the FP64 pipe): positive doubles
// order as their bits, 0 wraps to the top.  The second form is false for
// infinity too.
__device__ __forceinline__ bool positive(double x) {
  return (unsigned long long)__double_as_longlong(x) - 1ull < 0x7ff0000000000000ull;
}
__device__ __forceinline__ bool positive_finite(double x) {
  return (unsigned long long)__double_as_longlong(x) - 1ull < 0x7fefffffffffffffull;
}
__device__ __forceinline__ bool positive(float x) { return x > 0.0f; }
// lo < x < hi for positive lo, hi: positive doubles order as their bits (false
// for NaN, no FP64 compare)
__device__ __forceinline__ bool between_pos(double x, double lo, double hi) {
  const long long b = __double_as_longlong(x);
  return b > __double_as_longlong(lo) && b < __double_as_longlong(hi);
}
__device__ __forceinline__ bool between_pos(float x, float lo, float hi) { return x > lo && x < hi; }
// |x| < 2^-E by the exponent field
template <int E>
__device__ __forceinline__ bool below_pow2(double x) {
  return ((unsigned)__double2hiint(x) & 0x7fffffffu) < ((1023u - E) << 20);
}
template <int E>
__device__ __forceinline__ bool below_pow2(float x) { return fabsf(x) < 1.0f / (float)(1u << E); }

// Interval index and fraction of a table position g in [0, n]: false outside
// (NaN included).  In FP64 the index and the whole part come out of the high
// word by shifts (positions below 2^20), so the only FP64 instruction is the
// fraction's subtraction; conversions each way and compares would be four more.
// With the bit tests above, the stellar cells of a mixed stage on 128^3 take
// 947 us against 1032.
__device__ __forceinline__ bool interval(double g, int n, int &i, double &u) {
  const int hi = __double2hiint(g);
  const int e = (hi >> 20) - 1023;          // negative g: hi < 0, e < -1023
  if (hi < 0 || e > 19) {                   // -0, or too far out for the high word alone
    if (!(g >= 0.0 && g <= (double)n)) return false;
    i = min((int)g, n - 1);
    u = g - (double)i;
    return true;
  }
  const bool whole = e >= 0;
  const int sh = 20 - (whole ? e : 0);
  i = whole ? ((hi & 0xfffff) | 0x100000) >> sh : 0;
  u = g - (whole ? __hiloint2double((hi >> sh) << sh, 0) : 0.0);
  if (i >= n) {                             // the last node itself, or beyond
    if (i > n || u > 0.0) return false;
    i = n - 1;
    u = 1.0;
  }
  return true;
}
__device__ __forceinline__ bool interval(float g, int n, int &i, float &u) {
  if (!(g >= 0.0f && g <= (float)n)) return false;
  i = (int)g;
  if (i > n - 1) i = n - 1;
  u = g - (float)i;
  return true;
}

// x < 0 ? 0 : x by the sign bit (-0 gives +0); NaN stays NaN
__device__ __forceinline__ double not_below_zero(double x) {
  const int hi = __double2hiint(x);
  return (hi < 0 && (unsigned)hi <= 0xfff00000u) ? 0.0 : x;
}
__device__ __forceinline__ float not_below_zero(float x) { return x < 0.0f ? 0.0f : x; }

// sqrt(x) and, in the second form, 1/sqrt(x): with y ~ 1/sqrt(x) and r = 1 -
// x y^2, both are the approximation times 1 + r/2 + 3 r^2/8 (remaining error
// 5 r^3 / 16 < 2^-55).  Five (six) FP64 instructions.  An argument below the
// normal range, of either sign, gives 0 (infinity for the reciprocal), other
// negative ones and +infinity NaN.
__device__ __forceinline__ double sqrt_nr(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double t = x * y, r = fma(-t, y, 1.0);
  const double s = fma(t, r * fma(r, 0.375, 0.5), t);
  return below_normal(x) ? 0.0 : s;
}
__device__ __forceinline__ float sqrt_nr(float x) { return sqrtf(x); }

__device__ __forceinline__ void sqrt_rsqrt_nr(double x, double &s, double &rs) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double t = x * y, r = fma(-t, y, 1.0);
  const double p = r * fma(r, 0.375, 0.5);
  const bool z = below_normal(x);
  s = z ? 0.0 : fma(t, p, t);
  rs = z ? __longlong_as_double(0x7ff0000000000000ll) : fma(y, p, y);
}

}  // namespace phl

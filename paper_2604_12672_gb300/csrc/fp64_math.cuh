// fp64_math.cuh -- reciprocal and roots with few FP64-pipe instructions.
//
// GB300 runs FP64 at 1/64 of its FP32 rate, so the FP64 kernels are bound by
// the number of FP64 instructions; a full-range division or root takes a
// dozen and more.  These start from the hardware's gross approximations
// (PTX rcp.approx.ftz.f64, rsqrt.approx.ftz.f64: relative error below 2^-19)
// and take one third-order step of the Newton-Halley iteration, which leaves
// a relative error below 2^-56 plus the rounding of the last operation: about
// one unit in the last place for normal arguments.  The FP32 overloads are
// the plain operations.
#pragma once
#include <cuda_runtime.h>

namespace phl {

// 1/x: y (1 + e + e^2), e = 1 - x y.  Three FP64 multiply-adds.  0 and
// infinity give NaN.
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

// x > 0 without an FP64 compare (those run on the FP64 pipe): true for
// positive finite values from 2^-1042 up; false for NaN and infinity too.
__device__ __forceinline__ bool positive(double x) { return (unsigned)__double2hiint(x) - 1u < 0x7fefffffu; }
__device__ __forceinline__ bool positive(float x) { return x > 0.0f; }
// x < 0 ? 0 : x by the sign bit; NaN stays NaN
__device__ __forceinline__ double not_below_zero(double x) {
  const int hi = __double2hiint(x);
  return (hi < 0 && (unsigned)hi <= 0xfff00000u) ? 0.0 : x;
}
__device__ __forceinline__ float not_below_zero(float x) { return x < 0.0f ? 0.0f : x; }

// sqrt(x) and, in the second form, 1/sqrt(x): with y ~ 1/sqrt(x) and r = 1 -
// x y^2, both are the approximation times 1 + r/2 + 3 r^2/8 (remaining error
// 5 r^3 / 16 < 2^-57).  Five (six) FP64 instructions.  An argument below the
// normal range gives 0 (infinity for the reciprocal), a negative one NaN.
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

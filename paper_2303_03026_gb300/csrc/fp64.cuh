// Reciprocal, square root and comparisons for code bound by the FP64 pipe.
//
// GB300 issues 2 FP64 lanes per clock and SM (a 32nd of a warp's width per
// scheduler and cycle), so in double every operation of that pipe counts and
// the integer pipe is idle.  The IEEE division and square root take 8 to 10 FP64
// operations each; here the hardware's approximation (PTX rcp.approx /
// rsqrt.approx, the upper 32 bits of the result) is refined by one third-order
// Householder step, which leaves the truncation error below 2^-58:
//   reciprocal    e = 1 - b x:   x (1 + e + e^2)             3 FP64 operations
//   square root   e = 1 - a y^2: y (1 + e/2 + 3 e^2/8)       5
// within 1 ulp of the rounded result (tests/test_gpu_fp64_math.py).  Signs and
// orders are read from the bit patterns on the integer pipe.
// float keeps the plain operators: its units are compiled with the hardware's
// approximations.
#pragma once

#include <cuda_runtime.h>

namespace amrvac {

constexpr unsigned long long F64_INF = 0x7ff0000000000000ull;

__device__ __forceinline__ unsigned long long bits64(double x) {
  return (unsigned long long)__double_as_longlong(x);
}

// biased exponent 1 .. 2045: zero, subnormal, 2^1023 and above, infinities and
// NaN (whose approximation is 0 or infinite) are left to the caller's fallback.
// (A reciprocal that would be subnormal, of 2^1022 and above, is 0, and that of a
// subnormal number infinite.)
__device__ __forceinline__ bool mid_range(double x) {
  const unsigned e = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
  return e - 1u < 2045u;
}

__device__ __forceinline__ double rcp_T(double b) {
  double x;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(b));
  const double e = fma(-b, x, 1.0);
  const double r = fma(x, fma(e, e, e), x);
  return mid_range(b) ? r : x;  // +-inf of 0, +-0 of an infinity, NaN of NaN
}
__device__ __forceinline__ float rcp_T(float b) { return 1.f / b; }

// (a subnormal argument is returned as it is, of the order of zero here)
__device__ __forceinline__ double sqrt_T(double a) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  const double h = a * y;
  const double e = fma(-h, y, 1.0);
  const double r = fma(h, e * fma(e, 0.375, 0.5), h);
  // zero, +inf and NaN are their own roots; the root of -inf is the NaN of h
  const unsigned hi = (unsigned)__double2hiint(a);
  const bool mid = ((hi >> 20) & 0x7ffu) - 1u < 2046u;
  return mid ? r : (hi == 0xfff00000u ? h : a);
}
__device__ __forceinline__ float sqrt_T(float a) { return sqrtf(a); }

// sqrt(a) and 1/sqrt(a) together: 6 FP64 operations
__device__ __forceinline__ void sqrt_pair(double a, double& s, double& is) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  const double e = fma(-(a * y), y, 1.0);
  const double r = fma(y, e * fma(e, 0.375, 0.5), y);
  const bool mid = mid_range(a);
  is = mid ? r : y;
  s = mid ? a * r : a;
}
__device__ __forceinline__ void sqrt_pair(float a, float& s, float& is) {
  s = sqrtf(a);
  is = 1.f / s;
}

// x > 0 and x >= 0 (false for NaN)
__device__ __forceinline__ bool gt0(double x) { return bits64(x) - 1ull < F64_INF; }
__device__ __forceinline__ bool ge0(double x) {
  return bits64(x) <= F64_INF || bits64(x) == 0x8000000000000000ull;
}
__device__ __forceinline__ bool gt0(float x) { return x > 0.f; }
__device__ __forceinline__ bool ge0(float x) { return x >= 0.f; }

// smaller and larger of two values that are not negative
__device__ __forceinline__ double min_pos(double a, double b) {
  return bits64(a) < bits64(b) ? a : b;
}
__device__ __forceinline__ float min_pos(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ double max_pos(double a, double b) {
  return bits64(a) < bits64(b) ? b : a;
}
__device__ __forceinline__ float max_pos(float a, float b) { return fmaxf(a, b); }
// a <= b for values that are not negative
__device__ __forceinline__ bool le_pos(double a, double b) { return bits64(a) <= bits64(b); }
__device__ __forceinline__ bool le_pos(float a, float b) { return a <= b; }

}  // namespace amrvac

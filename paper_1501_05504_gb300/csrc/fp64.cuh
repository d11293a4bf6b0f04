// Device helpers that keep FP64 instructions out of scalar chains.  GB300 issues
// FP64 at 1/64 of its FP32 rate (a warp instruction in ~64 cycles of a
// sub-partition); integer and FP32 instructions are nearly free beside it.
#pragma once

#include <cstdint>

namespace dmrg3s {
namespace {

// A double's top 24 bits as a float with the power of two 2^(e - 1023) taken out
// (truncated; 0 where that is below the float range), and a float (normal) times
// 2^e as a double (0 below the double range).  Integer instructions.
__device__ __forceinline__ float float_of(double x, int e) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int fe = (int)((u >> 52) & 0x7ff) - e + 127;
  const unsigned sign = (unsigned)(u >> 32) & 0x80000000u;
  return fe < 1 ? 0.f : __uint_as_float(sign | (unsigned)fe << 23 | ((unsigned)(u >> 29) & 0x7fffffu));
}
__device__ __forceinline__ double double_of(float x, int e) {
  const unsigned u = __float_as_uint(x);
  const int de = (int)((u >> 23) & 0xff) + 896 + e;
  const unsigned long long m = (unsigned long long)(u & 0x7fffffu) << 29;
  const unsigned long long sign = (unsigned long long)(u & 0x80000000u) << 32;
  return de < 1 ? 0.0 : __longlong_as_double((long long)(sign | (unsigned long long)de << 52 | m));
}
__device__ __forceinline__ int exponent_of(double x) {   // biased by 1023; 0: zero or subnormal
  return (int)(__double_as_longlong(x) >> 52) & 0x7ff;
}
// 2^-(exponent of x), for a finite x
__device__ __forceinline__ double inverse_scale(double x) {
  const int e = exponent_of(x);
  return double_of(1.0f, 1023 - (e < 1 ? 1 : e > 2040 ? 2040 : e));
}

// 1 / x within one unit in the last place of the rounded value (|x| within
// 2^+-1000): an FP32 reciprocal r0 of the mantissa, then the third-order Newton step
// 1 / x = r0 (1 + e + e^2 + ..) with e = 1 - x r0 below 2^-21 (e^3 is left out, 2^-63; the
// last multiply-add rounds once).  Three dependent FP64 instructions.
__device__ __forceinline__ double recip(double x) {
  const int e = exponent_of(x);
  const double r0 = double_of(1.0f / float_of(x, e), 1023 - e);
  const double d = fma(-x, r0, 1.0);
  return fma(r0, fma(d, d, d), r0);
}

// sqrt(x) within one unit in the last place of the rounded value (0 < x < 2^1000,
// normal): with x = m 2^(2k), m in [1, 4), the FP32 rsqrt of m and Goldschmidt's
// coupled Newton iteration for g ~ sqrt(m) and h ~ 1 / (2 sqrt(m)), then Markstein's
// correction g + h (m - g^2) (IBM J. Res. Dev. 34, 1990), which rounds once.  Six
// dependent FP64 instructions.
__device__ __forceinline__ double sqrt_of(double x) {
  const int e = exponent_of(x), k = (e - 1023) >> 1;
  const double m = __longlong_as_double(__double_as_longlong(x) - ((long long)(2 * k) << 52));
  const double y = double_of(rsqrtf((float)m), 0);
  double g = m * y, h = 0.5 * y;
  const double r = fma(-g, h, 0.5);
  g = fma(g, r, g);
  h = fma(h, r, h);
  g = fma(fma(-g, g, m), h, g);
  return __longlong_as_double(__double_as_longlong(g) + ((long long)k << 52));
}

}  // namespace
}  // namespace dmrg3s

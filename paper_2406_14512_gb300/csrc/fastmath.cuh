// fastmath.cuh -- reciprocals, reciprocal square roots and conversions at the
// cost of few instructions, FP64 ones above all: this GPU's FP64 pipe does two
// operations per clock and SM, and its library roots, divisions and float ->
// double conversions (one operation each) are what bounds FP64 work here.
#pragma once
#include <cuda_runtime.h>

namespace hff {

// FP32 reciprocal and reciprocal square root as the single approximate
// hardware instructions (about 1-2 ulp, denormals flushed): their arguments
// here are squared norms, radii and ratios of per-step increments, never
// denormal, and the results enter quantities compared with the FP64 oracle at
// 1e-5 relative.  FP64 ones from the hardware's approximations y (the upper 32
// bits of a double, 20 bits after the point: taken as better than 2^-19) by one
// step of a series.  With e = 1 - x y the reciprocal is y / (1 - e) =
// y (1 + e + e^2 + e^3 + O(e^4)), the remainder below 2^-75.  With e = 1 - x y^2,
// where y^2 is exact, the reciprocal square root is y (1 - e)^(-1/2) =
// y (1 + e/2 + 3 e^2 / 8 + O(e^3)), the remainder (5/16) e^3 below 2^-55.  What is
// left is the rounding of the last operation.  Over 4e6 arguments the reciprocal
// is that of 1 / x and the root that of rsqrt to the last bit (without e^3, and
// with x y rounded before its product with y, they were off by 1.002 and 1.25
// times half an ulp).  Four and five FP64 operations instead of the eight to ten
// of the library's: the FP64 push is bound by the FP64 pipe, two operations per
// clock and SM.  Arguments near the ends of the range go to the library.
__device__ __forceinline__ float rsq(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ unsigned exponent_field(double x) { return ((unsigned)__double2hiint(x) >> 20) & 0x7ffu; }
__device__ __forceinline__ bool mid_range(double x) { return exponent_field(x) - 32u < 2047u - 64u; }
__device__ __forceinline__ double rsq(double x) {
  if (!mid_range(x)) return rsqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y * y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ double rcp(double x) {
  if (!mid_range(x)) return 1.0 / x;
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(fma(e, e, e), e, e), y);
}

// float -> double: for normal numbers the bits moved on the integer pipe (a
// conversion costs as much as an FP64 addition)
__device__ __forceinline__ double to_double(float x) {
  const unsigned b = __float_as_uint(x), e = (b >> 23) & 0xffu;
  if (e - 1u >= 254u) return (double)x;   // zero, denormal, infinity, NaN
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}
__device__ __forceinline__ double to_double(double x) { return x; }

}  // namespace hff

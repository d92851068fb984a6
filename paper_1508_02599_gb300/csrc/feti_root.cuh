// Reciprocals and reciprocal roots of positive normal numbers without the FP64
// divide and root, whose FP64 instructions hold a scheduler for 64 clocks each.
//
// The seed is the FP32 result for the mantissa (for the root: of d or 2 d, exponent
// even), the power of two is put on in integers.  One third-order Householder step
// (error e -> e^3) takes its 22 bits to full precision in three (five) FP64
// operations: within 1 (1.3) half-ulps of the exact value.
#pragma once
#include "feti_fixed.cuh"

namespace feti {
namespace {

__device__ __forceinline__ float mant_f32(double d) {  // in [1, 2), truncated
  return __int_as_float(0x3f800000 | ((__double2hiint(d) << 3) & 0x7ffff8) | ((unsigned)__double2loint(d) >> 29));
}
__device__ __forceinline__ double widen(float y, int e) {  // y 2^e for a normal y, in integers
  const int b = __float_as_int(y);
  return __hiloint2double(((((b >> 23) & 0xff) + 896 + e) << 20) | ((b >> 3) & 0xfffff), b << 29);
}
// 1 / d for d below 2^1022, above which the seed would leave the normal range
__device__ __forceinline__ double recip(double d) {
  const double y = widen(__frcp_rn(mant_f32(d)), 1023 - bexp64(d));
  const double e = fma(-d, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double inv_sqrt(double d) {
  const int k = bexp64(d) - 1023, odd = k & 1;
  const double y = widen(rsqrtf(mant_f32(d) * (odd ? 2.0f : 1.0f)), (odd - k) >> 1);
  const double e = fma(-d * y, y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ float recip(float d) { return 1.0f / d; }
__device__ __forceinline__ float inv_sqrt(float d) { return 1.0f / sqrtf(d); }

__device__ __forceinline__ bool positive(double d) {  // positive, normal and finite, in integers
  const int hi = __double2hiint(d);
  return hi >= 0x00100000 && hi < 0x7ff00000;
}
__device__ __forceinline__ bool positive(float d) { return d > 0.0f && isfinite(d); }

}  // namespace
}  // namespace feti

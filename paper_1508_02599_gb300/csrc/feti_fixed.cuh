// Floating point to integers scaled by a power of two, rounded to nearest, ties
// to even.  Many values drop only a bit or two in these conversions, where ties
// away from zero would be a bias that all entries share (it made the inverse of
// a nearly singular local matrix six times less accurate).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace feti {
namespace {

// q 2^-r, q < 2^61 and a multiple of 2, 0 <= r <= 62
__device__ __forceinline__ long long shift_even(unsigned long long q, int r) {
  return (long long)((q + (((1ull << r) - 1) >> 1) + ((q >> r) & 1)) >> r);
}

// a b + c as one instruction (the compiler's own form of the expression takes
// one and a half, 28 against 46 lanes per clock and SM)
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(c) : "r"(a), "r"(b));
  return c;
}

// biased exponent of an FP64 number (0: zero or subnormal, 2047: not finite)
__device__ __forceinline__ int bexp64(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// The 53-bit integer mantissa of x (0 for zero and subnormal x) times
// 2^(EXTRA - r), rounded, with the sign of x; r < 0 only where x is zero
template <int EXTRA>
__device__ __forceinline__ long long fixed64(double x, int r) {
  const long long b = __double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7ff;
  const unsigned long long m = e ? ((unsigned long long)b & 0xfffffffffffffull) | 0x10000000000000ull : 0ull;
  const long long v = shift_even(m << EXTRA, min(max(r, 0), 62));
  return b < 0 ? -v : v;
}

}  // namespace
}  // namespace feti

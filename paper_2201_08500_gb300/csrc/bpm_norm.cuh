// Sums of |E|^2 in FP64 of FP32 fields.
#pragma once

#include <cuda_runtime.h>

namespace bpm {

// double(f) of a normal float in integer instructions: the conversion runs at
// the FP64 rate (two a clock and SM).
__device__ __forceinline__ double widen_f64(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned long long a = ((unsigned long long)(b & 0x7FFFFFFFu) + (896ull << 23)) << 29;
  return __longlong_as_double((long long)(a | ((unsigned long long)(b & 0x80000000u) << 32)));
}
// double(f) of any float (a conversion for the rest, even one that no lane takes,
// would hold the FP64 pipe all the same: sums over 128 planes of 512 x 512 513 -> 243 us).
__device__ __forceinline__ double widen_any(float f) {
  const bool small = (__float_as_uint(f) & 0x7F800000u) == 0;  // zero or denormal
  const float g = small ? f * 0x1p100f : f;
  const unsigned b = __float_as_uint(g), m = b & 0x7FFFFFFFu;
  unsigned long long a = ((unsigned long long)m + (small ? 796ull << 23 : 896ull << 23)) << 29;
  if (m == 0) a = 0;
  if (m >= 0x7F800000u) a |= 0x7FFull << 52;  // infinity, NaN
  return __longlong_as_double((long long)(a | ((unsigned long long)(b & 0x80000000u) << 32)));
}

// s + |f|^2: two FP64 instructions (with conversions, a product and a separate
// sum it was five, 20 us a channel of 8192 points on one SM).
__device__ __forceinline__ double add_norm(double s, float2 f) {
  const double x = widen_any(f.x), y = widen_any(f.y);
  return fma(x, x, fma(y, y, s));
}

}  // namespace bpm

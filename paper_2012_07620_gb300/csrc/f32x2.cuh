// Packed FP32 arithmetic (two floats in a 64-bit register): one instruction,
// the same IEEE results as two scalar ones.
#pragma once

#include <stdint.h>

namespace rr {

using f32x2 = unsigned long long;

__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// a - b: the product by -1 is exact, so the rounding is the subtraction's.
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  constexpr f32x2 minus_one = 0xbf800000bf800000ull;
  return fma2(b, minus_one, a);
}
__device__ __forceinline__ f32x2 twice(float a) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ float lo_of(f32x2 v) { return __uint_as_float(uint32_t(v)); }
__device__ __forceinline__ float hi_of(f32x2 v) { return __uint_as_float(uint32_t(v >> 32)); }

}  // namespace rr

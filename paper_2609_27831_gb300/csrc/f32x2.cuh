// Packed fp32 arithmetic on exact integers.
#pragma once

#include <cstdint>

namespace oz2 {

// Two fp32 values in a register pair; a packed instruction rounds each as the
// scalar one does.
struct F32x2 { uint64_t v; };
__device__ __forceinline__ F32x2 f2_pack(float lo, float hi) {
  F32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ F32x2 f2_pack(uint32_t lo, uint32_t hi) {   // bits
  F32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "r"(lo), "r"(hi));
  return r;
}
__device__ __forceinline__ void f2_unpack(F32x2 x, uint32_t& lo, uint32_t& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(x.v));
}
// the bf16 pair of two values exact in bf16
__device__ __forceinline__ uint32_t f2_bf16(F32x2 x) {
  uint32_t lo, hi;
  f2_unpack(x, lo, hi);
  return __byte_perm(lo, hi, 0x7632);
}
__device__ __forceinline__ F32x2 f2_fma(F32x2 a, F32x2 b, F32x2 c) {
  F32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ F32x2 f2_add(F32x2 a, F32x2 b) {
  F32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
// x y rounded to the nearest integer (|x y| < 2^22)
__device__ __forceinline__ F32x2 f2_nearest(F32x2 x, F32x2 y) {
  return f2_add(f2_fma(x, y, f2_pack(12582912.0f, 12582912.0f)), f2_pack(-12582912.0f, -12582912.0f));
}

}  // namespace oz2

// Pairs: two float32 lanes in one 64-bit register, for the packed add / mul / fma instructions of sm_100
// (each handles two elements per issue slot; IEEE round-to-nearest, same results as the scalar forms).  One thing differs: add2 of a mul2
// may be compiled into a single fused operation, which rounds once, so neither may be relied on to round by itself there.
#pragma once
#include <cstdint>

namespace repq {

typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ f32x2 splat2(float v) { return pack2(v, v); }
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
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
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// Two consecutive codes (even index first) pushed into the low byte / low half of a word that already holds the
// codes after them, with saturation to [0, 15] / [0, 255] (cvt.pack.sat: d = c << 8 | sat(e1) << 4 | sat(e0), c << 16 | sat(e1) << 8 | sat(e0)).
__device__ __forceinline__ uint32_t push_pair_u4(int e0, int e1, uint32_t c) {
  uint32_t d;
  asm("cvt.pack.sat.u4.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(e1), "r"(e0), "r"(c));
  return d;
}
__device__ __forceinline__ uint32_t push_pair_u8(int e0, int e1, uint32_t c) {
  uint32_t d;
  asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(e1), "r"(e0), "r"(c));
  return d;
}

}  // namespace repq

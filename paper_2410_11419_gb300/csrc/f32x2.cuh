// Two FP32 values in a 64-bit register and the packed FP32 instructions of
// sm_100 and later on them (add / mul / fma .rn.f32x2: each half rounds as
// the scalar instruction does).  One packed instruction occupies an issue slot
// and two cycles of the FMA pipe; a scalar FFMA or FADD with distinct operands
// also takes nearly two (measured: power and sum of one pixel, 4 operations,
// 6.9 cycles of an SM sub-partition scalar, 5.8 per pixel packed), so the
// composites, which are bound by issue slots and the FMA pipe, run on pairs
// of pixels.  Predicated scalar updates lose to an unconditional ex2 and a
// select on the power test: a receiver's pixel takes 12.9 cycles predicated
// and 9.5 packed, an occluder's 22.6 and 10.1.
#pragma once
#include <stdint.h>

namespace gs3 {
namespace {

using f32x2 = unsigned long long;

__device__ __forceinline__ f32x2 pk2(float lo, float hi) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ f32x2 dup2(float x) { return pk2(x, x); }
__device__ __forceinline__ void unpk2(f32x2 d, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(d));
}
__device__ __forceinline__ float lo2(f32x2 d) { return __uint_as_float((uint32_t)d); }
__device__ __forceinline__ float hi2(f32x2 d) { return __uint_as_float((uint32_t)(d >> 32)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

}  // namespace
}  // namespace gs3

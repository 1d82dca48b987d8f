// Packed float32 pairs (sm_100+): one instruction works on two float32 values held in a
// 64-bit register pair.  On GB300 the packed multiply-add has the FLOP rate of two scalar
// ones (80.2 against 78.3 TFLOP/s measured on independent chains) in half the issue slots,
// so a kernel that shares the issue port with loads, integer work and shuffles gains.
#pragma once

#include <cuda_runtime.h>

namespace mrstat {
namespace pk {

using f2 = unsigned long long;

__device__ __forceinline__ f2 make(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ f2 both(float v) { return make(v, v); }
__device__ __forceinline__ float2 split(f2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f2 fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

}  // namespace pk
}  // namespace mrstat

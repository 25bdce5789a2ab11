// Two FP32 multiply-adds per instruction (fma.rn.f32x2), each rounded like fmaf.
// The FP32 pipes give about the same rate either way (71 TFLOP/s with single
// multiply-adds, 75 with pairs); a pair takes half the issue slots, which leaves
// room for the shared-memory loads around it.
#pragma once

typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 pack2f(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2f(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
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

// Packed FP32 arithmetic (two values per 64-bit register pair): one instruction rounds both
// halves as the scalar one would, so the results are the scalar code's bits at half the issue
// slots.  For kernels bound by instruction issue whose lanes own two neighbouring features.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace dq {
namespace {

typedef unsigned long long f2;  // {low word: first value, high word: second value}

__device__ __forceinline__ f2 f2_pack(float x, float y) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ f2 f2_dup(float x) { return f2_pack(x, x); }
__device__ __forceinline__ float2 f2_unpack(f2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// a - b (the fused form of a + (-1) b rounds once, like the subtraction)
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) { return f2_fma(b, f2_dup(-1.f), a); }

}  // namespace
}  // namespace dq

// Packed FP32 arithmetic (sm_100 and later): two values per 64-bit register pair, one
// instruction for both, each rounded as the scalar operation.  The FMA pipe takes as
// long as for two scalar instructions; what is saved is issue slots.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace kmv {

__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack_f32x2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t mul_f32x2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// a - b (one rounding: b times -1 is exact).
__device__ __forceinline__ uint64_t sub_f32x2(uint64_t a, uint64_t b) {
  return fma_f32x2(b, pack_f32x2(-1.f, -1.f), a);
}


__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float lo_f32x2(uint64_t v) {
  float a, b;
  unpack_f32x2(v, a, b);
  return a;
}
__device__ __forceinline__ float hi_f32x2(uint64_t v) {
  float a, b;
  unpack_f32x2(v, a, b);
  return b;
}

}  // namespace kmv

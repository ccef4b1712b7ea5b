// Device helpers shared by the plain-FP32 (SIMT) kernels.
#pragma once

#include "kmv_internal.cuh"

namespace kmv {

// Rows of X / V / G staged in shared memory per step of the column loop.
constexpr int kJT = 64;

__device__ __forceinline__ float ex2_approx(float v) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}

// sc[k] = sqrt(h) / l_k for the system's lengthscales (h = log2(e)/2), so that
// K0_ij = 2^(-sum_k (sc_k x_ik - sc_k x_jk)^2) = exp(-sum_k (x_ik - x_jk)^2 / (2 l_k^2)).
__device__ __forceinline__ void load_scale(const double* th, int d, int ard, float* sc) {
  for (int k = threadIdx.x; k < d; k += blockDim.x)
    sc[k] = (float)(sqrt(kHalfLog2e) * exp(-th[1 + (ard ? k : 0)]));
}

// Deterministic block sum of one double per thread; result valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += red[i];
  return t;
}

// Running sum as an unevaluated pair s + c: each addition's rounding error,
// recovered exactly by Knuth's TwoSum, is added to c, so (double)s + (double)c
// differs from the exact sum of the terms by about u^2 times the sum of their
// magnitudes (u = 2^-24) instead of u times it.
__device__ __forceinline__ void two_sum_add(float& s, float& c, float x) {
  const float t = __fadd_rn(s, x);
  const float bp = __fsub_rn(t, s);
  const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(x, bp));
  c = __fadd_rn(c, err);
  s = t;
}

// Adds u v to the pair (s, e): the product's rounding error is recovered by an FMA.
__device__ __forceinline__ void pair_add_product(float& s, float& e, float u, float v) {
  const float p = __fmul_rn(u, v);
  two_sum_add(s, e, p);
  e = __fadd_rn(e, __fmaf_rn(u, v, -p));
}
// Sum of the warp's pairs, in every lane.
__device__ __forceinline__ void pair_warp_sum(float& s, float& e) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float so = __shfl_xor_sync(0xffffffffu, s, o), eo = __shfl_xor_sync(0xffffffffu, e, o);
    two_sum_add(s, e, so);
    e = __fadd_rn(e, eo);
  }
}

inline int pow2ceil(int v) {
  int p = 1;
  while (p < v) p <<= 1;
  return p;
}

}  // namespace kmv

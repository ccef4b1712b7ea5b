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

// Adds u v to the pair (s, e): the product's rounding error is recovered by an FMA.  FP32's
// range holds for the product, and for its error (2^-24 of it): for sums of which only
// FP32 accuracy near the size of u and v is needed (the preconditioner's projections),
// not for the r.r, r.z and p.q of a solver, whose squares leave FP32's range where the
// vectors are still well inside it.
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

// block_sum of N values at once, each in block_sum's order: the shuffles of the values
// interleave, where N calls would wait for N chains of dependent FP64 adds (some 900
// clocks each).  red: blockDim / 32 rows of N; out(v, sum) is called by thread v < n.
template <int N, class Out>
__device__ __forceinline__ void block_sum_many(double (&v)[N], int n, double* red, Out&& out) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) {
#pragma unroll
    for (int k = 0; k < N; ++k) red[w * N + k] = v[k];
  }
  __syncthreads();
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    double t = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += red[i * N + k];
    out(k, t);
  }
}

// Sums NC (16 or 32) pairs per lane over the warp: the lanes halve the vector between
// them step by step; lane l returns with column l % NC in (s[0], e[0]).
template <int NC>
__device__ __forceinline__ void pair_reduce_scatter(float (&s)[NC], float (&e)[NC]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int h = NC / 2; h >= 1; h /= 2) {
    const bool up = lane & h;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const float so = __shfl_xor_sync(0xffffffffu, up ? s[i] : s[i + h], h);
      const float eo = __shfl_xor_sync(0xffffffffu, up ? e[i] : e[i + h], h);
      float sk = up ? s[i + h] : s[i], ek = up ? e[i + h] : e[i];
      two_sum_add(sk, ek, so);
      s[i] = sk;
      e[i] = __fadd_rn(ek, eo);
    }
  }
  if (NC == 16) {
    const float so = __shfl_xor_sync(0xffffffffu, s[0], 16), eo = __shfl_xor_sync(0xffffffffu, e[0], 16);
    two_sum_add(s[0], e[0], so);
    e[0] = __fadd_rn(e[0], eo);
  }
}
// Block sums of NC (16 or 32) values per thread (kTile threads): out(col, sum) by thread
// col < n.  The lanes halve the vector between them step by step, NC - 1 adds a lane
// where a tree per value takes 5 NC (the FP64 pipe gives 2 lanes per clock and SM).
// red: kTile / 32 rows of NC.
template <int NC, class Out>
__device__ __forceinline__ void block_sums(double (&v)[NC], int n, double* red, Out&& out) {
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
  for (int h = NC / 2; h >= 1; h /= 2) {
    const bool up = l & h;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double other = __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + h], h);
      v[i] = (up ? v[i + h] : v[i]) + other;
    }
  }
  if (NC == 16) v[0] += __shfl_xor_sync(0xffffffffu, v[0], 16);
  __syncthreads();
  if (l < NC) red[w * NC + l] = v[0];
  __syncthreads();
  if ((int)threadIdx.x < n) {
    double t = 0.0;
#pragma unroll
    for (int i = 0; i < kTile / 32; ++i) t += red[i * NC + threadIdx.x];
    out((int)threadIdx.x, t);
  }
}

inline int pow2ceil(int v) {
  int p = 1;
  while (p < v) p <<= 1;
  return p;
}

}  // namespace kmv

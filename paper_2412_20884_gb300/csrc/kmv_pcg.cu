// Preconditioned CG (the textbook recurrences with z = P^{-1} r) for the
// batched single right-hand-side solves, with the randomized Nystrom
// preconditioner of kmv_nystrom.cu applied as
//   z = r + U (d o (U^T r)),   d_k = (lambda_r + mu) / (lambda_k + mu) - 1,
// mu = sigma_s^2 of the system's current theta (the Woodbury form for
// A = K + sigma^2 I; the factorisation may come from an earlier theta).
// Per iteration: q = A p (with p.q fused in the product), alpha, x and r,
// U^T r per tile, the per-system coefficients, z and r.z, beta, p.  FP64
// scalars from per-tile partials summed in a fixed order.
#include <algorithm>

#include "cg_common.cuh"
#include "kmv_internal.cuh"
#include "simt_common.cuh"

namespace kmv {
namespace {

// Sum of a system's per-tile partials by one warp (every lane gets it).
__device__ __forceinline__ double tile_sum(const DevLayout& L, int b, int c, int chains, const double* partial,
                                           int stride, int k) {
  double acc = 0.0;
  for (int it = L.inst_item0[b] + (int)(threadIdx.x & 31); it < L.inst_item0[b + 1]; it += 32)
    acc += partial[((int64_t)it * chains + c) * stride + k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return acc;
}
constexpr int kSysWarps = 4;   // systems (one warp each) per CTA of the per-system kernels

// r = rhs - q (warm) or rhs (cold, x = 0); partials of r.r and rhs.rhs
__global__ void pcg_init_kernel(DevLayout L, int chains, int64_t n_total, const float* rhs, int64_t rhs_stride,
                                const float* q, float* x, float* r, int warm, double* partial2) {
  __shared__ double red[kTile / 32];
  const int item = blockIdx.x, c = blockIdx.y;
  const int b = L.item_inst[item];
  const int64_t i = L.item_row0[item] + threadIdx.x;
  double rr = 0.0, bb = 0.0;
  if (i < L.offsets[b + 1]) {
    const int64_t v = (int64_t)c * n_total + i;
    const float bv = rhs[(int64_t)c * rhs_stride + i];
    float rv = bv;
    if (warm) rv = bv - q[v];
    else x[v] = 0.f;
    r[v] = rv;
    rr = (double)rv * rv;
    bb = (double)bv * bv;
  }
  const double t0 = block_sum(rr, red);
  const double t1 = block_sum(bb, red);
  if (threadIdx.x == 0) {
    partial2[((int64_t)item * chains + c) * 2] = t0;
    partial2[((int64_t)item * chains + c) * 2 + 1] = t1;
  }
}

__global__ void pcg_factors_kernel(int n_sys, int rank, int n_theta, const double* theta, const double* lam, double* d) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= (int64_t)n_sys * rank) return;
  const int s = (int)(e / rank), k = (int)(e - (int64_t)s * rank);
  const double mu = exp(theta[(int64_t)s * n_theta + n_theta - 1]);
  const double lr = lam[(int64_t)s * rank + rank - 1];
  d[e] = (lr + mu) / (lam[(int64_t)s * rank + k] + mu) - 1.0;
}

// partial[tile, c, k] = sum over the tile's rows of U[c, k, i] r_i, one warp per k, of
// the r in shared memory (rs).  The products are split exactly (p = u r, its error by an
// FMA) and summed as (sum, error) pairs: the FP64 pipe runs at 2 lanes per clock and SM,
// and FP64 products took 28 us per application at N = 8192, 8 chains, rank 64.
__device__ __forceinline__ void pcg_project(const float* rs, int64_t r0, int64_t r1, const float* U, int64_t n_total,
                                            int rank, double* partial) {
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  float rv[kTile / 32];
#pragma unroll
  for (int u = 0; u < kTile / 32; ++u) rv[u] = rs[l + 32 * u];
#pragma unroll 2
  for (int k = w; k < rank; k += kTile / 32) {
    const float* Uk = U + (int64_t)k * n_total + r0 + l;
    float uk[kTile / 32];
#pragma unroll
    for (int u = 0; u < kTile / 32; ++u) uk[u] = r0 + l + 32 * u < r1 ? Uk[32 * u] : 0.f;
    float s = 0.f, e = 0.f;
#pragma unroll
    for (int u = 0; u < kTile / 32; ++u) pair_add_product(s, e, uk[u], rv[u]);
    pair_warp_sum(s, e);
    if (l == 0) partial[k] = (double)s + (double)e;
  }
}

// x += alpha p, r -= alpha q and the partials of r.r (UPDATE), then the projections of
// the tile's r.
template <bool UPDATE>
__global__ void pcg_proj_kernel(DevLayout L, int chains, int64_t n_total, int rank, const float* U, const PcgSys* sys,
                                const int32_t* active, float* x, float* r, const float* p, const float* q,
                                double* partial, double* proj) {
  __shared__ double red[kTile / 32];
  __shared__ float rs[kTile];
  chain_trigger();
  const int item = blockIdx.x, c = blockIdx.y;
  const int b = L.item_inst[item];
  const int s = b * chains + c;
  const int64_t r0 = L.item_row0[item], r1 = L.offsets[b + 1];
  chain_wait();
  if (active && !active[s]) return;
  const int64_t i = r0 + threadIdx.x, v = (int64_t)c * n_total + i;
  float rv = i < r1 ? r[v] : 0.f;
  if (UPDATE && i < r1) {
    const float al = (float)sys[s].alpha;
    x[v] = fmaf(al, p[v], x[v]);
    rv = fmaf(-al, q[v], rv);
    r[v] = rv;
  }
  rs[threadIdx.x] = rv;
  if (UPDATE) {
    const double t = block_sum((double)rv * rv, red);
    if (threadIdx.x == 0) partial[(int64_t)item * chains + c] = t;
  } else {
    __syncthreads();
  }
  pcg_project(rs, r0, r1, U + (int64_t)c * rank * n_total, n_total, rank,
              proj + ((int64_t)item * chains + c) * rank);
}

// coef[s, k] = d[s, k] * sum over the instance's tiles of partial[., k]: 32 columns k
// and 8 shares of the tiles per CTA.
constexpr int kCoefShares = 8;
__global__ void __launch_bounds__(32 * kCoefShares) pcg_coef_kernel(DevLayout L, int chains, int rank, const double* d,
                                                                    const double* partial, const int32_t* active,
                                                                    double* coef) {
  __shared__ double red[kCoefShares][32];
  chain_trigger();
  const int s = blockIdx.x, lane = threadIdx.x & 31, y = threadIdx.x >> 5, k = blockIdx.y * 32 + lane;
  const int b = s / chains, c = s - b * chains;
  const int i0 = L.inst_item0[b], i1 = L.inst_item0[b + 1];
  chain_wait();
  if (active && !active[s]) return;
  double acc = 0.0;
  if (k < rank) {
#pragma unroll 4
    for (int it = i0 + y; it < i1; it += kCoefShares) acc += partial[((int64_t)it * chains + c) * rank + k];
  }
  red[y][lane] = acc;
  __syncthreads();
  if (y != 0 || k >= rank) return;
#pragma unroll
  for (int u = 1; u < kCoefShares; ++u) acc += red[u][lane];
  coef[(int64_t)s * rank + k] = d[(int64_t)s * rank + k] * acc;
}

// z = r + U coef; partials of r.z.  Inside an iteration (sys set) the CTA of each
// system that finishes last takes its beta and stopping test and, for a system of at
// most p_rows rows, forms p = z + beta p.
__global__ void pcg_apply_kernel(DevLayout L, int chains, int64_t n_total, int rank, const float* U,
                                 const double* coef, const float* r, float* z, int32_t* active, double* prz,
                                 PcgSys* sys, const double* prr, uint32_t* count, int32_t* n_active, double tol,
                                 int maxiter, int p_rows, float* p) {
  __shared__ double red[kTile / 32];
  __shared__ float cf[kMaxRank];
  __shared__ int s_last;
  __shared__ float s_beta;
  chain_trigger();
  const int item = blockIdx.x, c = blockIdx.y;
  const int b = L.item_inst[item];
  const int s = b * chains + c;
  const int64_t r1 = L.offsets[b + 1], i = L.item_row0[item] + threadIdx.x;
  const int n_of_system = L.inst_item0[b + 1] - L.inst_item0[b];
  chain_wait();
  if (active && !active[s]) return;
  for (int k = threadIdx.x; k < rank; k += blockDim.x) cf[k] = (float)coef[(int64_t)s * rank + k];
  __syncthreads();
  double rz = 0.0;
  if (i < r1) {
    const int64_t v = (int64_t)c * n_total + i;
    const float rv = r[v];
    const float* Ui = U + (int64_t)c * rank * n_total + i;
    float acc = 0.f;
#pragma unroll 8
    for (int k = 0; k < rank; ++k) acc = fmaf(Ui[(int64_t)k * n_total], cf[k], acc);
    const float zv = rv + acc;
    z[v] = zv;
    rz = (double)rv * zv;
  }
  const double t = block_sum(rz, red);
  if (threadIdx.x == 0) {
    prz[(int64_t)item * chains + c] = t;
    s_last = sys && last_arrival(&count[s], 1u, (uint32_t)n_of_system);
  }
  if (!sys) return;
  __syncthreads();
  if (!s_last) return;
  const double rr_new = sys_sum_block(L, b, c, chains, prr, 1, 0, red);
  __syncthreads();
  const double rz_new = sys_sum_block(L, b, c, chains, prz, 1, 0, red);
  if (threadIdx.x == 0) {
    const bool go = pcg_rz_step(sys[s], rr_new, rz_new, tol, maxiter);
    if (!go) {
      active[s] = 0;
      atomicSub(n_active, 1);
    }
    s_last = go;
    s_beta = (float)sys[s].beta;
  }
  const int64_t rows0 = L.offsets[b];
  if (p_rows == 0 || r1 - rows0 > p_rows) return;
  __syncthreads();
  if (s_last) form_direction(p, z, s_beta, (int64_t)c * n_total + rows0, (int64_t)c * n_total + r1);
}

// rr, bb, rz of every system; active while rr > tol^2 bb; beta = 0 (p = z)
__global__ void pcg_setup_kernel(DevLayout L, int n_inst, int chains, const double* partial2, const double* prz,
                                 double tol, PcgSys* sys, int32_t* active, int32_t* n_active) {
  const int s = blockIdx.x * kSysWarps + (threadIdx.x >> 5);
  if (s >= n_inst * chains) return;
  const int b = s / chains, c = s - b * chains;
  const double rr = tile_sum(L, b, c, chains, partial2, 2, 0), bb = tile_sum(L, b, c, chains, partial2, 2, 1);
  const double rz = tile_sum(L, b, c, chains, prz, 1, 0);
  if ((threadIdx.x & 31) != 0) return;
  PcgSys& y = sys[s];
  y.rr = rr;
  y.bb = bb;
  y.rz = rz;
  y.alpha = y.beta = 0.0;
  y.iters = 0;
  y.status = isfinite(y.rr) ? KMV_OK : KMV_ENONFINITE;
  const int act = (y.status == KMV_OK && y.bb > 0.0 && y.rr > tol * tol * y.bb) ? 1 : 0;
  active[s] = act;
  if (act) atomicAdd(n_active, 1);
}

__global__ void pcg_alpha_kernel(DevLayout L, int n_inst, int chains, const double* partial, PcgSys* sys,
                                 int32_t* active, int32_t* n_active) {
  const int s = blockIdx.x * kSysWarps + (threadIdx.x >> 5);
  if (s >= n_inst * chains || !active[s]) return;
  const int b = s / chains, c = s - b * chains;
  const double pq = tile_sum(L, b, c, chains, partial, 1, 0);
  if ((threadIdx.x & 31) == 0 && !pcg_pq_step(sys[s], pq)) {
    active[s] = 0;
    atomicSub(n_active, 1);
  }
}

// p = z + beta p
__global__ void pcg_update_p_kernel(DevLayout L, int chains, int64_t n_total, const PcgSys* sys,
                                    const int32_t* active, const float* z, float* p) {
  chain_trigger();
  chain_wait();
  const int item = blockIdx.x, c = blockIdx.y;
  const int b = L.item_inst[item];
  const int s = b * chains + c;
  if (!active[s]) return;
  const int64_t i = L.item_row0[item] + threadIdx.x;
  if (i >= L.offsets[b + 1]) return;
  const int64_t v = (int64_t)c * n_total + i;
  p[v] = fmaf((float)sys[s].beta, p[v], z[v]);
}

__global__ void pcg_finish_kernel(int n_sys, const PcgSys* sys, const int32_t* active, int32_t* status,
                                  int32_t* iters) {
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n_sys; s += gridDim.x * blockDim.x) {
    status[s] = sys[s].status != KMV_OK ? sys[s].status : (active[s] ? KMV_ENOTCONV : KMV_OK);
    if (iters) iters[s] = sys[s].iters;
  }
}

}  // namespace

cudaError_t launch_pcg_init(const DevLayout& L, int n_items, int chains, int64_t n_total, const float* rhs,
                            int64_t rhs_stride, const float* q, float* x, float* r, int warm, double* partial2,
                            cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  pcg_init_kernel<<<dim3(n_items, chains), kTile, 0, st>>>(L, chains, n_total, rhs, rhs_stride, q, x, r, warm,
                                                           partial2);
  return cudaGetLastError();
}

cudaError_t launch_pcg_factors(const PcgPrecond& P, int n_sys, int n_theta, const double* theta, double* d,
                               cudaStream_t st) {
  const int64_t n = (int64_t)n_sys * P.rank;
  pcg_factors_kernel<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(n_sys, P.rank, n_theta, theta, P.lam, d);
  return cudaGetLastError();
}

cudaError_t launch_pcg_precond(const DevLayout& L, int n_items, int n_inst, int chains, int64_t n_total,
                               const PcgPrecond& P, const double* d, const float* r, float* z, const int32_t* active,
                               double* proj, double* coef, double* prz, bool chained, cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  const dim3 grid(n_items, chains);
  cudaError_t e = launch_chained(chained, pcg_proj_kernel<false>, grid, kTile, 0, st, L, chains, n_total, P.rank, P.U,
                                 nullptr, active, nullptr, const_cast<float*>(r), nullptr, nullptr, nullptr, proj);
  if (e == cudaSuccess)
    e = launch_chained(chained, pcg_coef_kernel, dim3(n_inst * chains, (P.rank + 31) / 32), 32 * kCoefShares, 0, st, L,
                       chains, P.rank, d, proj, active, coef);
  if (e == cudaSuccess)
    e = launch_chained(chained, pcg_apply_kernel, grid, kTile, 0, st, L, chains, n_total, P.rank, P.U, coef, r, z,
                       const_cast<int32_t*>(active), prz, nullptr, nullptr, nullptr, nullptr, 0.0, 0, 0, nullptr);
  return e;
}

cudaError_t launch_pcg_iterate(const DevLayout& L, int n_items, int n_inst, int chains, int64_t n_total,
                               const PcgPrecond& P, const double* d, PcgSys* sys, int32_t* active, int32_t* n_active,
                               float* x, float* r, float* p, const float* q, float* z, double* partial, double* proj,
                               double* coef, double* prz, uint32_t* count, double tol, int maxiter, int p_rows,
                               bool chained, cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  const dim3 grid(n_items, chains);
  cudaError_t e = launch_chained(chained, pcg_proj_kernel<true>, grid, kTile, 0, st, L, chains, n_total, P.rank, P.U,
                                 sys, active, x, r, p, q, partial, proj);
  if (e == cudaSuccess)
    e = launch_chained(chained, pcg_coef_kernel, dim3(n_inst * chains, (P.rank + 31) / 32), 32 * kCoefShares, 0, st, L,
                       chains, P.rank, d, proj, active, coef);
  if (e == cudaSuccess)
    e = launch_chained(chained, pcg_apply_kernel, grid, kTile, 0, st, L, chains, n_total, P.rank, P.U, coef, r, z,
                       active, prz, sys, partial, count, n_active, tol, maxiter, p_rows, p);
  return e;
}

cudaError_t launch_pcg_setup(const DevLayout& L, int n_inst, int chains, const double* partial2, const double* prz,
                             double tol, PcgSys* sys, int32_t* active, int32_t* n_active, cudaStream_t st) {
  const int n = n_inst * chains;
  pcg_setup_kernel<<<(n + kSysWarps - 1) / kSysWarps, 32 * kSysWarps, 0, st>>>(L, n_inst, chains, partial2, prz, tol,
                                                                              sys, active, n_active);
  return cudaGetLastError();
}

cudaError_t launch_pcg_alpha(const DevLayout& L, int n_inst, int chains, const double* partial, PcgSys* sys,
                             int32_t* active, int32_t* n_active, cudaStream_t st) {
  const int n = n_inst * chains;
  pcg_alpha_kernel<<<(n + kSysWarps - 1) / kSysWarps, 32 * kSysWarps, 0, st>>>(L, n_inst, chains, partial, sys, active,
                                                                              n_active);
  return cudaGetLastError();
}

cudaError_t launch_pcg_update_p(const DevLayout& L, int n_items, int chains, int64_t n_total, const PcgSys* sys,
                                const int32_t* active, const float* z, float* p, bool chained, cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  return launch_chained(chained, pcg_update_p_kernel, dim3(n_items, chains), kTile, 0, st, L, chains, n_total, sys,
                        active, z, p);
}

cudaError_t launch_pcg_finish(int n_sys, const PcgSys* sys, const int32_t* active, int32_t* status, int32_t* iters,
                              cudaStream_t st) {
  if (n_sys == 0) return cudaSuccess;
  pcg_finish_kernel<<<(n_sys + 255) / 256, 256, 0, st>>>(n_sys, sys, active, status, iters);
  return cudaGetLastError();
}

}  // namespace kmv

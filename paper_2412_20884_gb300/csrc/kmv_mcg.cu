// Conjugate gradients on several shifted systems per (instance, chain) at once:
// (A_s + shift_{s,q} I) x_q = b_q for the m columns q of every system s, one
// m-column product per iteration (the shifted systems of the pole expansion of
// App. A, Sec. 3.1).  Each column runs its own CG (its own alpha, beta and
// stopping test); a system whose columns have all stopped drops out of the
// product.  FP64 scalars, per-(tile, chain, column) partial sums reduced in a
// fixed order, so the iterates are bitwise reproducible.
//
// The columns' dot products are FP64 throughout (a solve is to give the same iterates
// for any scale of its right-hand side, and FP32 squares of a residual below 1e-19 are
// subnormal), all columns of a row tile in one reduce-scatter; the per-column scalar
// steps run in the CTA that finishes a system last, a warp per column.  (A block sum per
// column and one thread per system took 63 + 91 us per iteration for 8 systems of 64
// tiles and 15 columns.)
#include <algorithm>

#include "cg_common.cuh"
#include "kmv_internal.cuh"
#include "simt_common.cuh"

namespace kmv {
namespace {

// Sum of a system's per-tile partials of one column by one warp (every lane gets it).
__device__ __forceinline__ double col_sum(const DevLayout& L, int b, int c, int chains, int m, int col,
                                          const double* partial, int stride = 1, int k = 0) {
  double acc = 0.0;
  for (int it = L.inst_item0[b] + (int)(threadIdx.x & 31); it < L.inst_item0[b + 1]; it += 32)
    acc += __ldcg(&partial[(((int64_t)it * chains + c) * m + col) * stride + k]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return acc;
}

// x = 0 (cold) or kept (warm, with q = A x given); r = b - q; p = r; partials of r.r and b.b.
// b is (chains, N) shared by the m columns when b_cols == 0, else (chains, N, m).
__global__ void mcg_init_kernel(DevLayout L, int chains, int64_t n_total, int m, const float* b, int b_cols,
                                const float* q, int warm, float* x, float* r, float* p, double* partial2) {
  __shared__ double red[kTile / 32];
  const int item = blockIdx.x, c = blockIdx.y;
  const int bi = L.item_inst[item];
  const int64_t i = L.item_row0[item] + threadIdx.x;
  const bool valid = i < L.offsets[bi + 1];
  for (int col = 0; col < m; ++col) {
    double rr = 0.0, bb = 0.0;
    if (valid) {
      const int64_t v = ((int64_t)c * n_total + i) * m + col;
      const float bv = b_cols ? b[v] : b[(int64_t)c * n_total + i];
      float rv = bv;
      if (warm) rv = bv - q[v];
      else x[v] = 0.f;
      r[v] = rv;
      p[v] = rv;
      rr = (double)rv * rv;
      bb = (double)bv * bv;
    }
    const int64_t o = (((int64_t)item * chains + c) * m + col) * 2;
    double t = block_sum(rr, red);
    if (threadIdx.x == 0) partial2[o] = t;
    t = block_sum(bb, red);
    if (threadIdx.x == 0) partial2[o + 1] = t;
  }
}

// Per (system, column), a warp each: the sums of the tiles' partials; a column is
// active while r.r > tol^2 b.b.  sys_any[s] = the number of active columns of s.
constexpr int kColWarps = 4;
__global__ void mcg_reduce_init_kernel(DevLayout L, int n_inst, int chains, int m, const double* partial2,
                                       double tol, McgCol* st, int32_t* sys_any, int32_t* n_active) {
  const int64_t e = (int64_t)blockIdx.x * kColWarps + (threadIdx.x >> 5);
  if (e >= (int64_t)n_inst * chains * m) return;
  const int s = (int)(e / m), col = (int)(e - (int64_t)s * m);
  const int bi = s / chains, c = s - bi * chains;
  const double rr = col_sum(L, bi, c, chains, m, col, partial2, 2, 0);
  const double bb = col_sum(L, bi, c, chains, m, col, partial2, 2, 1);
  if ((threadIdx.x & 31) != 0) return;
  McgCol& k = st[e];
  k.rr = rr;
  k.bb = bb;
  k.alpha = k.beta = 0.0;
  k.iters = 0;
  k.status = KMV_OK;
  k.pad = 0;
  k.active = (bb > 0.0 && rr > tol * tol * bb) ? 1 : 0;
  if (!isfinite(rr)) {
    k.active = 0;
    k.status = KMV_ENONFINITE;
  }
  if (k.active) {
    atomicAdd(&sys_any[s], 1);
    atomicAdd(n_active, 1);
  }
}

// alpha = r.r / p.q (r.z / p.q when preconditioned) of one active column; a
// non-positive p.q is a breakdown.
__device__ __forceinline__ bool mcg_alpha_step(McgCol& k, double pq, int pre) {
  const double num = pre ? k.rz : k.rr;
  if (!(pq > 0.0) || !isfinite(pq) || !(num > 0.0)) {
    k.alpha = 0.0;
    k.active = 0;
    k.status = (isfinite(pq) && isfinite(num)) ? KMV_ENOTCONV : KMV_ENONFINITE;
    return false;
  }
  k.alpha = num / pq;
  return true;
}

// beta = r.r_new / r.r (r.z_new / r.z when preconditioned) of one active column and its
// stopping test: converged (r.r <= tol^2 b.b) or at maxiter.
__device__ __forceinline__ bool mcg_beta_step(McgCol& k, double rr, double rz, int pre, double tol, int maxiter) {
  if (pre) {
    k.beta = rz / k.rz;
    k.rz = rz;
  } else {
    k.beta = rr / k.rr;
  }
  k.rr = rr;
  k.iters += 1;
  if (!isfinite(rr)) {
    k.active = 0;
    k.status = KMV_ENONFINITE;
  } else if (rr <= tol * tol * k.bb) {
    k.active = 0;
  } else if (k.iters >= maxiter) {
    k.active = 0;
    k.status = KMV_ENOTCONV;
  }
  return k.active != 0;
}

// One column left the solve (a warp's lane 0).
__device__ __forceinline__ void mcg_drop(int32_t* sys_any, int32_t* n_active, int s) {
  atomicSub(&sys_any[s], 1);
  atomicSub(n_active, 1);
}

// partials of p.q per column; the system's last CTA takes the columns' alpha steps
template <int NC>
__global__ void __launch_bounds__(kTile) mcg_dot_kernel(DevLayout L, int chains, int64_t n_total, int m, const float* p,
                                                        const float* q, int32_t* sys_any, double* partial,
                                                        uint32_t* count, McgCol* st, int pre, int32_t* n_active) {
  __shared__ double red[kTile / 32 * NC];
  __shared__ int s_last;
  chain_trigger();
  const int item = blockIdx.x, c = blockIdx.y;
  const int bi = L.item_inst[item];
  const int s = bi * chains + c;
  const int64_t i = L.item_row0[item] + threadIdx.x;
  const bool valid = i < L.offsets[bi + 1];
  chain_wait();
  if (!sys_any[s]) return;
  double v[NC];
#pragma unroll
  for (int col = 0; col < NC; ++col) {
    v[col] = 0.0;
    if (valid && col < m) {
      const int64_t o = ((int64_t)c * n_total + i) * m + col;
      v[col] = (double)p[o] * q[o];
    }
  }
  block_sums<NC>(v, m, red, [&](int col, double t) { partial[((int64_t)item * chains + c) * m + col] = t; });
  __syncthreads();
  if (threadIdx.x == 0) s_last = last_arrival(&count[s], 1u, (uint32_t)(L.inst_item0[bi + 1] - L.inst_item0[bi]));
  __syncthreads();
  if (!s_last) return;
  for (int col = threadIdx.x >> 5; col < m; col += kTile / 32) {
    McgCol& k = st[(int64_t)s * m + col];
    if (!k.active) {
      if ((threadIdx.x & 31) == 0) k.alpha = 0.0;
      continue;
    }
    const double pq = col_sum(L, bi, c, chains, m, col, partial);
    if ((threadIdx.x & 31) == 0 && !mcg_alpha_step(k, pq, pre)) mcg_drop(sys_any, n_active, s);
  }
}

// x += alpha p, r -= alpha q on the active columns; partials of the new r.r; without a
// preconditioner (count set) the system's last CTA takes the columns' beta steps
template <int NC>
__global__ void __launch_bounds__(kTile) mcg_update_xr_kernel(DevLayout L, int chains, int64_t n_total, int m,
                                                              McgCol* st, int32_t* sys_any, float* x, float* r,
                                                              const float* p, const float* q, double* partial,
                                                              uint32_t* count, double tol, int maxiter,
                                                              int32_t* n_active) {
  __shared__ double red[kTile / 32 * NC];
  __shared__ float al[NC];
  __shared__ int on[NC];
  __shared__ int s_last;
  chain_trigger();
  const int item = blockIdx.x, c = blockIdx.y;
  const int bi = L.item_inst[item];
  const int s = bi * chains + c;
  const int64_t i = L.item_row0[item] + threadIdx.x;
  const bool valid = i < L.offsets[bi + 1];
  chain_wait();
  if (!sys_any[s]) return;
  if ((int)threadIdx.x < m) {
    const McgCol& k = st[(int64_t)s * m + threadIdx.x];
    al[threadIdx.x] = (float)k.alpha;
    on[threadIdx.x] = k.active;
  }
  __syncthreads();
  double v[NC];
#pragma unroll
  for (int col = 0; col < NC; ++col) {
    v[col] = 0.0;
    if (valid && col < m) {
      const int64_t o = ((int64_t)c * n_total + i) * m + col;
      float rv = r[o];
      if (on[col]) {
        x[o] = fmaf(al[col], p[o], x[o]);
        rv = fmaf(-al[col], q[o], rv);
        r[o] = rv;
      }
      v[col] = (double)rv * rv;
    }
  }
  block_sums<NC>(v, m, red, [&](int col, double t) { partial[((int64_t)item * chains + c) * m + col] = t; });
  if (!count) return;
  __syncthreads();
  if (threadIdx.x == 0) s_last = last_arrival(&count[s], 1u, (uint32_t)(L.inst_item0[bi + 1] - L.inst_item0[bi]));
  __syncthreads();
  if (!s_last) return;
  for (int col = threadIdx.x >> 5; col < m; col += kTile / 32) {
    McgCol& k = st[(int64_t)s * m + col];
    if (!k.active) continue;
    const double rr = col_sum(L, bi, c, chains, m, col, partial);
    if ((threadIdx.x & 31) == 0 && !mcg_beta_step(k, rr, 0.0, 0, tol, maxiter)) mcg_drop(sys_any, n_active, s);
  }
}

// p = r + beta p on the active columns (r is z when preconditioned)
__global__ void mcg_update_p_kernel(DevLayout L, int chains, int64_t n_total, int m, const McgCol* st,
                                    const int32_t* sys_any, const float* r, float* p) {
  chain_trigger();
  chain_wait();
  const int item = blockIdx.x, c = blockIdx.y;
  const int bi = L.item_inst[item];
  const int s = bi * chains + c;
  if (!sys_any[s]) return;
  const int64_t i = L.item_row0[item] + threadIdx.x;
  if (i >= L.offsets[bi + 1]) return;
  for (int col = 0; col < m; ++col) {
    const McgCol& k = st[(int64_t)s * m + col];
    if (!k.active) continue;
    const int64_t o = ((int64_t)c * n_total + i) * m + col;
    p[o] = fmaf((float)k.beta, p[o], r[o]);
  }
}

// Column results of a finished solve: col_status = the column's status
// (KMV_ENOTCONV if still active), col_iters = its iterations.  With accumulate
// (an inner solve of the refinement) the iterations add up and only a
// non-finite inner solve marks the column.
__global__ void mcg_finish_kernel(int64_t n_cols, const McgCol* cols, int accumulate, int32_t* col_status,
                                  int32_t* col_iters) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n_cols; e += (int64_t)gridDim.x * blockDim.x) {
    const McgCol& k = cols[e];
    if (accumulate) {
      col_iters[e] += k.iters;
      if (k.status == KMV_ENONFINITE) col_status[e] = KMV_ENONFINITE;
    } else {
      col_status[e] = k.active ? KMV_ENOTCONV : k.status;
      col_iters[e] = k.iters;
    }
  }
}

// r[., ., q] = 0 for the columns the refinement no longer corrects.
__global__ void mcg_mask_kernel(DevLayout L, int chains, int64_t n_total, int m, const McgCol* cols, float* r) {
  const int item = blockIdx.x, c = blockIdx.y;
  const int bi = L.item_inst[item];
  const int s = bi * chains + c;
  const int64_t i = L.item_row0[item] + threadIdx.x;
  if (i >= L.offsets[bi + 1]) return;
  for (int col = 0; col < m; ++col)
    if (!cols[(int64_t)s * m + col].active) r[((int64_t)c * n_total + i) * m + col] = 0.f;
}

// Refinement step bookkeeping per column, as for the single-column refinement:
// a column whose true residual fell by less than half since the last step has
// reached the floor of the FP32 operator and stops; one whose residual rose is
// marked (pad = 1) for the last correction to be taken back.  n_active =
// columns left, worst = the largest rr / bb among them.  One block.
__global__ void mcg_refine_kernel(int64_t n_cols, int outer, McgCol* cols, double* prev_rr, int32_t* n_active,
                                  double* worst) {
  __shared__ int cnt[8];
  __shared__ double wmax[8];
  int v = 0;
  double wr = 0.0;
  for (int64_t e = threadIdx.x; e < n_cols; e += blockDim.x) {
    McgCol& k = cols[e];
    if (k.active && outer > 0 && k.rr > 0.25 * prev_rr[e]) {
      k.active = 0;
      if (k.rr > prev_rr[e]) {
        k.pad = 1;
        k.rr = prev_rr[e];
      }
    }
    prev_rr[e] = k.rr;
    v += k.active;
    if (k.active && k.bb > 0.0) wr = fmax(wr, k.rr / k.bb);
  }
  for (int o = 16; o > 0; o >>= 1) {
    v += __shfl_down_sync(0xffffffffu, v, o);
    wr = fmax(wr, __shfl_down_sync(0xffffffffu, wr, o));
  }
  if ((threadIdx.x & 31) == 0) {
    cnt[threadIdx.x >> 5] = v;
    wmax[threadIdx.x >> 5] = wr;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    double mx = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      t += cnt[w];
      mx = fmax(mx, wmax[w]);
    }
    *n_active = t;
    *worst = mx;
  }
}

// x[., ., q] -= dx[., ., q] for the columns whose last correction raised the residual.
__global__ void mcg_undo_kernel(DevLayout L, int chains, int64_t n_total, int m, const McgCol* cols,
                                const float* dx, float* x) {
  const int item = blockIdx.x, c = blockIdx.y;
  const int bi = L.item_inst[item];
  const int s = bi * chains + c;
  const int64_t i = L.item_row0[item] + threadIdx.x;
  if (i >= L.offsets[bi + 1]) return;
  for (int col = 0; col < m; ++col) {
    if (!cols[(int64_t)s * m + col].pad) continue;
    const int64_t o = ((int64_t)c * n_total + i) * m + col;
    x[o] -= dx[o];
  }
}

// Final refinement status: a column still active after the last step did not converge.
__global__ void mcg_refine_finish_kernel(int64_t n_cols, const McgCol* cols, int32_t* col_status) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n_cols; e += (int64_t)gridDim.x * blockDim.x) {
    if (col_status[e] != KMV_OK) continue;
    if (cols[e].status != KMV_OK) col_status[e] = cols[e].status;
    else if (cols[e].active) col_status[e] = KMV_ENOTCONV;
  }
}

// Multi-column projection: partial[tile, c, q, k] = sum over the tile's rows of
// U[c, k, i] r[c, i, q]; the tile's r columns are staged in shared memory and
// each U row segment is read once for all columns (a warp per k).
template <int NC>
__global__ void __launch_bounds__(kTile) mcg_proj_kernel(DevLayout L, int chains, int64_t n_total, int m, int rank,
                                                         const float* U, const float* r, const int32_t* sys_any,
                                                         double* partial) {
  __shared__ float rs[NC][kTile];
  chain_trigger();
  const int item = blockIdx.x, c = blockIdx.y;
  const int b = L.item_inst[item];
  const int64_t r0 = L.item_row0[item], r1 = L.offsets[b + 1];
  chain_wait();
  if (sys_any && !sys_any[b * chains + c]) return;
  for (int e = threadIdx.x; e < NC * kTile; e += blockDim.x) {
    const int row = e / NC, q = e - row * NC;
    const int64_t i = r0 + row;
    rs[q][row] = i < r1 && q < m ? r[((int64_t)c * n_total + i) * m + q] : 0.f;
  }
  __syncthreads();
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  for (int k = w; k < rank; k += kTile / 32) {
    const float* Uk = U + ((int64_t)c * rank + k) * n_total;
    float u[kTile / 32];
#pragma unroll
    for (int t = 0; t < kTile / 32; ++t) {
      const int64_t i = r0 + l + 32 * t;
      u[t] = i < r1 ? Uk[i] : 0.f;
    }
    float s[NC], e[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      s[q] = e[q] = 0.f;
#pragma unroll
      for (int t = 0; t < kTile / 32; ++t) pair_add_product(s[q], e[q], u[t], rs[q][l + 32 * t]);
    }
    pair_reduce_scatter<NC>(s, e);
    if (l < m) partial[(((int64_t)item * chains + c) * m + l) * rank + k] = (double)s[0] + (double)e[0];
  }
}

// d[s, q, k] = (lambda_r + mu_q) / (lambda_k + mu_q) - 1, mu_q = sigma_s^2 + shift[s, q]
__global__ void mcg_factors_kernel(int64_t n, int m, int rank, int n_theta, const double* theta, const float* shifts,
                                   const double* lam, double* d) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= n) return;
  const int k = (int)(e % rank);
  const int64_t sq = e / rank;
  const int q = (int)(sq % m), s = (int)(sq / m);
  const double mu = exp(theta[(int64_t)s * n_theta + n_theta - 1]) + (double)shifts[(int64_t)s * m + q];
  const double lr = lam[(int64_t)s * rank + rank - 1];
  d[e] = (lr + mu) / (lam[(int64_t)s * rank + k] + mu) - 1.0;
}

// coef[s, q, k] = d[s, q, k] * sum over the instance's tiles of partial[., q, k]: 32
// columns k and 8 shares of the tiles per CTA.
constexpr int kCoefShares = 8;
__global__ void __launch_bounds__(32 * kCoefShares) mcg_coef_kernel(DevLayout L, int chains, int m, int rank,
                                                                    const double* d, const double* partial,
                                                                    const int32_t* sys_any, double* coef) {
  __shared__ double red[kCoefShares][32];
  chain_trigger();
  const int s = blockIdx.x, q = blockIdx.z, lane = threadIdx.x & 31, y = threadIdx.x >> 5, k = blockIdx.y * 32 + lane;
  const int b = s / chains, c = s - b * chains;
  const int i0 = L.inst_item0[b], i1 = L.inst_item0[b + 1];
  chain_wait();
  if (sys_any && !sys_any[s]) return;
  double acc = 0.0;
  if (k < rank) {
#pragma unroll 4
    for (int it = i0 + y; it < i1; it += kCoefShares) acc += partial[(((int64_t)it * chains + c) * m + q) * rank + k];
  }
  red[y][lane] = acc;
  __syncthreads();
  if (y != 0 || k >= rank) return;
#pragma unroll
  for (int u = 1; u < kCoefShares; ++u) acc += red[u][lane];
  const int64_t e = ((int64_t)s * m + q) * rank + k;
  coef[e] = d[e] * acc;
}

// z[c, i, q] = r[c, i, q] + sum_k U[c, k, i] coef[s, q, k]; partials of r.z per column;
// inside an iteration (count set) the system's last CTA takes the columns' beta steps
template <int NC>
__global__ void __launch_bounds__(kTile) mcg_apply_kernel(DevLayout L, int chains, int64_t n_total, int m, int rank,
                                                          const float* U, const double* coef, const float* r, float* z,
                                                          int32_t* sys_any, double* prz, uint32_t* count, McgCol* st,
                                                          const double* prr, double tol, int maxiter,
                                                          int32_t* n_active) {
  extern __shared__ __align__(16) float cf[];   // rank x NC
  __shared__ double red[kTile / 32 * NC];
  __shared__ int s_last;
  chain_trigger();
  const int item = blockIdx.x, c = blockIdx.y;
  const int b = L.item_inst[item];
  const int s = b * chains + c;
  const int64_t i = L.item_row0[item] + threadIdx.x;
  const bool valid = i < L.offsets[b + 1];
  chain_wait();
  if (sys_any && !sys_any[s]) return;
  for (int e = threadIdx.x; e < NC * rank; e += blockDim.x) {
    const int q = e / rank, k = e - q * rank;
    cf[k * NC + q] = q < m ? (float)coef[((int64_t)s * m + q) * rank + k] : 0.f;
  }
  __syncthreads();
  float acc[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) acc[q] = 0.f;
  if (valid) {
    const float* Ui = U + (int64_t)c * rank * n_total + i;
#pragma unroll 4
    for (int k = 0; k < rank; ++k) {
      const float u = Ui[(int64_t)k * n_total];
#pragma unroll
      for (int q = 0; q < NC; q += 4) {
        const float4 f = *reinterpret_cast<const float4*>(cf + k * NC + q);
        acc[q] = fmaf(u, f.x, acc[q]);
        acc[q + 1] = fmaf(u, f.y, acc[q + 1]);
        acc[q + 2] = fmaf(u, f.z, acc[q + 2]);
        acc[q + 3] = fmaf(u, f.w, acc[q + 3]);
      }
    }
  }
  double v[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    v[q] = 0.0;
    if (valid && q < m) {
      const int64_t o = ((int64_t)c * n_total + i) * m + q;
      const float rv = r[o];
      const float zv = rv + acc[q];
      z[o] = zv;
      v[q] = (double)rv * zv;
    }
  }
  block_sums<NC>(v, m, red, [&](int q, double t) { prz[((int64_t)item * chains + c) * m + q] = t; });
  if (!count) return;
  __syncthreads();
  if (threadIdx.x == 0) s_last = last_arrival(&count[s], 1u, (uint32_t)(L.inst_item0[b + 1] - L.inst_item0[b]));
  __syncthreads();
  if (!s_last) return;
  for (int col = threadIdx.x >> 5; col < m; col += kTile / 32) {
    McgCol& k = st[(int64_t)s * m + col];
    if (!k.active) continue;
    const double rr = col_sum(L, b, c, chains, m, col, prr), rz = col_sum(L, b, c, chains, m, col, prz);
    if ((threadIdx.x & 31) == 0 && !mcg_beta_step(k, rr, rz, 1, tol, maxiter)) mcg_drop(sys_any, n_active, s);
  }
}

// rz of every column from the per-tile partials (after the first preconditioning)
__global__ void mcg_set_rz_kernel(DevLayout L, int n_inst, int chains, int m, const double* prz, McgCol* cols) {
  const int64_t e = (int64_t)blockIdx.x * kColWarps + (threadIdx.x >> 5);
  if (e >= (int64_t)n_inst * chains * m) return;
  const int s = (int)(e / m), col = (int)(e - (int64_t)s * m);
  const int b = s / chains, c = s - b * chains;
  const double rz = col_sum(L, b, c, chains, m, col, prz);
  if ((threadIdx.x & 31) == 0) cols[e].rz = rz;
}

}  // namespace

cudaError_t launch_mcg_factors(const PcgPrecond& P, int n_sys, int m, int n_theta, const double* theta,
                               const float* shifts, double* d, cudaStream_t st) {
  const int64_t n = (int64_t)n_sys * m * P.rank;
  mcg_factors_kernel<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(n, m, P.rank, n_theta, theta, shifts, P.lam, d);
  return cudaGetLastError();
}

template <int NC>
static cudaError_t mcg_precond_nc(const DevLayout& L, int n_items, int n_inst, int chains, int64_t n_total, int m,
                                  const PcgPrecond& P, const double* d, const float* r, float* z, int32_t* sys_any,
                                  double* proj, double* coef, double* prz, const McgBetaHook& h, bool chained,
                                  cudaStream_t st) {
  const dim3 grid(n_items, chains);
  cudaError_t e = launch_chained(chained, mcg_proj_kernel<NC>, grid, kTile, 0, st, L, chains, n_total, m, P.rank, P.U, r,
                                 sys_any, proj);
  if (e == cudaSuccess)
    e = launch_chained(chained, mcg_coef_kernel, dim3(n_inst * chains, (P.rank + 31) / 32, m), 32 * kCoefShares, 0, st,
                       L, chains, m, P.rank, d, proj, sys_any, coef);
  if (e == cudaSuccess)
    e = launch_chained(chained, mcg_apply_kernel<NC>, grid, kTile, sizeof(float) * NC * P.rank, st, L, chains, n_total,
                       m, P.rank, P.U, coef, r, z, sys_any, prz, h.count, h.cols, h.prr, h.tol, h.maxiter, h.n_active);
  return e;
}

cudaError_t launch_mcg_precond(const DevLayout& L, int n_items, int n_inst, int chains, int64_t n_total, int m,
                               const PcgPrecond& P, const double* d, const float* r, float* z, int32_t* sys_any,
                               double* proj, double* coef, double* prz, const McgBetaHook& h, bool chained,
                               cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  return m <= 16 ? mcg_precond_nc<16>(L, n_items, n_inst, chains, n_total, m, P, d, r, z, sys_any, proj, coef, prz, h,
                                      chained, st)
                 : mcg_precond_nc<32>(L, n_items, n_inst, chains, n_total, m, P, d, r, z, sys_any, proj, coef, prz, h,
                                      chained, st);
}

cudaError_t launch_mcg_set_rz(const DevLayout& L, int n_inst, int chains, int m, const double* prz, McgCol* cols,
                              cudaStream_t st) {
  const int64_t n = (int64_t)n_inst * chains * m;
  mcg_set_rz_kernel<<<(unsigned)((n + kColWarps - 1) / kColWarps), 32 * kColWarps, 0, st>>>(L, n_inst, chains, m, prz,
                                                                                          cols);
  return cudaGetLastError();
}

cudaError_t launch_mcg_finish(int64_t n_cols, const McgCol* cols, int accumulate, int32_t* col_status,
                              int32_t* col_iters, cudaStream_t st) {
  if (n_cols == 0) return cudaSuccess;
  const int blocks = (int)std::min<int64_t>((n_cols + 255) / 256, 1024);
  mcg_finish_kernel<<<blocks, 256, 0, st>>>(n_cols, cols, accumulate, col_status, col_iters);
  return cudaGetLastError();
}

cudaError_t launch_mcg_mask(const DevLayout& L, int n_items, int chains, int64_t n_total, int m, const McgCol* cols,
                            float* r, cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  mcg_mask_kernel<<<dim3(n_items, chains), kTile, 0, st>>>(L, chains, n_total, m, cols, r);
  return cudaGetLastError();
}

cudaError_t launch_mcg_refine(int64_t n_cols, int outer, McgCol* cols, double* prev_rr, int32_t* n_active,
                              double* worst, cudaStream_t st) {
  mcg_refine_kernel<<<1, 256, 0, st>>>(n_cols, outer, cols, prev_rr, n_active, worst);
  return cudaGetLastError();
}

cudaError_t launch_mcg_undo(const DevLayout& L, int n_items, int chains, int64_t n_total, int m, const McgCol* cols,
                            const float* dx, float* x, cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  mcg_undo_kernel<<<dim3(n_items, chains), kTile, 0, st>>>(L, chains, n_total, m, cols, dx, x);
  return cudaGetLastError();
}

cudaError_t launch_mcg_refine_finish(int64_t n_cols, const McgCol* cols, int32_t* col_status, cudaStream_t st) {
  if (n_cols == 0) return cudaSuccess;
  const int blocks = (int)std::min<int64_t>((n_cols + 255) / 256, 1024);
  mcg_refine_finish_kernel<<<blocks, 256, 0, st>>>(n_cols, cols, col_status);
  return cudaGetLastError();
}

cudaError_t launch_mcg_init(const DevLayout& L, int n_items, int chains, int64_t n_total, int m, const float* b,
                            int b_cols, const float* q, int warm, float* x, float* r, float* p, double* partial2,
                            cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  mcg_init_kernel<<<dim3(n_items, chains), kTile, 0, st>>>(L, chains, n_total, m, b, b_cols, q, warm, x, r, p,
                                                           partial2);
  return cudaGetLastError();
}

cudaError_t launch_mcg_reduce_init(const DevLayout& L, int n_inst, int chains, int m, const double* partial2,
                                   double tol, McgCol* st, int32_t* sys_any, int32_t* n_active, cudaStream_t s) {
  const int64_t n = (int64_t)n_inst * chains * m;
  const cudaError_t e = cudaMemsetAsync(sys_any, 0, sizeof(int32_t) * (size_t)n_inst * chains, s);
  if (e != cudaSuccess) return e;
  mcg_reduce_init_kernel<<<(unsigned)((n + kColWarps - 1) / kColWarps), 32 * kColWarps, 0, s>>>(
      L, n_inst, chains, m, partial2, tol, st, sys_any, n_active);
  return cudaGetLastError();
}

cudaError_t launch_mcg_dot(const DevLayout& L, int n_items, int chains, int64_t n_total, int m, const float* p,
                           const float* q, int32_t* sys_any, double* partial, uint32_t* count, McgCol* cols, int pre,
                           int32_t* n_active, bool chained, cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  return launch_chained(chained, m <= 16 ? mcg_dot_kernel<16> : mcg_dot_kernel<32>, dim3(n_items, chains), kTile, 0, st,
                        L, chains, n_total, m, p, q, sys_any, partial, count, cols, pre, n_active);
}

cudaError_t launch_mcg_update_xr(const DevLayout& L, int n_items, int chains, int64_t n_total, int m, McgCol* cols,
                                 int32_t* sys_any, float* x, float* r, const float* p, const float* q, double* partial,
                                 uint32_t* count, double tol, int maxiter, int32_t* n_active, bool chained,
                                 cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  return launch_chained(chained, m <= 16 ? mcg_update_xr_kernel<16> : mcg_update_xr_kernel<32>, dim3(n_items, chains),
                        kTile, 0, st, L, chains, n_total, m, cols, sys_any, x, r, p, q, partial, count, tol, maxiter,
                        n_active);
}

cudaError_t launch_mcg_update_p(const DevLayout& L, int n_items, int chains, int64_t n_total, int m,
                                const McgCol* stt, const int32_t* sys_any, const float* r, float* p, bool chained,
                                cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  return launch_chained(chained, mcg_update_p_kernel, dim3(n_items, chains), kTile, 0, st, L, chains, n_total, m, stt,
                        sys_any, r, p);
}

}  // namespace kmv

// The implicit midpoint step of Sec. 3.2.3 (Eq. implicitsystem), solved by
// Anderson acceleration (App. B) of the fixed-point map of Eq. Phi on the
// stacked vector z = (theta, pi, x) of every system:
//   Phi(z) = (theta_0 + dt (pi_0 + pi)/2,
//             pi_0 - dt f_phi((theta_0 + theta)/2, x),
//             x + R (y - A((theta_0 + theta)/2) x)),
// with f_phi the frozen-x force of Sec. 3.2.1 (plus the prior's gradient) and
// R = (Nystrom P^{-1} or I) / c, c ~ rho(that A(theta_0)) from a power iteration.
// Anderson: the last k pairs (g_i = Phi(z_i), f_i = z_i - g_i) kept in a ring;
// alpha minimises |sum alpha_i f_i| subject to sum alpha_i = 1 (from the k x k
// Gram matrix of the f_i, FP64, updated by one row per iteration), and the next
// iterate is sum alpha_i g_i.  theta, pi (FP64) and x (FP32) form one vector;
// inner products are FP64, per-tile partials summed in a fixed order.
#include <algorithm>

#include "kmv_internal.cuh"
#include "simt_common.cuh"

namespace kmv {
namespace {

__device__ __forceinline__ double tsum(const DevLayout& L, int b, int c, int chains, const double* partial, int stride,
                                       int k) {
  double acc = 0.0;
#pragma unroll 4
  for (int it = L.inst_item0[b]; it < L.inst_item0[b + 1]; ++it) acc += partial[((int64_t)it * chains + c) * stride + k];
  return acc;
}
// The same sum by a full warp (every lane gets it), for systems of many tiles.
__device__ __forceinline__ double tsum_warp(const DevLayout& L, int b, int c, int chains, const double* partial,
                                            int stride, int k) {
  double acc = 0.0;
  for (int it = L.inst_item0[b] + (int)(threadIdx.x & 31); it < L.inst_item0[b + 1]; it += 32)
    acc += partial[((int64_t)it * chains + c) * stride + k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return acc;
}
constexpr int kSerialTiles = 64;   // up to here a lane sums a system's tiles alone, in their order

// theta_bar = (theta_0 + theta) / 2
__global__ void imp_mid_kernel(int n, const double* th0, const double* th, double* tb) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x)
    tb[e] = 0.5 * (th0[e] + th[e]);
}

// r = y - q; partials of r.r and y.y
__global__ void imp_resid_kernel(DevLayout L, int chains, int64_t n_total, const float* y, const float* q,
                                 const int32_t* active, float* r, double* partial2) {
  __shared__ double red[kTile / 32 * 2];
  chain_trigger();
  const int item = blockIdx.x, c = blockIdx.y;
  const int b = L.item_inst[item];
  const int64_t i = L.item_row0[item] + threadIdx.x, r1 = L.offsets[b + 1];
  chain_wait();
  if (!active[b * chains + c]) return;
  double ry[2] = {0.0, 0.0};
  if (i < r1) {
    const int64_t v = (int64_t)c * n_total + i;
    const float rv = y[i] - q[v];
    r[v] = rv;
    ry[0] = (double)rv * rv;
    ry[1] = (double)y[i] * y[i];
  }
  block_sum_many<2>(ry, 2, red, [&](int k, double t) { partial2[((int64_t)item * chains + c) * 2 + k] = t; });
}

// x part of Phi: g_x = x + z / c, f_x = x - g_x into ring slot `slot`; partials of
// <f_x, F_x[i]> for the stored slots i < cnt
__global__ void imp_x_kernel(DevLayout L, int chains, int64_t n_total, int k, int slot, int cnt, const float* x,
                             const float* z, const double* cscale, const int32_t* active, float* Gx, float* Fx,
                             double* partial) {
  __shared__ double red[kTile / 32 * kMaxAA];
  __shared__ float s_inv;
  chain_trigger();
  const int item = blockIdx.x, c = blockIdx.y;
  const int b = L.item_inst[item];
  const int s = b * chains + c;
  const int64_t i = L.item_row0[item] + threadIdx.x;
  const bool valid = i < L.offsets[b + 1];
  const int64_t vec = (int64_t)chains * n_total, v = (int64_t)c * n_total + i;
  chain_wait();
  if (!active[s]) return;
  if (threadIdx.x == 0) s_inv = (float)(1.0 / cscale[s]);
  // the stored f of the row, while the division runs
  float fj[kMaxAA];
#pragma unroll
  for (int j = 0; j < kMaxAA; ++j) fj[j] = valid && j < cnt && j != slot ? Fx[(int64_t)j * vec + v] : 0.f;
  __syncthreads();
  float f = 0.f;
  if (valid) {
    const float step = s_inv * z[v];
    Gx[(int64_t)slot * vec + v] = x[v] + step;
    f = -step;
    Fx[(int64_t)slot * vec + v] = f;
  }
  double t[kMaxAA];
#pragma unroll
  for (int j = 0; j < kMaxAA; ++j) t[j] = j < cnt ? (double)f * (double)(j == slot ? f : fj[j]) : 0.0;
  auto put = [&](int j, double sum) { partial[((int64_t)item * chains + c) * k + j] = sum; };
  if (cnt <= 10) {
    // the usual depth: fewer sums
    double u[10];
#pragma unroll
    for (int j = 0; j < 10; ++j) u[j] = t[j];
    block_sum_many<10>(u, cnt, red, put);
  } else {
    block_sum_many<kMaxAA>(t, cnt, red, put);
  }
}

// theta, pi part of Phi, the new Gram row, the stopping test, the Anderson
// coefficients, and the next theta, pi (sum_i alpha_i G_tp[i], or the newest Phi of a
// system that finishes) with its midpoint; one warp per system.  State per system: H
// (k x k Gram), alpha (k); ring slots of G_tp, F_tp (k x 2n).  Lane p takes component
// p, lane j Gram entry j, lane i row i of the Cholesky factor, every sum in its serial
// order.  An FP64 operation takes 65 clocks, a division or square root some 600, and
// one thread took 68 us per iteration.
constexpr int kAAWarps = 2;
__global__ void __launch_bounds__(32 * kAAWarps) imp_aa_kernel(
    DevLayout L, int n_inst, int chains, int n, int k, int slot, int cnt, const double* th0, const double* pi0,
    double* th, double* pi, const double* grad, const double* mu, const double* prec, const uint8_t* mask, double dt,
    const double* xpart, const double* rpart, double tol, int iter, int maxiter, double* Gtp, double* Ftp, double* H,
    double* alpha, int32_t* active, int32_t* done_now, int32_t* status, int32_t* iters, int32_t* n_active,
    double* best_rr, int32_t* best_it, double* tb_next) {
  chain_trigger();
  chain_wait();
  const int s = blockIdx.x * kAAWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (s >= n_inst * chains) return;
  if (!active[s]) {
    if (lane == 0) done_now[s] = 0;
    return;
  }
  const int b = s / chains, c = s - b * chains;
  const int nn = 2 * n;
  const int64_t n_sys = (int64_t)n_inst * chains;
  double* g = Gtp + ((int64_t)slot * n_sys + s) * nn;
  double* f = Ftp + ((int64_t)slot * n_sys + s) * nn;
  double fm = 0.0, gm = 0.0;
  for (int p = lane; p < n; p += 32) {
    const int64_t e = (int64_t)s * n + p;
    const double free = (mask == nullptr || mask[p]) ? 1.0 : 0.0;
    const double tb = 0.5 * (th0[e] + th[e]);
    double F = grad[e];
    if (prec) F += prec[p] * (tb - mu[p]);
    const double gt = th0[e] + dt * 0.5 * (pi0[e] + pi[e]) * free;
    const double gp = pi0[e] - dt * F * free;
    g[p] = gt;
    g[n + p] = gp;
    f[p] = th[e] - gt;
    f[n + p] = pi[e] - gp;
    fm = fmax(fm, fmax(fabs(f[p]), fabs(f[n + p])));
    gm = fmax(gm, fmax(fabs(gt), fabs(gp)));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    fm = fmax(fm, __shfl_xor_sync(0xffffffffu, fm, o));
    gm = fmax(gm, __shfl_xor_sync(0xffffffffu, gm, o));
  }
  __syncwarp();
  // new Gram row: the theta-pi part plus the x part's tile partials; r.r and y.y in
  // the lanes after it
  double* Hs = H + (int64_t)s * k * k;
  double v = 0.0;
  if (L.inst_item0[b + 1] - L.inst_item0[b] <= kSerialTiles) {
    if (lane < cnt + 2)
      v = lane < cnt ? tsum(L, b, c, chains, xpart, k, lane) : tsum(L, b, c, chains, rpart, 2, lane - cnt);
  } else {
    for (int j = 0; j < cnt + 2; ++j) {
      const double t = j < cnt ? tsum_warp(L, b, c, chains, xpart, k, j) : tsum_warp(L, b, c, chains, rpart, 2, j - cnt);
      if (lane == j) v = t;
    }
  }
  const double rr = __shfl_sync(0xffffffffu, v, cnt), yy = __shfl_sync(0xffffffffu, v, cnt + 1);
  if (lane < cnt) {
    const double* fj = Ftp + ((int64_t)lane * n_sys + s) * nn;
    for (int p = 0; p < nn; ++p) v += f[p] * fj[p];
    Hs[slot * k + lane] = v;
    Hs[lane * k + slot] = v;
  }
  const double hss = __shfl_sync(0xffffffffu, v, slot);
  __syncwarp();
  // the linear residual stops falling at the floor of the FP32 product (about
  // 2^-24 |A| |x|): below 1e-3 |y|, no halving for 8k iterations counts as
  // having reached it
  const bool better = iter == 0 || rr < 0.25 * best_rr[s];
  const int since = better ? 0 : iter - best_it[s];
  __syncwarp();
  if (lane == 0) {
    iters[s] = iter + 1;
    if (better) {
      best_rr[s] = rr;
      best_it[s] = iter;
    }
  }
  const bool at_floor = since >= 8 * k && rr <= 1e-6 * yy;
  const bool finite = isfinite(rr) && isfinite(fm) && isfinite(hss);
  const bool conv = (rr <= tol * tol * yy || at_floor) && fm <= tol * (1.0 + gm);
  const bool finish = !finite || conv || iter + 1 >= maxiter;
  double al = 0.0;   // lane i < cnt: alpha_i
  if (finish) {
    // the result is this iteration's Phi(z)
    if (lane == 0) {
      status[s] = !finite ? KMV_ENONFINITE : (conv ? KMV_OK : KMV_ENOTCONV);
      active[s] = 0;
      done_now[s] = 1;
      atomicSub(n_active, 1);
    }
  } else {
    // alpha = H^{-1} 1 / (1^T H^{-1} 1), by Cholesky of H + ridge (newest slot alone on
    // failure); lane cnt carries the right-hand side 1 through the elimination
    double dmax = 0.0;
    for (int i = 0; i < cnt; ++i) dmax = fmax(dmax, Hs[i * k + i]);
    bool ok = dmax > 0.0;
    double row[kMaxAA];   // row `lane` of the factor; lane cnt: the forward solution
#pragma unroll
    for (int j = 0; j < kMaxAA; ++j) row[j] = 0.0;
#pragma unroll
    for (int j = 0; j < kMaxAA; ++j) {
      if (j < cnt && ok) {
        double w = lane < cnt ? Hs[lane * k + j] + (lane == j ? 1e-13 * dmax : 0.0) : 1.0;
#pragma unroll
        for (int p = 0; p < j; ++p) w -= row[p] * __shfl_sync(0xffffffffu, row[p], j);
        const double piv = __shfl_sync(0xffffffffu, w, j);
        ok = piv > 0.0;
        const double d = sqrt(piv);
        row[j] = lane == j ? d : w / d;
      }
    }
    if (ok) {
      // back: Hc^T a = u
      double a = 0.0;   // lane i: a_i once solved
#pragma unroll
      for (int i = kMaxAA - 1; i >= 0; --i) {
        if (i < cnt) {
          double w = __shfl_sync(0xffffffffu, row[i], cnt);
#pragma unroll
          for (int p = i + 1; p < kMaxAA; ++p)
            if (p < cnt) w -= __shfl_sync(0xffffffffu, row[i], p) * __shfl_sync(0xffffffffu, a, p);
          w = w / __shfl_sync(0xffffffffu, row[i], i);
          if (lane == i) a = w;
        }
      }
      double sa = 0.0;
      for (int i = 0; i < cnt; ++i) sa += __shfl_sync(0xffffffffu, a, i);
      ok = sa != 0.0 && isfinite(sa);
      if (ok) al = a / sa;
    }
    if (!ok) al = lane == slot ? 1.0 : 0.0;
    if (lane < cnt) alpha[(int64_t)s * k + lane] = al;
    if (lane == 0) done_now[s] = 0;
  }
  // theta, pi of the next iterate and the midpoint it is evaluated at
  for (int p0 = 0; p0 < nn; p0 += 32) {
    const int p = p0 + lane;
    double v2 = 0.0;
    if (finish) {
      if (p < nn) v2 = g[p];
    } else {
      for (int i = 0; i < cnt; ++i) {
        const double ai = __shfl_sync(0xffffffffu, al, i);
        if (p < nn) v2 += ai * Gtp[((int64_t)i * n_sys + s) * nn + p];
      }
    }
    if (p < n) {
      th[(int64_t)s * n + p] = v2;
      tb_next[(int64_t)s * n + p] = 0.5 * (th0[(int64_t)s * n + p] + v2);
    } else if (p < nn) {
      pi[(int64_t)s * n + p - n] = v2;
    }
  }
}

// x = sum_i alpha_i G_x[i] (continuing) or the newest Phi's x (finished this iteration),
// and the next force's columns [x, phi], [-x/2, phi/2] (phi's entries stand).
__global__ void imp_x_mix_kernel(DevLayout L, int chains, int64_t n_total, int k, int slot, int cnt,
                                 const float* Gx, const double* alpha, const int32_t* active,
                                 const int32_t* done_now, float* x, float* Vf, float* Gf) {
  chain_trigger();
  const int item = blockIdx.x, c = blockIdx.y;
  const int b = L.item_inst[item];
  const int s = b * chains + c;
  const int64_t i = L.item_row0[item] + threadIdx.x, r1 = L.offsets[b + 1];
  const int64_t vec = (int64_t)chains * n_total, v = (int64_t)c * n_total + i;
  chain_wait();
  const bool done = done_now[s];
  if ((!active[s] && !done) || i >= r1) return;
  float xv;
  if (done) {
    xv = Gx[(int64_t)slot * vec + v];
  } else {
    double acc = 0.0;
#pragma unroll 4
    for (int j = 0; j < cnt; ++j) acc += alpha[(int64_t)s * k + j] * (double)Gx[(int64_t)j * vec + v];
    xv = (float)acc;
  }
  x[v] = xv;
  Vf[2 * v] = xv;
  Gf[2 * v] = -0.5f * xv;
}

// --- power iteration for c ~ rho(R~ A(theta_0)), R~ = P^{-1} or I -----------------------

// v = w / |w| per system (partial of w.w given), and the running estimate c = |w| / |v_prev| (|v_prev| = 1)
__global__ void imp_norm_kernel(DevLayout L, int n_inst, int chains, const double* partial, double* cscale) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n_inst * chains) return;
  const int b = s / chains, c = s - b * chains;
  cscale[s] = sqrt(tsum(L, b, c, chains, partial, 1, 0));
}

__global__ void imp_scale_kernel(DevLayout L, int chains, int64_t n_total, const double* norm, const float* w,
                                 float* v, double* partial) {
  __shared__ double red[kTile / 32];
  const int item = blockIdx.x, c = blockIdx.y;
  const int b = L.item_inst[item];
  const int s = b * chains + c;
  const int64_t i = L.item_row0[item] + threadIdx.x;
  double t = 0.0;
  if (i < L.offsets[b + 1]) {
    const int64_t e = (int64_t)c * n_total + i;
    const double nv = norm ? norm[s] : 0.0;
    const float val = norm ? (nv > 0.0 ? (float)(w[e] / nv) : 0.f) : w[e];
    v[e] = val;
    t = (double)val * val;
  }
  t = block_sum(t, red);
  if (threadIdx.x == 0) partial[(int64_t)item * chains + c] = t;
}

__global__ void imp_cfinal_kernel(int n_sys, double safety, double* cscale) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n_sys) return;
  const double v = cscale[s] * safety;
  cscale[s] = (v > 0.0 && isfinite(v)) ? v : 1.0;
}

__global__ void fill_i32_kernel(int32_t* v, int n, int32_t val) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) v[e] = val;
}

}  // namespace

cudaError_t launch_fill_i32(int32_t* v, int n, int32_t val, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  fill_i32_kernel<<<(n + 255) / 256, 256, 0, st>>>(v, n, val);
  return cudaGetLastError();
}

cudaError_t launch_imp_mid(int n, const double* th0, const double* th, double* tb, cudaStream_t st) {
  imp_mid_kernel<<<(n + 255) / 256, 256, 0, st>>>(n, th0, th, tb);
  return cudaGetLastError();
}

cudaError_t launch_imp_resid(const DevLayout& L, int n_items, int chains, int64_t n_total, const float* y,
                             const float* q, const int32_t* active, float* r, double* partial2, bool chained,
                             cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  return launch_chained(chained, imp_resid_kernel, dim3(n_items, chains), kTile, 0, st, L, chains, n_total, y, q, active,
                        r, partial2);
}

cudaError_t launch_imp_x(const DevLayout& L, int n_items, int chains, int64_t n_total, int k, int slot, int cnt,
                         const float* x, const float* z, const double* cscale, const int32_t* active, float* Gx,
                         float* Fx, double* partial, bool chained, cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  return launch_chained(chained, imp_x_kernel, dim3(n_items, chains), kTile, 0, st, L, chains, n_total, k, slot, cnt, x,
                        z, cscale, active, Gx, Fx, partial);
}

cudaError_t launch_imp_aa(const DevLayout& L, int n_inst, int chains, int n, int k, int slot, int cnt,
                          const double* th0, const double* pi0, double* th, double* pi, const double* grad,
                          const double* mu, const double* prec, const uint8_t* mask, double dt, const double* xpart,
                          const double* rpart, double tol, int iter, int maxiter, double* Gtp, double* Ftp, double* H,
                          double* alpha, int32_t* active, int32_t* done_now, int32_t* status, int32_t* iters,
                          int32_t* n_active, double* best_rr, int32_t* best_it, double* tb_next, bool chained,
                          cudaStream_t st) {
  const int n_sys = n_inst * chains;
  return launch_chained(chained, imp_aa_kernel, dim3((n_sys + kAAWarps - 1) / kAAWarps), 32 * kAAWarps, 0, st, L, n_inst,
                        chains, n, k, slot, cnt, th0, pi0, th, pi, grad, mu, prec, mask, dt, xpart, rpart, tol, iter,
                        maxiter, Gtp, Ftp, H, alpha, active, done_now, status, iters, n_active, best_rr, best_it,
                        tb_next);
}

cudaError_t launch_imp_mix(const DevLayout& L, int n_items, int chains, int64_t n_total, int k, int slot, int cnt,
                           const float* Gx, const double* alpha, const int32_t* active, const int32_t* done_now,
                           float* x, float* Vf, float* Gf, bool chained, cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  return launch_chained(chained, imp_x_mix_kernel, dim3(n_items, chains), kTile, 0, st, L, chains, n_total, k, slot, cnt,
                        Gx, alpha, active, done_now, x, Vf, Gf);
}

cudaError_t launch_imp_scale(const DevLayout& L, int n_items, int chains, int64_t n_total, const double* norm,
                             const float* w, float* v, double* partial, cudaStream_t st) {
  if (n_items == 0) return cudaSuccess;
  imp_scale_kernel<<<dim3(n_items, chains), kTile, 0, st>>>(L, chains, n_total, norm, w, v, partial);
  return cudaGetLastError();
}

cudaError_t launch_imp_norm(const DevLayout& L, int n_inst, int chains, const double* partial, double* cscale,
                            cudaStream_t st) {
  const int n = n_inst * chains;
  imp_norm_kernel<<<(n + 127) / 128, 128, 0, st>>>(L, n_inst, chains, partial, cscale);
  return cudaGetLastError();
}

cudaError_t launch_imp_cfinal(int n_sys, double safety, double* cscale, cudaStream_t st) {
  imp_cfinal_kernel<<<(n_sys + 127) / 128, 128, 0, st>>>(n_sys, safety, cscale);
  return cudaGetLastError();
}

}  // namespace kmv

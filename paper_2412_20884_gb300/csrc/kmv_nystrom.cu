// Randomized Nystrom preconditioner (Frangella, Tropp and Udell), which the
// paper uses for its solves (Sec. 3.1, end; Sec. 3.2.3; Sec. 4), one per
// system s = (instance, chain):
//   Y = K Omega (one r-column product, no noise term), nu a small shift (below),
//   Y_nu = Y + nu Omega,  Omega^T Y_nu = L L^T,  B = Y_nu L^{-T} = U S W^T,
//   Lambda = max(S^2 - nu, 0),  K ~ U Lambda U^T,
// and for A = K + mu I the Woodbury form
//   P^{-1} = (lambda_r + mu) U (Lambda + mu)^{-1} U^T + (I - U U^T).
// B's SVD is taken through r x r matrices: with the three Gram matrices
// O^T Y, O^T O and Y^T Y (one pass over the rows), B^T B = L^{-1} Y_nu^T Y_nu
// L^{-T} = M, M = W S^2 W^T by cyclic Jacobi (FP64), and U = Y_nu T with
// T = L^{-T} W S^{-1}.  U is stored column by column, (chains, r, N_total),
// so that U^T r and U w read it with coalesced rows in the CG.
#include <algorithm>
#include <cmath>

#include "kmv_internal.cuh"
#include "simt_common.cuh"

namespace kmv {
namespace {

constexpr int kGB = 32;   // Gram / U block edge

// grams[s] = [O^T Y, O^T O, Y^T Y] (r x r each, FP64 products and sums), one
// 32 x 32 block of one matrix per CTA, rows staged 32 at a time.  FP64 throughout: the
// columns of U = Y_nu T come out orthonormal only as far as these sums are exact, and
// the preconditioner stays positive definite only while that error is below
// (lambda_r + mu) / (lambda_1 + mu).  Every entry is one chain over the rows in order.
// Bound by the FP64 pipe (2 lanes per clock and SM, conversions included): the staged
// values are converted once, and the symmetric matrices' lower blocks are mirrored
// (u v and v u round alike): 36 blocks in place of 48 at r = 128, 24.8 ms before at
// N = 16,384 with 8 chains.
__global__ void __launch_bounds__(256) ny_gram_kernel(DevLayout L, int chains, int64_t n_total, int r, int nb,
                                                      const float* Om, const float* Y, double* grams) {
  __shared__ double ak[kGB][kGB + 1], bl[kGB][kGB + 1];
  const int s = blockIdx.x;
  const int b = s / chains, c = s - b * chains;
  // block index -> matrix g and block (kb, lb): all of O^T Y, the upper blocks of the others
  int e = blockIdx.y, g = 0, kb, lb;
  if (e < nb * nb) {
    kb = e / nb;
    lb = e - kb * nb;
  } else {
    e -= nb * nb;
    const int half = nb * (nb + 1) / 2;
    g = 1 + e / half;
    e -= (g - 1) * half;
    kb = 0;
    while (e >= nb - kb) e -= nb - kb++;
    lb = kb + e;
  }
  const float* A = g == 2 ? Y : Om;
  const float* B = g == 1 ? Om : Y;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 32 x 8
  const int64_t j0 = L.offsets[b], j1 = L.offsets[b + 1];
  double acc[4] = {};
  float fa[4], fb[4];   // the next rows, loaded while the current ones are summed
  auto fetch = [&](int64_t i0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int64_t i = i0 + ty + 8 * q;
      const int k = kb * kGB + tx, l = lb * kGB + tx;
      const int64_t base = ((int64_t)c * n_total + i) * r;
      fa[q] = i < j1 && k < r ? A[base + k] : 0.f;
      fb[q] = i < j1 && l < r ? B[base + l] : 0.f;
    }
  };
  fetch(j0);
  for (int64_t i0 = j0; i0 < j1; i0 += kGB) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      ak[ty + 8 * q][tx] = fa[q];
      bl[ty + 8 * q][tx] = fb[q];
    }
    __syncthreads();
    if (i0 + kGB < j1) fetch(i0 + kGB);
#pragma unroll 4
    for (int rr = 0; rr < kGB; ++rr) {
      const double v = bl[rr][tx];
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] = fma(ak[rr][ty + 8 * q], v, acc[q]);
    }
    __syncthreads();
  }
  const int l = lb * kGB + tx;
  double* out = grams + ((int64_t)s * 3 + g) * r * r;
  for (int q = 0; q < 4; ++q) {
    const int k = kb * kGB + ty + 8 * q;
    if (k < r && l < r) {
      out[k * r + l] = acc[q];
      if (g > 0 && kb != lb) out[l * r + k] = acc[q];
    }
  }
}

// W = sym(O^T Y) + nu O^T O (block-wide).
__device__ void fill_w(const double* OY, const double* OO, double nu, int r, double* W) {
  for (int e = threadIdx.x; e < r * r; e += blockDim.x) {
    const int k = e / r, l = e - k * r;
    W[e] = 0.5 * (OY[e] + OY[l * r + k]) + nu * OO[e];
  }
  __syncthreads();
}

// In-place Cholesky W = L L^T (lower triangle) by the whole block, right-looking;
// false (for every thread) at a pivot that is not positive and finite.
__device__ bool block_cholesky(double* W, int r, int* fail) {
  const int tid = threadIdx.x, nt = blockDim.x;
  if (tid == 0) *fail = 0;
  __syncthreads();
  for (int j = 0; j < r; ++j) {
    if (tid == 0) {
      const double piv = W[j * r + j];
      if (!(piv > 0.0) || !isfinite(piv)) *fail = 1;
      else W[j * r + j] = sqrt(piv);
    }
    __syncthreads();
    if (*fail) break;
    const double djj = W[j * r + j];
    for (int i = j + 1 + tid; i < r; i += nt) W[i * r + j] /= djj;
    __syncthreads();
    const int m = r - j - 1;
    for (int e = tid; e < m * m; e += nt) {
      const int i = j + 1 + e / m, k = j + 1 + e % m;
      if (k <= i) W[i * r + k] -= W[i * r + j] * W[k * r + j];
    }
    __syncthreads();
  }
  const bool ok = *fail == 0;
  __syncthreads();
  return ok;
}

// The r x r part per system (FP64, matrices in the system's scratch), in three
// kernels: here (one CTA) nu, W = sym(O^T Y) + nu O^T O = L L^T and
// M = L^{-1} G_nu L^{-T}; then the Jacobi eigendecomposition M = V S2 V^T; then,
// sorted descending, lam = max(S2 - nu, 0) and T = L^{-T} V S2^{-1/2}.
// A system whose Cholesky fails at every shift (or with fewer rows than r) gets
// lam = 0 and T = 0: its preconditioner is the identity.
__global__ void __launch_bounds__(256) ny_factor_kernel(DevLayout L, int chains, int r, const double* grams,
                                                        double* scratch, double* T, double* lam, double* nu_out,
                                                        int32_t* status) {
  __shared__ double red[8];
  __shared__ double cs[8][2];
  __shared__ int fail;
  const int s = blockIdx.x;
  const int b = s / chains;
  const int64_t nb_rows = L.offsets[b + 1] - L.offsets[b];
  const double* OY = grams + (int64_t)s * 3 * r * r;
  const double* OO = OY + r * r;
  const double* YY = OO + r * r;
  double* W = scratch + (int64_t)s * 4 * r * r;   // W, then L in its lower triangle
  double* G = W + r * r;                          // G_nu, then X = L^{-1} G_nu
  double* M = G + r * r;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int rr = r * r;

  // nu: Frangella et al.'s shift sqrt(N) eps |Y| for an orthonormal test matrix,
  // with eps the FP64 unit roundoff and |Y| / |Omega| (Frobenius) for the
  // Gaussian one; Y carries the FP32 product's rounding, so nu is raised by
  // decades until the Cholesky of W succeeds, then by one decade more.
  double ty = 0.0, to = 0.0;
  for (int k = tid; k < r; k += nt) {
    ty += YY[k * r + k];
    to += OO[k * r + k];
  }
  for (int o = 16; o > 0; o >>= 1) {
    ty += __shfl_down_sync(0xffffffffu, ty, o);
    to += __shfl_down_sync(0xffffffffu, to, o);
  }
  if ((tid & 31) == 0) {
    red[tid >> 5] = ty;
    cs[tid >> 5][0] = to;
  }
  __syncthreads();
  if (tid == 0) {
    double a = 0.0, c = 0.0;
    for (int w = 0; w < nt / 32; ++w) {
      a += red[w];
      c += cs[w][0];
    }
    red[0] = sqrt((double)nb_rows) * 0x1p-52 * sqrt(fmax(a, 0.0) / fmax(c, 1e-300));
    fail = (nb_rows < r || !(a > 0.0)) ? 1 : 0;
  }
  __syncthreads();
  double nu = red[0];
  bool ok = fail == 0;
  __syncthreads();
  if (ok) {
    ok = false;
    for (int attempt = 0; attempt < 18 && !ok; ++attempt) {
      if (attempt > 0) nu *= 10.0;
      fill_w(OY, OO, nu, r, W);
      ok = block_cholesky(W, r, &fail);
    }
    if (ok) {
      nu *= 10.0;
      fill_w(OY, OO, nu, r, W);
      ok = block_cholesky(W, r, &fail);
    }
  }
  if (!ok) {
    for (int e = tid; e < rr; e += nt) T[(int64_t)s * rr + e] = 0.0;
    for (int k = tid; k < r; k += nt) lam[(int64_t)s * r + k] = 0.0;
    if (tid == 0) {
      nu_out[s] = 0.0;
      status[s] = KMV_ENOTCONV;
    }
    return;
  }
  for (int e = tid; e < rr; e += nt) {
    const int k = e / r, l = e - k * r;
    const double oy = 0.5 * (OY[e] + OY[l * r + k]);
    G[e] = YY[e] + 2.0 * nu * oy + nu * nu * OO[e];
  }
  __syncthreads();
  // X = L^{-1} G_nu, column by column (one thread per column)
  for (int c = tid; c < r; c += nt)
    for (int i = 0; i < r; ++i) {
      double v = G[i * r + c];
      for (int p = 0; p < i; ++p) v -= W[i * r + p] * G[p * r + c];
      G[i * r + c] = v / W[i * r + i];
    }
  __syncthreads();
  // M = L^{-1} X^T: column c of M solves L m = (row c of X)
  for (int c = tid; c < r; c += nt)
    for (int i = 0; i < r; ++i) {
      double v = G[c * r + i];
      for (int p = 0; p < i; ++p) v -= W[i * r + p] * M[p * r + c];
      M[i * r + c] = v / W[i * r + i];
    }
  __syncthreads();
  for (int e = tid; e < rr; e += nt) {
    const int k = e / r, l = e - k * r;
    if (k < l) {
      const double v = 0.5 * (M[e] + M[l * r + k]);
      M[e] = v;
      M[l * r + k] = v;
    }
  }
  if (tid == 0) {
    nu_out[s] = nu;
    status[s] = KMV_OK;
  }
}

// Cyclic Jacobi on a system's M (r x r), round-robin pairs (r rounded up to even; index
// r is a bye), V the product of the rotations.  A round's rotations are disjoint, so the
// 2 x 2 block of M at the rows of pair I and the columns of pair J is rotated on both
// sides by one thread from values of before the round, and every element sees the same
// operations in the same order however the blocks are spread.  Some 100 K FP64
// operations per round against 2 lanes per clock and SM: one CTA per system took
// 106 ms for 8 systems of rank 128, so a cluster of `cl` CTAs shares the blocks (M in
// L2, V by rows in shared memory) with one cluster barrier per round.
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
constexpr int kJacThreads = 256;
__global__ void __launch_bounds__(kJacThreads) ny_jacobi_kernel(int r, int cl, double* scratch, const int32_t* status) {
  extern __shared__ double vrow[];   // this CTA's rows of V
  __shared__ double red[kJacThreads / 32];
  __shared__ double cs[kMaxRank / 2 + 1][2];
  const int s = blockIdx.x / cl, rank = blockIdx.x % cl;
  if (status[s] != KMV_OK) return;   // (the whole cluster)
  double* M = scratch + (int64_t)s * 4 * r * r + 2 * (int64_t)r * r;
  double* V = M + (int64_t)r * r;
  const int tid = threadIdx.x, rr = r * r;
  const int v0 = r * rank / cl, v1 = r * (rank + 1) / cl, nv = v1 - v0;
  for (int e = tid; e < nv * r; e += kJacThreads) vrow[e] = e / r + v0 == e % r ? 1.0 : 0.0;
  const int n2 = r + (r & 1), np = n2 / 2;
  const int per = (np * np + cl - 1) / cl, e0 = rank * per, e1 = min(np * np, e0 + per);
  auto pair_of = [&](int t, int k, int& p, int& q) {
    if (k == 0) {
      p = t;
      q = n2 - 1;
    } else {
      p = t + k;
      if (p >= n2 - 1) p -= n2 - 1;
      q = t - k;
      if (q < 0) q += n2 - 1;
    }
    if (p > q) {
      const int u = p;
      p = q;
      q = u;
    }
  };
  __syncthreads();
  for (int sweep = 0; sweep < 20; ++sweep) {
    for (int t = 0; t < n2 - 1; ++t) {
      // rotations of the round (every CTA of the cluster computes them all)
      for (int k = tid; k < np; k += kJacThreads) {
        int p, q;
        pair_of(t, k, p, q);
        double c = 1.0, sn = 0.0;
        if (q < r) {
          const double apq = __ldcg(&M[p * r + q]);
          if (apq != 0.0) {
            const double th = (__ldcg(&M[q * r + q]) - __ldcg(&M[p * r + p])) / (2.0 * apq);
            const double tt = copysign(1.0, th) / (fabs(th) + sqrt(th * th + 1.0));
            c = 1.0 / sqrt(tt * tt + 1.0);
            sn = tt * c;
          }
        }
        cs[k][0] = c;
        cs[k][1] = sn;
      }
      // two blocks at a time; the first two loaded before the rotations are known
      double m00[2], m01[2], m10[2], m11[2];
      int at[2][4];
      auto load = [&](int e, int u) {
        at[u][0] = -1;
        if (e >= e1) return;
        int pi, qi, pj, qj;
        const int I = e / np, J = e - I * np;
        pair_of(t, I, pi, qi);
        pair_of(t, J, pj, qj);
        at[u][0] = pi * r + pj;
        at[u][1] = qj < r ? pi * r + qj : -1;
        at[u][2] = qi < r ? qi * r + pj : -1;
        at[u][3] = qi < r && qj < r ? qi * r + qj : -1;
        m00[u] = __ldcg(&M[at[u][0]]);
        m01[u] = at[u][1] >= 0 ? __ldcg(&M[at[u][1]]) : 0.0;
        m10[u] = at[u][2] >= 0 ? __ldcg(&M[at[u][2]]) : 0.0;
        m11[u] = at[u][3] >= 0 ? __ldcg(&M[at[u][3]]) : 0.0;
      };
      load(e0 + tid, 0);
      load(e0 + tid + kJacThreads, 1);
      __syncthreads();
      // every read of the old M by this cluster precedes every write of the new one:
      // the rotations read entries that other CTAs write
      cluster_barrier();
      for (int e = e0 + tid; e < e1; e += 2 * kJacThreads) {
        if (e != e0 + tid) {
          load(e, 0);
          load(e + kJacThreads, 1);
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          if (at[u][0] < 0) continue;
          const int eu = e + u * kJacThreads, I = eu / np, J = eu - I * np;
          if (at[u][2] >= 0) {
            const double c = cs[I][0], sn = cs[I][1];
            const double mp = m00[u], mq = m10[u];
            m00[u] = c * mp - sn * mq;
            m10[u] = sn * mp + c * mq;
            const double np_ = m01[u], nq = m11[u];
            m01[u] = c * np_ - sn * nq;
            m11[u] = sn * np_ + c * nq;
          }
          if (at[u][1] >= 0) {
            const double c = cs[J][0], sn = cs[J][1];
            const double mp = m00[u], mq = m01[u];
            m00[u] = c * mp - sn * mq;
            m01[u] = sn * mp + c * mq;
            const double np_ = m10[u], nq = m11[u];
            m10[u] = c * np_ - sn * nq;
            m11[u] = sn * np_ + c * nq;
            __stcg(&M[at[u][1]], m01[u]);
            if (at[u][3] >= 0) __stcg(&M[at[u][3]], m11[u]);
          }
          __stcg(&M[at[u][0]], m00[u]);
          if (at[u][2] >= 0) __stcg(&M[at[u][2]], m10[u]);
        }
      }
      for (int e = tid; e < np * nv; e += kJacThreads) {   // columns p, q of V J
        const int k = e % np, row = e / np;
        int p, q;
        pair_of(t, k, p, q);
        if (q >= r) continue;
        const double c = cs[k][0], sn = cs[k][1];
        const double vp = vrow[row * r + p], vq = vrow[row * r + q];
        vrow[row * r + p] = c * vp - sn * vq;
        vrow[row * r + q] = sn * vp + c * vq;
      }
      __syncthreads();   // cs is rewritten by the next round
      cluster_barrier();
    }
    // stop when the off-diagonal part is at rounding level (every CTA sums all of M, in
    // the same order, so that all of a cluster's stop together)
    double off = 0.0, all = 0.0;
    for (int e = tid; e < rr; e += kJacThreads) {
      const double m = __ldcg(&M[e]);
      const double v = m * m;
      all += v;
      if (e / r != e % r) off += v;
    }
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_down_sync(0xffffffffu, off, o);
      all += __shfl_down_sync(0xffffffffu, all, o);
    }
    __syncthreads();
    if ((tid & 31) == 0) red[tid >> 5] = off;
    __syncthreads();
    double off_t = 0.0;
    for (int w = 0; w < kJacThreads / 32; ++w) off_t += red[w];
    __syncthreads();
    if ((tid & 31) == 0) red[tid >> 5] = all;
    __syncthreads();
    double all_t = 0.0;
    for (int w = 0; w < kJacThreads / 32; ++w) all_t += red[w];
    __syncthreads();
    cluster_barrier();   // M is read to the end before the next sweep writes it
    if (off_t <= 1e-30 * all_t) break;
  }
  for (int e = tid; e < nv * r; e += kJacThreads) V[(int64_t)v0 * r + e] = vrow[e];
}

__global__ void __launch_bounds__(256) ny_finish_kernel(int r, double* scratch, double* T, double* lam,
                                                        const double* nu_in, const int32_t* status) {
  __shared__ int perm[kMaxRank];
  __shared__ double diag[kMaxRank];
  const int s = blockIdx.x;
  if (status[s] != KMV_OK) return;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int rr = r * r;
  const double* W = scratch + (int64_t)s * 4 * rr;
  double* G = scratch + (int64_t)s * 4 * rr + rr;
  const double* M = G + rr;
  const double* V = M + rr;
  const double nu = nu_in[s];
  for (int k = tid; k < r; k += nt) diag[k] = M[k * r + k];
  __syncthreads();
  // eigenvalues in descending order
  if (tid == 0) {
    for (int k = 0; k < r; ++k) perm[k] = k;
    for (int a = 0; a < r; ++a) {
      int best = a;
      for (int k = a + 1; k < r; ++k)
        if (diag[perm[k]] > diag[perm[best]]) best = k;
      const int u = perm[a];
      perm[a] = perm[best];
      perm[best] = u;
    }
  }
  __syncthreads();
  // T[:, j] = L^{-T} V[:, perm_j] / sqrt(s2_j) (back substitution per column)
  for (int j = tid; j < r; j += nt) {
    const int pj = perm[j];
    const double s2 = diag[pj];
    lam[(int64_t)s * r + j] = fmax(s2 - nu, 0.0);
    double* t = G + j;   // column j of G as scratch (X is no longer needed), stride r
    for (int i = r - 1; i >= 0; --i) {
      double v = V[i * r + pj];
      for (int p = i + 1; p < r; ++p) v -= W[p * r + i] * t[p * r];
      t[i * r] = v / W[i * r + i];
    }
    const double inv = s2 > 0.0 ? 1.0 / sqrt(s2) : 0.0;
    for (int i = 0; i < r; ++i) T[(int64_t)s * rr + i * r + j] = t[i * r] * inv;
  }
}

// U[c, j, i] = sum_l (Y[i, l] + nu_s Omega[i, l]) T_s[l, j] in FP64 (T's columns
// are scaled by 1/S, so the sum cancels), 16 columns j per CTA.
constexpr int kUB = 16;
__global__ void __launch_bounds__(kTile) ny_u_kernel(DevLayout L, int chains, int64_t n_total, int r,
                                                     const float* Om, const float* Y, const double* T,
                                                     const double* nu, float* U) {
  extern __shared__ double tcol[];   // r x 16 block of T
  const int item = blockIdx.x, c = blockIdx.y, jb = blockIdx.z;
  const int b = L.item_inst[item];
  const int s = b * chains + c;
  const double* Ts = T + (int64_t)s * r * r;
  for (int e = threadIdx.x; e < r * kUB; e += blockDim.x) {
    const int l = e / kUB, j = jb * kUB + e % kUB;
    tcol[e] = j < r ? Ts[l * r + j] : 0.0;
  }
  __syncthreads();
  const int64_t i = L.item_row0[item] + threadIdx.x;
  if (i >= L.offsets[b + 1]) return;
  const double nus = nu[s];
  const int64_t base = ((int64_t)c * n_total + i) * r;
  double acc[kUB];
#pragma unroll
  for (int j = 0; j < kUB; ++j) acc[j] = 0.0;
  for (int l = 0; l < r; ++l) {
    const double y = fma(nus, (double)Om[base + l], (double)Y[base + l]);
#pragma unroll
    for (int j = 0; j < kUB; ++j) acc[j] = fma(y, tcol[l * kUB + j], acc[j]);
  }
  for (int j = 0; j < kUB; ++j) {
    const int jj = jb * kUB + j;
    if (jj < r) U[((int64_t)c * r + jj) * n_total + i] = (float)acc[j];
  }
}

}  // namespace

cudaError_t launch_nystrom_finish(const DevLayout& L, int n_items, int n_inst, int chains, int64_t n_total, int r,
                                  const float* Om, const float* Y, double* grams, double* scratch, double* T,
                                  double* nu, float* U, double* lam, int32_t* status, int num_sms, cudaStream_t st) {
  const int n_sys = n_inst * chains;
  if (n_sys == 0) return cudaSuccess;
  const int nb = (r + kGB - 1) / kGB, nu_b = (r + kUB - 1) / kUB;
  ny_gram_kernel<<<dim3(n_sys, nb * nb + nb * (nb + 1)), 256, 0, st>>>(L, chains, n_total, r, nb, Om, Y, grams);
  ny_factor_kernel<<<n_sys, 256, 0, st>>>(L, chains, r, grams, scratch, T, lam, nu, status);
  // CTAs per system: as many as leave one per SM over all systems, at most 8
  int cl = 8;
  while (cl > 1 && (int64_t)n_sys * cl > num_sms) cl /= 2;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)n_sys * cl);
  cfg.blockDim = dim3(kJacThreads);
  cfg.dynamicSmemBytes = sizeof(double) * (size_t)((r + cl - 1) / cl) * r;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = cl;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaError_t e = cudaFuncSetAttribute(ny_jacobi_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)(sizeof(double) * kMaxRank * kMaxRank));
  if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, ny_jacobi_kernel, r, cl, scratch, (const int32_t*)status);
  if (e != cudaSuccess) return e;
  ny_finish_kernel<<<n_sys, 256, 0, st>>>(r, scratch, T, lam, nu, status);
  if (n_items > 0)
    ny_u_kernel<<<dim3(n_items, chains, nu_b), kTile, sizeof(double) * r * kUB, st>>>(L, chains, n_total, r, Om, Y,
                                                                                      T, nu, U);
  return cudaGetLastError();
}

}  // namespace kmv

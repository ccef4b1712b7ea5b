// Plain FP32 adjoint of L = sum G o (A V) on the FMA/MUFU pipes: the kernel.
//
// Same tiling as the forward kernel (kmv_simt_fwd.cuh): a CTA owns R * kTile rows i
// of one system, one chunk of at most MP columns and one range of columns j.  Per
// pair it recomputes K0_ij from direct differences and forms
//   W_ij = G_i . V_j             (this column chunk's share of (G V^T)_ij)
//   Q_ij = W_ij K0_ij
// and accumulates per row
//   sum_j Q_ij                                   -> d/dlog alpha
//   sum_j Q_ij (xh_ik - xh_jk)^2 (per k, or r^2) -> d/dlog l_k
//   sum_j K0_ij G_j                              -> dL/dV = A G
// With per-point amplitudes (Sec. 4) G and V enter as amp o G, amp o V.
// Because every dA/dtheta_p is symmetric, summing W_ij over all ordered
// pairs (i, j) gives the gradient without symmetrising W.  FP32 sums run over at
// most 512 columns and are then folded into FP64 sums; per-CTA FP64
// partials go to a buffer that launch_grad_finalize reduces in a fixed order.
//
// What bounds it: per pair 4 D + 2 m + 3 operations of the FMA pipe (m columns with
// dL/dV), one ex2, and the D + 2 m values of j that all lanes of a warp share (one
// clock of shared memory each per warp, so R rows per thread divide them by R).  One
// row per thread, one CTA per 128 rows and the whole J range took 4.38 ms at
// N = 20,000, d = 8, m = 16 (157 CTAs: one per SM) and 84 us at N = 2048, d = 1,
// m = 2 (16 CTAs); J units of 512 columns and R = 2 or 4 where rows are many give
// the figures at simt_bwd_plan.
#pragma once

#include "f32x2.cuh"
#include "simt_common.cuh"

namespace kmv {

constexpr int kXSB = kJT + 4;   // row stride of the staged x (floats)

template <int D, int MP, int R, bool ARD>
__global__ void __launch_bounds__(kTile) bwd_simt_kernel(KmvArgs a, SimtBwd f) {
  constexpr int DG = ARD ? D : 1;
  chain_trigger();
  chain_wait();
  const int dd = a.d;   // <= D; the dimensions past it are zero and add nothing
  const int tile = blockIdx.x, c = blockIdx.y, u = blockIdx.z % f.units, z = blockIdx.z / f.units;
  const int item0 = f.tile_item ? f.tile_item[tile] : tile;
  const int b = a.L.item_inst[item0];
  const int s = b * a.chains + c;
  if (a.sys_active && !a.sys_active[s]) return;
  const int64_t o0 = a.L.offsets[b], o1 = a.L.offsets[b + 1];
  const int64_t len = (int64_t)f.folds * kFoldTiles * kTile;
  const int64_t jb = o0 + u * len, je = min(o1, jb + len);
  if (je <= jb) return;

  // V by column (pairs of points for W), G by point (pairs of columns for dL/dV)
  __shared__ __align__(16) float sx[D * kXSB];
  __shared__ __align__(16) float sv[MP * kXSB];
  __shared__ __align__(16) float sg[kJT * MP];
  __shared__ float sc[D];
  __shared__ double as2[2];
  __shared__ double red[kTile / 32 * (2 + DG)];

  const int tid = threadIdx.x;
  const double* th = a.theta + (int64_t)s * a.n_theta;
  load_scale(th, dd, a.ard, sc);
  const bool want_gv = a.Y != nullptr;
  if (want_gv && tid >= 64 && tid < 66) as2[tid - 64] = exp(th[tid == 64 ? 0 : a.n_theta - 1]);
  if (dd < D)
    for (int e = tid; e < (D - dd) * kXSB; e += kTile) sx[dd * kXSB + e] = 0.f;
  const int c0 = z * f.chunk;
  const int mc = min(f.chunk, a.m - c0);
  const int64_t vbase = (int64_t)c * a.n_total;
  const int64_t r0 = a.L.item_row0[item0];
  __syncthreads();

  float xi[R][D], gi[R][MP], accq[R], accg[R][DG];
  uint64_t accv[R][MP / 2];   // columns 2q, 2q + 1 in a packed pair
  auto accv_at = [&](int r, int q) { return (q & 1) ? hi_f32x2(accv[r][q / 2]) : lo_f32x2(accv[r][q / 2]); };
  // running sums of the unit; those of many dimensions in local memory (64 FP64 sums are
  // 128 registers, used once in 512 columns), by a pointer hidden from the compiler, which
  // would put the array into registers and spill the loop's values
  constexpr bool kLocalG = R * DG >= 32;
  double sq[R], sg2[kLocalG ? 1 : R][kLocalG ? 1 : DG], sg_store[kLocalG ? R * DG : 1];
  double* sgl = sg_store;
  if constexpr (kLocalG) asm volatile("" : "+l"(sgl));
  bool first_g = true;
  // those of dL/dV: in registers with one row per thread and few dimensions, else in
  // local memory likewise
  constexpr bool kRegV = R == 1 && D < 32;
  constexpr int RV = kRegV ? MP : 1;
  double svp[RV];
#pragma unroll
  for (int q = 0; q < RV; ++q) svp[q] = 0.0;
  double gv_store[kRegV ? 1 : R * MP];
  double* gv = gv_store;
  asm volatile("" : "+l"(gv));
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t i = r0 + r * kTile + tid;
    const bool valid = i < o1;
    const float amp_i = (a.amp && valid) ? a.amp[vbase + i] : 1.f;
#pragma unroll
    for (int k = 0; k < D; ++k) xi[r][k] = (k < dd && valid) ? a.x[i * dd + k] * sc[k] : 0.f;
#pragma unroll
    for (int q = 0; q < MP; ++q) {
      gi[r][q] = (q < mc && valid) ? a.G[(vbase + i) * a.m + c0 + q] * amp_i : 0.f;
      accv[r][q / 2] = 0;
    }
    accq[r] = 0.f;
    sq[r] = 0.0;
#pragma unroll
    for (int k = 0; k < DG; ++k) {
      accg[r][k] = 0.f;
      if constexpr (!kLocalG) sg2[r][k] = 0.0;
    }
  }

  const uint32_t inv = dd > 1 ? 0xffffffffu / (uint32_t)dd + 1u : 0u;
  const bool several = je - jb > kFoldTiles * kTile;
  bool first = true;
  // adds the FP32 sums of dL/dV of this thread's rows to the FP64 ones
  auto fold_v = [&]() {
    if constexpr (kRegV) {
#pragma unroll
      for (int q = 0; q < RV; ++q) svp[q] += (double)accv_at(0, q);
#pragma unroll
      for (int q = 0; q < MP / 2; ++q) accv[0][q] = 0;
    } else {
#pragma unroll
      for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int q = 0; q < MP; ++q) {
          const double v = (double)accv_at(r, q);
          gv[r * MP + q] = first ? v : gv[r * MP + q] + v;
        }
#pragma unroll
        for (int q = 0; q < MP / 2; ++q) accv[r][q] = 0;
      }
      first = false;
    }
  };
  auto fold_g = [&]() {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      sq[r] += (double)accq[r];
      accq[r] = 0.f;
#pragma unroll
      for (int k = 0; k < DG; ++k) {
        if constexpr (kLocalG) {
          if (k < dd) {   // (the FP64 pipe is slow)
            const double v = (double)accg[r][k];
            sgl[r * DG + k] = first_g ? v : sgl[r * DG + k] + v;
          }
        } else {
          if (k < dd) sg2[r][k] += (double)accg[r][k];
        }
        accg[r][k] = 0.f;
      }
    }
    first_g = false;
  };

  int step = 0;
  for (int64_t jt = jb; jt < je; jt += kJT, ++step) {
    const int nj = (int)min((int64_t)kJT, je - jt);
    for (int e = tid; e < kJT * dd; e += kTile) {
      const int r = dd > 1 ? (int)__umulhi((uint32_t)e, inv) : e, k = e - r * dd;
      sx[k * kXSB + r] = r < nj ? a.x[jt * dd + e] * sc[k] : 0.f;
    }
    for (int e = tid; e < kJT * MP; e += kTile) {
      const int r = e / MP, q = e - r * MP;
      const bool in = r < nj && q < mc;
      const int64_t idx = (vbase + jt + r) * a.m + c0 + q;
      const float am = (in && a.amp) ? a.amp[vbase + jt + r] : 1.f;
      sv[q * kXSB + r] = in ? a.V[idx] * am : 0.f;
      sg[e] = (in && want_gv) ? a.G[idx] * am : 0.f;
    }
    __syncthreads();
    // two points j at a time (their chains interleave), all R rows; one row per thread
    // has eight in flight where registers allow
#pragma unroll (R == 1 && D * MP <= 32 ? 4 : 1)
    for (int jj = 0; jj < kJT; jj += 2) {
      uint64_t r2[R], df2[R][DG];
#pragma unroll
      for (int r = 0; r < R; ++r) r2[r] = 0;
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const uint64_t x2 = *reinterpret_cast<const uint64_t*>(sx + k * kXSB + jj);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const uint64_t df = sub_f32x2(pack_f32x2(xi[r][k], xi[r][k]), x2);
          if (ARD) {
            const uint64_t q2 = mul_f32x2(df, df);
            df2[r][ARD ? k : 0] = q2;
            r2[r] = add_f32x2(r2[r], q2);
          } else {
            r2[r] = fma_f32x2(df, df, r2[r]);
          }
        }
      }
      uint64_t w[R];
#pragma unroll
      for (int r = 0; r < R; ++r) w[r] = 0;
#pragma unroll
      for (int q = 0; q < MP; ++q) {
        const uint64_t v2 = *reinterpret_cast<const uint64_t*>(sv + q * kXSB + jj);
#pragma unroll
        for (int r = 0; r < R; ++r) w[r] = fma_f32x2(pack_f32x2(gi[r][q], gi[r][q]), v2, w[r]);
      }
      float p[R][2];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        p[r][0] = ex2_approx(-lo_f32x2(r2[r]));
        p[r][1] = ex2_approx(-hi_f32x2(r2[r]));
        const uint64_t Q2 = mul_f32x2(w[r], pack_f32x2(p[r][0], p[r][1]));
        const float Q0 = lo_f32x2(Q2), Q1 = hi_f32x2(Q2);
        accq[r] = __fadd_rn(__fadd_rn(accq[r], Q0), Q1);
        if (ARD) {
#pragma unroll
          for (int k = 0; k < DG; ++k) {
            accg[r][k] = __fmaf_rn(Q0, lo_f32x2(df2[r][k]), accg[r][k]);
            accg[r][k] = __fmaf_rn(Q1, hi_f32x2(df2[r][k]), accg[r][k]);
          }
        } else {
          accg[r][0] = __fmaf_rn(Q0, lo_f32x2(r2[r]), accg[r][0]);
          accg[r][0] = __fmaf_rn(Q1, hi_f32x2(r2[r]), accg[r][0]);
        }
      }
      if (want_gv) {
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          const float* gj = sg + (jj + t) * MP;
          uint64_t pp[R];
#pragma unroll
          for (int r = 0; r < R; ++r) pp[r] = pack_f32x2(p[r][t], p[r][t]);
          if constexpr (MP == 2) {
            const uint64_t v2 = *reinterpret_cast<const uint64_t*>(gj);
#pragma unroll
            for (int r = 0; r < R; ++r) accv[r][0] = fma_f32x2(pp[r], v2, accv[r][0]);
          } else {
#pragma unroll
            for (int q = 0; q < MP / 2; q += 2) {
              const ulonglong2 v2 = *reinterpret_cast<const ulonglong2*>(gj + 2 * q);
#pragma unroll
              for (int r = 0; r < R; ++r) {
                accv[r][q] = fma_f32x2(pp[r], v2.x, accv[r][q]);
                accv[r][(q + 1) % (MP / 2)] = fma_f32x2(pp[r], v2.y, accv[r][(q + 1) % (MP / 2)]);
              }
            }
          }
        }
      }
    }
    __syncthreads();
    if (several && jt + kJT < je && (step + 1) % (kFoldTiles * kTile / kJT) == 0) {
      fold_g();
      if (want_gv) fold_v();
    }
  }
  fold_g();
  const bool direct = f.units == 1;
  // the FP64 sum of an element of dL/dV with the last FP32 sum added
  auto gv_total = [&](int r, int q) {
    const double v = (double)accv_at(r, q);
    if constexpr (kRegV) return svp[q % RV] + v;
    else return first ? v : gv[r * MP + q] + v;
  };
  if (want_gv && !direct) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int64_t i = r0 + r * kTile + tid;
      if (i < o1) {
#pragma unroll
        for (int q = 0; q < MP; ++q)
          if (q < mc) f.part[(((size_t)u * a.chains + c) * a.m + c0 + q) * (size_t)a.n_total + i] = gv_total(r, q);
      }
    }
  }

  // noise gradient and, in a single unit, dL/dV
  double noise = 0.0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t i = r0 + r * kTile + tid;
    if (i < o1 && (u == 0 || (want_gv && direct))) {
      const double ai = want_gv ? as2[0] * (double)(a.amp ? a.amp[vbase + i] : 1.f) : 0.0;
#pragma unroll
      for (int q = 0; q < MP; ++q) {
        if (q < mc) {
          const int64_t idx = (vbase + i) * a.m + c0 + q;
          const double g = (double)a.G[idx];
          if (u == 0) noise += g * (double)a.V[idx];
          if (want_gv && direct) a.Y[idx] = (float)(ai * gv_total(r, q) + as2[1] * g);
        }
      }
    }
  }
  // Per-CTA partials: [sum Q, sum Q d2 (k entries or 1), sum G.V]
  double* out = a.grad_partial + ((((int64_t)item0 * a.chains + c) * f.nz + z) * f.units + u) * a.n_theta;
  constexpr int NE = 2 + DG;
  double ev[NE];   // [q, g_0 .. , noise]
  ev[0] = 0.0;
#pragma unroll
  for (int r = 0; r < R; ++r) ev[0] += sq[r];
#pragma unroll
  for (int k = 0; k < DG; ++k) {
    ev[1 + k] = 0.0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if constexpr (kLocalG) ev[1 + k] += k < dd ? sgl[r * DG + k] : 0.0;
      else ev[1 + k] += sg2[r][k];
    }
  }
  ev[NE - 1] = noise;
  block_sum_many<NE>(ev, NE, red, [&](int e, double t) {
    // the dimensions past d are not written
    if (e == NE - 1) out[a.n_theta - 1] = t;
    else if (e < a.n_theta - 1) out[e] = t;
  });
}

// Rows per thread of the wide variant: R (2 D + 2 MP + D) registers and more.
constexpr int bwd_rows(int D, int MP) { return D <= 4 && MP <= 4 ? 4 : D + MP <= 32 ? 2 : 1; }

template <int D, int MP, bool ARD>
cudaError_t bwd_launch_mp(const KmvArgs& a, const SimtBwd& f, dim3 grid, cudaStream_t st) {
  if (f.rows == 1) {
    return launch_chained(a.chained, bwd_simt_kernel<D, MP, 1, ARD>, grid, kTile, 0, st, a, f);
  }
  constexpr int R = bwd_rows(D, MP);
  if constexpr (R > 1)
    if (f.rows == R) return launch_chained(a.chained, bwd_simt_kernel<D, MP, R, ARD>, grid, kTile, 0, st, a, f);
  return cudaErrorInvalidValue;
}

// The kernel for the dimension class D (kmv_simt_bwd_*.cu hold the instances).
template <int D, bool ARD>
cudaError_t bwd_launch_d(const KmvArgs& a, const SimtBwd& f, dim3 grid, cudaStream_t st) {
  switch (f.mp) {
    case 2: return bwd_launch_mp<D, 2, ARD>(a, f, grid, st);
    case 4: return bwd_launch_mp<D, 4, ARD>(a, f, grid, st);
    case 8: return bwd_launch_mp<D, 8, ARD>(a, f, grid, st);
    case 16: return bwd_launch_mp<D, 16, ARD>(a, f, grid, st);
    default: return bwd_launch_mp<D, 32, ARD>(a, f, grid, st);
  }
}

}  // namespace kmv

// Per-system CG steps shared by the CG kernels (kmv_cg.cu, kmv_pcg.cu, kmv_mscg.cu) and
// the products' epilogues when they carry the p.q step of a CG iteration (kmv_tc.cu,
// kmv_simt_fwd.cuh): every path takes the same steps from the same FP64 partials.  The
// partials of a system are summed in a fixed order, which differs between the fused
// paths (by the whole block that arrives last, sys_sum_block) and the separate kernels
// (by one thread, sys_sum), so these agree to the sums' rounding and not in every bit.
#pragma once

#include "kmv_internal.cuh"
#include "simt_common.cuh"

namespace kmv {

// Sum of a system's per-item partials in item order (fixed order: bitwise
// reproducible), by one thread: a serial chain of dependent FP64 adds.
__device__ __forceinline__ double sys_sum(const DevLayout& L, int b, int c, int chains,
                                          const double* partial, int stride, int k) {
  double acc = 0.0;
  for (int it = L.inst_item0[b]; it < L.inst_item0[b + 1]; ++it)
    acc += partial[((int64_t)it * chains + c) * stride + k];
  return acc;
}

// The same sum by a whole block (all threads call; the result is valid in
// thread 0): a strided share per thread, then block_sum, the same order on every
// run with the same block size.  One thread's chain over 128 items measured
// 13 us of the 18 us of the CG vector update at N = 16,384 (8 chains).  The loads
// bypass L1: other CTAs of this launch wrote the partials.
__device__ __forceinline__ double sys_sum_block(const DevLayout& L, int b, int c, int chains, const double* partial,
                                                int stride, int k, double* red) {
  double acc = 0.0;
  for (int it = L.inst_item0[b] + (int)threadIdx.x; it < L.inst_item0[b + 1]; it += (int)blockDim.x)
    acc += __ldcg(&partial[((int64_t)it * chains + c) * stride + k]);
  return block_sum(acc, red);
}

// alpha = r.r / p.q of one system; false when the system stops here (a
// non-finite p.q, or a breakdown: the operator is not positive definite along
// p, which a perturbed operator can be; the current iterate is kept).
__device__ __forceinline__ bool cg_pq_step(CgSys& S, double pq) {
  S.pq = pq;
  if (!isfinite(pq)) {
    S.status = KMV_ENONFINITE;
    S.alpha = 0.0;
    return false;
  }
  if (!(pq > 0.0)) {
    S.status = KMV_ENOTCONV;
    S.alpha = 0.0;
    return false;
  }
  S.alpha = S.rr / pq;
  return true;
}

// The new r.r of one system: beta, the iteration count and the stopping
// tests (converged at rr <= tol^2 b.b, or out of iterations); false when the
// system stops.
__device__ __forceinline__ bool cg_rr_step(CgSys& S, double rr, double tol, int maxiter) {
  bool active = true;
  S.iters += 1;
  if (!isfinite(rr)) {
    S.status = KMV_ENONFINITE;
    active = false;
  } else if (rr <= tol * tol * S.bb) {
    active = false;
  } else if (S.iters >= maxiter) {
    S.status = KMV_ENOTCONV;
    active = false;
  }
  S.beta = rr / S.rr;
  S.rr = rr;
  return active;
}

// Multi-shift CG (kmv_mscg.cu, whose header gives the recurrences): alpha of
// the base system and, per active shift j, zeta_j' and alpha_j, by one full warp,
// lane j for shift j (m <= 32 = kMaxShifts): an FP64 division takes some 600 clocks
// on this GPU, and the shifts' are independent (one thread for 15 shifts took most
// of the 22 us of this step's CTA at N = 4096).  false (every lane) when the base
// recurrence breaks down (p.Bp not positive or not finite), which stops every shift
// still running.
__device__ __forceinline__ bool mscg_alpha_step(MscgSys& y, MscgShift* sh, int m, double pq) {
  const int lane = threadIdx.x & 31;
  MscgShift& k = sh[lane < m ? lane : 0];
  const bool on = lane < m && k.active;
  if (!(pq > 0.0) || !isfinite(pq)) {
    if (on) {
      k.active = 0;
      k.status = isfinite(pq) ? KMV_ENOTCONV : KMV_ENONFINITE;
    }
    return false;
  }
  const double alpha = y.rr / pq;
  if (lane < m && !on) k.alpha_s = 0.0;
  if (on) {
    const double den = alpha * y.beta_prev * (k.zeta_prev - k.zeta) +
                       k.zeta_prev * y.alpha_prev * (1.0 + k.sigma * alpha);
    const double zn = k.zeta * k.zeta_prev * y.alpha_prev / den;
    if (!isfinite(zn) || k.zeta == 0.0) {
      k.active = 0;
      k.status = KMV_ENONFINITE;
      k.alpha_s = 0.0;
    } else {
      k.zeta_next = zn;
      k.alpha_s = alpha * zn / k.zeta;
    }
  }
  __syncwarp();
  if (lane == 0) y.alpha = alpha;
  return true;
}

// Multi-shift CG: beta of the base system from the new r.r, and per active
// shift the stopping test (|zeta_j'|^2 r.r <= tol^2 b.b, or out of
// iterations), beta_j and the advance of zeta, by one full warp as above.  false
// (every lane) when no shift is left.
__device__ __forceinline__ bool mscg_beta_step(MscgSys& y, MscgShift* sh, int m, double rr, double tol,
                                               int maxiter) {
  const int lane = threadIdx.x & 31;
  MscgShift& k = sh[lane < m ? lane : 0];
  const double beta = rr / y.rr;
  const double lim = tol * tol * y.bb;
  int left = 0;
  if (lane < m && k.active) {
    k.iters += 1;
    const double ratio = k.zeta_next / k.zeta;
    const double res2 = k.zeta_next * k.zeta_next * rr;
    if (!isfinite(res2) || !isfinite(beta)) {
      k.active = 0;
      k.status = KMV_ENONFINITE;
    } else if (res2 <= lim) {
      k.active = 0;
    } else if (k.iters >= maxiter) {
      k.active = 0;
      k.status = KMV_ENOTCONV;
    } else {
      k.beta_s = beta * ratio * ratio;
      k.zeta_prev = k.zeta;
      k.zeta = k.zeta_next;
    }
    left = k.active;
  }
  const int any = __any_sync(0xffffffffu, left);
  if (lane == 0) {
    y.iters += 1;
    y.rr = rr;
    y.beta = beta;
    y.alpha_prev = y.alpha;
    y.beta_prev = beta;
  }
  return any != 0;
}

// Called by thread 0 of each CTA that has written `n` of a system's `total`
// partials, after a block barrier behind the writes: true for the CTA that completes
// the system, which then sees every partial of it (and whatever the other CTAs wrote
// and read before their barriers).  One acquire-release atomic: a fence on either side
// of a relaxed one cost 700 clocks each.  Resets the counter for the next use.
__device__ __forceinline__ bool last_arrival(uint32_t* count, uint32_t n, uint32_t total) {
  uint32_t old;
  asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(count), "r"(n) : "memory");
  const bool last = old + n == total;
  if (last) *count = 0;
  return last;
}

// p = r + beta p over [v0, v1) by one CTA, eight rows of loads in flight per thread
// (r bypasses L1: other CTAs of this launch wrote it).
__device__ __forceinline__ void form_direction(float* p, const float* r, float beta, int64_t v0, int64_t v1) {
  for (int64_t v = v0 + threadIdx.x; v < v1; v += 8 * kTile) {
    float rv[8], pv[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const bool in = v + k * kTile < v1;
      rv[k] = in ? __ldcg(&r[v + k * kTile]) : 0.f;
      pv[k] = in ? p[v + k * kTile] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (v + k * kTile < v1) p[v + k * kTile] = fmaf(beta, pv[k], rv[k]);
  }
}

// alpha = r.z / p.q of one preconditioned system; false when it stops here.
__device__ __forceinline__ bool pcg_pq_step(PcgSys& y, double pq) {
  if (!(pq > 0.0) || !isfinite(pq) || !(y.rz > 0.0)) {
    y.status = isfinite(pq) && isfinite(y.rz) ? KMV_ENOTCONV : KMV_ENONFINITE;
    y.alpha = 0.0;
    return false;
  }
  y.alpha = y.rz / pq;
  return true;
}

// beta = r.z' / r.z and the stopping test on r.r of one preconditioned system.
__device__ __forceinline__ bool pcg_rz_step(PcgSys& y, double rr, double rz, double tol, int maxiter) {
  y.iters += 1;
  y.beta = rz / y.rz;
  y.rr = rr;
  y.rz = rz;
  if (!isfinite(rr) || !isfinite(rz)) {
    y.status = KMV_ENONFINITE;
    return false;
  }
  if (rr <= tol * tol * y.bb) return false;
  if (y.iters >= maxiter) {
    y.status = KMV_ENOTCONV;
    return false;
  }
  return true;
}

// The p.q (alpha) step of system s inside a (multi-shift) CG iteration, by the
// whole CTA that completed the system's dot partials.
__device__ __forceinline__ void cg_finish_pq(const DevLayout& L, const KmvArgs& a, int b, int c, int s, double* red) {
  double pq = sys_sum_block(L, b, c, a.chains, a.dot_partial, 1, 0, red);
  if (threadIdx.x >= 32) return;
  pq = __shfl_sync(0xffffffffu, pq, 0);
  bool go;
  if (a.cg_sys || a.pcg_sys) {
    if (threadIdx.x != 0) return;
    go = a.cg_sys ? cg_pq_step(a.cg_sys[s], pq) : pcg_pq_step(a.pcg_sys[s], pq);
  } else {
    go = mscg_alpha_step(a.ms_sys[s], a.ms_sh + (int64_t)s * a.ms_m, a.ms_m, pq);
  }
  if (threadIdx.x == 0 && !go) {
    a.cg_active[s] = 0;
    atomicSub(a.cg_n_active, 1);
  }
}

}  // namespace kmv

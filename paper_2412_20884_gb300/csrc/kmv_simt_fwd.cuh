// Plain FP32 forward product Y = A(theta) V on the FMA/MUFU pipes: the kernel.
//
// A CTA of kTile threads owns R * kTile rows i of one (instance, chain) system
// (thread t the rows t, t + 128, ..), one chunk of at most MP columns of V and one
// range of columns j.  It streams the points j through shared memory kJT at a time
// and, per pair, evaluates
//   K0_ij = 2^(-sum_k (xh_ik - xh_jk)^2),  xh = x sqrt(log2(e)/2) / l,
// from direct differences (no |x|^2 expansion, so no cancellation), then
// accumulates K0_ij V_j in FP32.  Every 512 columns the FP32 sums are folded into
// FP64 sums.  Epilogue (Eq. kerdef): Y_i = alpha * acc_i +
// (sigma^2 + shift) V_i.  With per-point amplitudes (the kernel family of Sec. 4)
// V_j enters as amp_j V_j and acc_i is scaled by amp_i.
//
// What bounds it: per pair 2 D + m operations of the FMA pipe (128 lanes per clock
// and SM), one ex2 (32 per clock), and a load of the D + m values of j that every
// lane of a warp shares.  Such a broadcast still returns 128 bytes per clock and SM,
// so with one row per thread the loads alone took D + m clocks per 32 pairs against
// (2 D + m) / 4 for the arithmetic; R = 4 rows per thread divide them by four, and
// the loads are 16 bytes wide (x is staged dimension by dimension).  Distances of two
// points and sums of two columns share packed f32x2 instructions: the FMA pipe runs them
// at the same rate per value (60 packed against 114 scalar instructions per clock and
// SM), but the scalar form needed an issue slot per clock and scheduler for it alone.
// At N = 20,000, d = 8, m = 16 one row per thread and one CTA per SM took 2.18 ms;
// at N = 8192, d = 3, 8 chains, m = 1 0.274 ms (figures after the change stand at
// simt_fwd_plan).
#pragma once

#include "cg_common.cuh"
#include "f32x2.cuh"
#include "simt_common.cuh"

namespace kmv {

constexpr int kXS = kJT + 4;   // row stride of the staged x (floats): 16-byte aligned, spreads the writes over banks

// The J units of an instance of nb rows: chunks of `per` J tiles, units of `span`
// tiles within them (32-bit arithmetic: a 64-bit division takes some 490 clocks).
struct SimtUnits {
  uint32_t n_jt, per, span, n_chunks;
  __device__ __forceinline__ SimtUnits(const SimtFwd& f, int64_t nb) {
    n_jt = (uint32_t)((nb + kJT - 1) / kJT);
    per = f.js > 1 ? (n_jt + f.js - 1) / f.js : n_jt;
    span = (uint32_t)f.folds * (kFoldTiles * kTile / kJT);
    n_chunks = f.js > 1 ? (n_jt + per - 1) / per : 1;
  }
  // first J tile and end of unit u of chunk jc; empty when not less
  __device__ __forceinline__ void range(uint32_t jc, uint32_t u, uint32_t& t0, uint32_t& t1) const {
    t0 = jc * per + u * span;
    t1 = min(min(n_jt, (jc + 1) * per), t0 + span);
  }
  __device__ __forceinline__ uint32_t in_chunk(uint32_t jc) const {
    return (min(n_jt, (jc + 1) * per) - jc * per + span - 1) / span;
  }
  __device__ __forceinline__ uint32_t count() const { return (n_chunks - 1) * in_chunk(0) + in_chunk(n_chunks - 1); }
};
__device__ __forceinline__ size_t simt_part_at(const KmvArgs& a, int unit, int c, int col, int64_t i) {
  return (((size_t)unit * a.chains + c) * a.m + col) * (size_t)a.n_total + i;
}

// Adds n sums a fixed step apart to s, eight loads in flight at a time (one after the
// other, 16 of them took 5 us of a small product's last CTA).
__device__ __forceinline__ void simt_add_parts(const double* p, size_t step, uint32_t n, double& s) {
  for (uint32_t u0 = 0; u0 < n; u0 += 8) {
    double v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = u0 + k < n ? __ldcg(p + (u0 + k) * step) : 0.0;
    if (u0 + 8 <= n) {
      // (a tree: 16 dependent FP64 adds of 65 clocks were 0.4 us of a small product)
      s += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    } else {
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (u0 + k < n) s += v[k];
    }
  }
}

// Sum of the units' sums of one element, in a fixed order.
__device__ __forceinline__ double simt_part_sum(const KmvArgs& a, const SimtFwd& f, const SimtUnits& U, int c, int col,
                                                int64_t i) {
  double s = 0.0;
  const size_t step = (size_t)a.chains * a.m * (size_t)a.n_total;
  const double* p = f.part + simt_part_at(a, 0, c, col, i);
  // one run of units, or a run per chunk where this instance's chunks have fewer than upc
  // (upc == 1 without the divisions)
  const bool one_run = f.upc == 1 || U.in_chunk(0) == (uint32_t)f.upc;
  const uint32_t runs = one_run ? 1 : U.n_chunks;
  for (uint32_t jc = 0; jc < runs; ++jc)
    simt_add_parts(p + jc * f.upc * step, step, f.upc == 1 ? U.n_chunks : one_run ? U.count() : U.in_chunk(jc), s);
  return s;
}

// The same for units of one fold, which a product by ticket stores as the FP32 sums that
// they are.  The FP64 pipe gives 2 lanes per clock and SM: 16 FP64 adds of 128 rows in a
// small product's last CTA took 1.3 of its 8.7 us.  Here every addition's rounding error is
// kept, and the errors' own in a third term, which is more than FP64's precision; sums
// that leave FP32's range (and infinities) are taken again in FP64.
__device__ __forceinline__ double simt_part_sum_f32(const KmvArgs& a, const SimtFwd& f, const SimtUnits& U, int c,
                                                    int col, int64_t i) {
  const size_t step = (size_t)a.chains * a.m * (size_t)a.n_total;
  const float* p = reinterpret_cast<const float*>(f.part) + simt_part_at(a, 0, c, col, i);
  const bool one_run = f.upc == 1 || U.in_chunk(0) == (uint32_t)f.upc;
  const uint32_t runs = one_run ? 1 : U.n_chunks;
  auto run_of = [&](uint32_t jc) { return f.upc == 1 ? U.n_chunks : one_run ? U.count() : U.in_chunk(jc); };
  float s = 0.f, e = 0.f, e2 = 0.f;
  for (uint32_t jc = 0; jc < runs; ++jc) {
    const uint32_t n = run_of(jc);
    for (uint32_t u0 = 0; u0 < n; u0 += 8) {
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = u0 + k < n ? __ldcg(p + (jc * f.upc + u0 + k) * step) : 0.f;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        float err = 0.f;
        two_sum_add(s, err, v[k]);
        two_sum_add(e, e2, err);
      }
    }
  }
  if (isfinite(s)) return (double)s + ((double)e + (double)e2);
  double t = 0.0;
  for (uint32_t jc = 0; jc < runs; ++jc)
    for (uint32_t u = 0, n = run_of(jc); u < n; ++u) t += (double)__ldcg(p + (jc * f.upc + u) * step);
  return t;
}

// alpha and sigma^2 of a system: two lanes, one exp (an FP64 exp takes some 1100
// clocks, and 2 lanes per clock and SM: once per CTA, not per thread).
__device__ __forceinline__ void load_alpha_s2(const KmvArgs& a, int s, double* as2) {
  if (threadIdx.x < 2) {
    const double* th = a.theta + (int64_t)s * a.n_theta;
    as2[threadIdx.x] = exp(th[threadIdx.x ? a.n_theta - 1 : 0]);
  }
}

// One element of Y from its sum and V_i; returns V_i Y_i.
__device__ __forceinline__ double simt_put_y(const KmvArgs& a, int s, int c, int64_t i, int col, double ai, double s2,
                                             double sum, float v) {
  const int64_t idx = ((int64_t)c * a.n_total + i) * a.m + col;
  const double shift = a.col_shift ? (double)a.col_shift[(int64_t)s * a.col_shift_stride + col] : 0.0;
  const double vi = (double)v;
  const double y = ai * sum + (a.no_diag ? 0.0 : (s2 + shift) * vi);
  a.Y[idx] = (float)y;
  if (a.Y64) a.Y64[idx] = y;
  return vi * y;
}

// The dot partials of `n` items starting at item0 (dots[r] of this thread's row in
// item item0 + r), and inside a CG iteration the system's p.q step by the CTA that
// completes it.
template <int R>
__device__ __forceinline__ void simt_put_dots(const KmvArgs& a, int b, int c, int s, int item0, int n,
                                              const double (&dots)[R], double* red, int* s_flag) {
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (r < n) {
      const double t = block_sum(dots[r], red);
      if (threadIdx.x == 0) a.dot_partial[(int64_t)(item0 + r) * a.chains + c] = t;
    }
  }
  if (!(a.cg_sys || a.ms_sys || a.pcg_sys)) return;
  if (threadIdx.x == 0)
    *s_flag = last_arrival(&a.cg_count[s], (uint32_t)n, (uint32_t)(a.L.inst_item0[b + 1] - a.L.inst_item0[b]));
  __syncthreads();
  if (*s_flag) cg_finish_pq(a.L, a, b, c, s, red);
}

// Least CTAs per SM asked of the compiler (0: none): at 3 and 4 dimensions it took 132 and
// 138 registers, three CTAs, for 16 columns (N = 3000, d = 3, m = 32: 47 against 31 us).
constexpr int fwd_min_ctas(int D, int MP, int R) { return R == 1 && MP == 16 && (D == 3 || D == 4) ? 4 : 0; }

__host__ __device__ constexpr int fwd_buffers(int D, int MP) { return 8 * (D * kXS + kJT * MP) <= 47 * 1024 ? 2 : 1; }

template <int D, int MP, int R>
__global__ void __launch_bounds__(kTile, fwd_min_ctas(D, MP, R)) fwd_simt_kernel(KmvArgs a, SimtFwd f) {
  chain_trigger();
  if (a.chained == 2) chain_wait();
  const int dd = a.d;   // <= D; the dimensions past it are zero and add nothing
  const int tile = blockIdx.x, c = blockIdx.y;
  const int u = blockIdx.z % f.upc, jc = (blockIdx.z / f.upc) % f.js, z = f.z0 + blockIdx.z / f.max_units;
  const int item0 = f.tile_item ? f.tile_item[tile] : tile;
  // one instance needs no look-ups (three dependent loads at the start of a small call)
  const bool single = f.n_inst == 1;
  const int b = single ? 0 : a.L.item_inst[item0];
  const int s = b * a.chains + c;
  const int64_t o0 = single ? 0 : a.L.offsets[b], o1 = single ? a.n_total : a.L.offsets[b + 1];
  const SimtUnits U(f, o1 - o0);
  uint32_t t0, t1;
  U.range(jc, u, t0, t1);
  if (t1 <= t0) return;   // an empty unit: the last ones of a short instance
  const int64_t jb = o0 + (int64_t)t0 * kJT, je = min(o1, o0 + (int64_t)t1 * kJT);

  // two buffers where they fit the 48 KB of static shared memory
  constexpr int NB = fwd_buffers(D, MP);
  __shared__ __align__(16) float sx[NB][D * kXS];
  __shared__ __align__(16) float sv[NB][kJT * MP];
  __shared__ float sc[D];
  __shared__ double as2[2];
  __shared__ double red[kTile / 32];
  __shared__ int s_flag;

  const int tid = threadIdx.x;
  const double* th = a.theta + (int64_t)s * a.n_theta;
  const int c0 = z * MP;
  const int mc = min(MP, a.m - c0);
  const int64_t vbase = (int64_t)c * a.n_total;
  const int64_t r0 = single ? (int64_t)item0 * kTile : a.L.item_row0[item0];

  float xi[R][D];
  // sums: columns 2q, 2q + 1 of a row in a packed pair (one column: plain)
  constexpr int NP = MP > 1 ? MP / 2 : 1;
  uint64_t acc[R][NP];
  auto acc_at = [&](int r, int q) { return (q & 1) ? hi_f32x2(acc[r][q / 2]) : lo_f32x2(acc[r][q / 2]); };
  // few columns: V_i for the epilogue too, loaded here so that the last CTA has it
  constexpr int PV = MP <= 2 ? MP : 1;
  float vi[R][PV];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t i = r0 + r * kTile + tid;
#pragma unroll
    for (int k = 0; k < D; ++k) xi[r][k] = (k < dd && i < o1) ? a.x[i * dd + k] : 0.f;
#pragma unroll
    for (int q = 0; q < NP; ++q) acc[r][q] = 0;
  }

  // the next J tile's points and vectors, loaded into registers while the current
  // one is worked on; e / dd by a multiplication (exact for e < 2^16)
  constexpr int NX = (kJT * D + kTile - 1) / kTile, NV = (kJT * MP + kTile - 1) / kTile;
  float fx[NX], fv[NV];
  const uint32_t inv = dd > 1 ? 0xffffffffu / (uint32_t)dd + 1u : 0u;
  auto split = [&](int e, int& r, int& k) {
    r = dd > 1 ? (int)__umulhi((uint32_t)e, inv) : e;
    k = e - r * dd;
  };
  auto fetch_x = [&](int64_t jt) {
    const int nj = (int)min((int64_t)kJT, je - jt);
#pragma unroll
    for (int n = 0; n < NX; ++n) {
      const int e = n * kTile + tid;
      fx[n] = e < nj * dd ? a.x[jt * dd + e] : 0.f;
    }
  };
  auto fetch_v = [&](int64_t jt) {
    const int nj = (int)min((int64_t)kJT, je - jt);
#pragma unroll
    for (int n = 0; n < NV; ++n) {
      const int e = n * kTile + tid, r = e / MP, q = e - r * MP;
      fv[n] = (r < nj && q < mc) ? a.V[(vbase + jt + r) * a.m + c0 + q] * (a.amp ? a.amp[vbase + jt + r] : 1.f) : 0.f;
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int n = 0; n < NX; ++n) {
      const int e = n * kTile + tid;
      if (e < kJT * dd) {
        int r, k;
        split(e, r, k);
        sx[buf][k * kXS + r] = fx[n] * sc[k];
      }
    }
#pragma unroll
    for (int n = 0; n < NV; ++n) {
      const int e = n * kTile + tid;
      if (NV * kTile == kJT * MP || e < kJT * MP) sv[buf][e] = fv[n];
    }
  };
  fetch_x(jb);
  // the scales, and by two lanes of another warp alpha and sigma^2 (read at the end),
  // while the loads above are in flight
  load_scale(th, dd, a.ard, sc);
  if ((f.max_units == 1 || f.ticket) && tid >= 96 && tid < 98) as2[tid - 96] = exp(th[tid == 96 ? 0 : a.n_theta - 1]);
  if (dd < D)
    for (int e = tid; e < (D - dd) * kXS; e += kTile) sx[0][dd * kXS + e] = sx[NB - 1][dd * kXS + e] = 0.f;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int k = 0; k < D; ++k)
      if (k < dd) xi[r][k] *= sc[k];
  // from here on, what the solver's kernels before this one write: V and the masks
  chain_wait();
  if (a.sys_active && !a.sys_active[s]) return;
  fetch_v(jb);
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int q = 0; q < PV; ++q) {
      const int64_t i = r0 + r * kTile + tid;
      vi[r][q] = (MP <= 2 && q < mc && i < o1) ? a.V[(vbase + i) * a.m + c0 + q] : 0.f;
    }

  const bool several = je - jb > kFoldTiles * kTile;   // several folds in this unit
  bool first = true;
  // The FP64 sums of several folds: in the thread's local memory, since R * MP doubles do
  // not fit beside the loop's registers and global memory for them (twice the size of V)
  // is not to be asked of a call with one unit per row.  The pointer is hidden from the
  // compiler, which would put the array into registers (N = 3000, d = 16, m = 4: 26 against
  // 20 us).  In registers for one row per thread, wide chunks and few dimensions, where
  // the loop has room for them (N = 300, d = 16, m = 32: 28 against 44 us).
  constexpr bool kInRegs = R == 1 && MP >= 16 && 2 * D <= MP;
  double run[kInRegs ? MP : 1], sums_store[kInRegs ? 1 : R * MP];
  double* sums = sums_store;
  if constexpr (kInRegs) {
#pragma unroll
    for (int q = 0; q < MP; ++q) run[q] = 0.0;
  } else {
    asm volatile("" : "+l"(sums));
  }
  // the sum of an element so far, with the FP32 sum added
  auto total = [&](int r, int q) {
    const double v = (double)acc_at(r, q);
    if constexpr (kInRegs)
      return several ? run[q] + v : v;
    else
      return first ? v : sums[r * MP + q] + v;
  };
  auto fold = [&]() {
#pragma unroll
    for (int r = 0; r < R; ++r) {
#pragma unroll
      for (int q = 0; q < MP; ++q) {
        if constexpr (kInRegs) run[q] = total(r, q);
        else sums[r * MP + q] = total(r, q);
      }
#pragma unroll
      for (int q = 0; q < NP; ++q) acc[r][q] = 0;
    }
    first = false;
  };

  store(0);
  __syncthreads();
  int step = 0;
  for (int64_t jt = jb; jt < je; jt += kJT, ++step) {
    const int buf = NB == 2 ? step & 1 : 0;
    const bool more = jt + kJT < je;
    if (more) {
      fetch_x(jt + kJT);
      fetch_v(jt + kJT);
    }
    const float* X = sx[buf];
    const float* V = sv[buf];
    // one row per thread leaves a chain of dependent steps: two steps in flight there
#pragma unroll (R == 1 && D * MP <= 64 ? 2 : 1)
    for (int jj = 0; jj < kJT; jj += 4) {
      uint64_t d01[R], d23[R];   // squared distances of the four points
#pragma unroll
      for (int r = 0; r < R; ++r) d01[r] = d23[r] = 0;
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const ulonglong2 x4 = *reinterpret_cast<const ulonglong2*>(X + k * kXS + jj);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const uint64_t xx = pack_f32x2(xi[r][k], xi[r][k]);
          const uint64_t da = sub_f32x2(xx, x4.x), db = sub_f32x2(xx, x4.y);
          d01[r] = fma_f32x2(da, da, d01[r]);
          d23[r] = fma_f32x2(db, db, d23[r]);
        }
      }
      float p[R][4];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        p[r][0] = ex2_approx(-lo_f32x2(d01[r]));
        p[r][1] = ex2_approx(-hi_f32x2(d01[r]));
        p[r][2] = ex2_approx(-lo_f32x2(d23[r]));
        p[r][3] = ex2_approx(-hi_f32x2(d23[r]));
      }
      // the vectors of the four points: 4 MP consecutive floats
      if (MP == 1) {
        const float4 v = *reinterpret_cast<const float4*>(V + jj);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          float s1 = lo_f32x2(acc[r][0]);
          s1 = fmaf(p[r][0], v.x, s1);
          s1 = fmaf(p[r][1], v.y, s1);
          s1 = fmaf(p[r][2], v.z, s1);
          s1 = fmaf(p[r][3], v.w, s1);
          acc[r][0] = pack_f32x2(s1, 0.f);
        }
      } else if (MP == 2) {
        const ulonglong2 va = *reinterpret_cast<const ulonglong2*>(V + 2 * jj);
        const ulonglong2 vb = *reinterpret_cast<const ulonglong2*>(V + 2 * jj + 4);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          acc[r][0] = fma_f32x2(pack_f32x2(p[r][0], p[r][0]), va.x, acc[r][0]);
          acc[r][0] = fma_f32x2(pack_f32x2(p[r][1], p[r][1]), va.y, acc[r][0]);
          acc[r][0] = fma_f32x2(pack_f32x2(p[r][2], p[r][2]), vb.x, acc[r][0]);
          acc[r][0] = fma_f32x2(pack_f32x2(p[r][3], p[r][3]), vb.y, acc[r][0]);
        }
      } else {
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          uint64_t pp[R];
#pragma unroll
          for (int r = 0; r < R; ++r) pp[r] = pack_f32x2(p[r][t], p[r][t]);
#pragma unroll
          for (int q = 0; q < MP; q += 4) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(V + (jj + t) * MP + q);
#pragma unroll
            for (int r = 0; r < R; ++r) {
              acc[r][(q / 2) % NP] = fma_f32x2(pp[r], v.x, acc[r][(q / 2) % NP]);
              acc[r][(q / 2 + 1) % NP] = fma_f32x2(pp[r], v.y, acc[r][(q / 2 + 1) % NP]);
            }
          }
        }
      }
    }
    if (NB == 1) __syncthreads();   // the one buffer has been read
    if (more) store(NB == 2 ? buf ^ 1 : 0);
    __syncthreads();
    if (several && more && (step + 1) % (kFoldTiles * kTile / kJT) == 0) fold();
  }

  const int n_it = min(R, a.L.inst_item0[b + 1] - item0);
  double dots[R];
  if (f.max_units == 1) {
    const double alpha = as2[0], s2 = as2[1];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      dots[r] = 0.0;
      const int64_t i = r0 + r * kTile + tid;
      if (i < o1) {
        const double ai = a.amp ? alpha * (double)a.amp[vbase + i] : alpha;
#pragma unroll
        for (int q = 0; q < MP; ++q)
          if (q < mc) {
            dots[r] += simt_put_y(a, s, c, i, c0 + q, ai, s2, total(r, q),
                                  MP <= 2 ? vi[r][q % PV] : a.V[(vbase + i) * a.m + c0 + q]);
          }
      }
    }
    if (a.dot_partial) simt_put_dots<R>(a, b, c, s, item0, n_it, dots, red, &s_flag);
    return;
  }
  const int unit = jc * f.upc + u;
  const bool f32_parts = f.ticket && f.folds == 1;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t i = r0 + r * kTile + tid;
    if (i < o1) {
#pragma unroll
      for (int q = 0; q < MP; ++q)
        if (q < mc) {
          if (MP <= 2 && f32_parts) reinterpret_cast<float*>(f.part)[simt_part_at(a, unit, c, c0 + q, i)] = acc_at(r, q);
          else f.part[simt_part_at(a, unit, c, c0 + q, i)] = total(r, q);
        }
    }
  }
  if (!f.ticket) return;
  // the tile's last unit to finish adds the units in order
  __syncthreads();
  if (tid == 0)
    s_flag = last_arrival(&f.count[((size_t)tile * a.chains + c) * f.nz + z], 1u, U.count());
  __syncthreads();
  if (!s_flag) return;
  const double alpha = as2[0], s2 = as2[1];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    dots[r] = 0.0;
    const int64_t i = r0 + r * kTile + tid;
    if (i < o1) {
      const double ai = a.amp ? alpha * (double)a.amp[vbase + i] : alpha;
#pragma unroll
      for (int q = 0; q < PV; ++q)   // (ticket: at most two columns)
        if (q < mc) dots[r] += simt_put_y(a, s, c, i, c0 + q, ai, s2,
                                            f32_parts ? simt_part_sum_f32(a, f, U, c, c0 + q, i)
                                                      : simt_part_sum(a, f, U, c, c0 + q, i),
                                            vi[r][q]);
    }
  }
  if (a.dot_partial) simt_put_dots<R>(a, b, c, s, item0, n_it, dots, red, &s_flag);
}

// Rows per thread of the wide variant (more rows cost registers: R (D + MP) and
// the probabilities of four points stay below the 255 of a thread).
constexpr int fwd_rows(int D, int MP) { return D <= 8 || (D <= 16 && MP <= 16) ? 4 : D <= 32 ? 2 : 1; }

// The widest chunk built: 32 columns where the distances cost as much as they do (one
// chunk of 64 was no faster than two of 32: 1.02 against 0.93 ms at N = 9001, d = 33,
// m = 64, and four of 16, padded to 64 dimensions, took 3.41 ms); below, two 16-column
// chunks of four rows are cheaper than one of 32 columns and two rows.
constexpr int fwd_most_columns(int D) { return D >= 16 ? 32 : 16; }

template <int D, int MP>
cudaError_t fwd_launch_mp(const KmvArgs& a, const SimtFwd& f, dim3 grid, cudaStream_t st) {
  if (f.rows == 1) {
    return launch_chained(a.chained, fwd_simt_kernel<D, MP, 1>, grid, kTile, 0, st, a, f);
  }
  constexpr int R = fwd_rows(D, MP);
  if constexpr (R > 1)
    if (f.rows == R) return launch_chained(a.chained, fwd_simt_kernel<D, MP, R>, grid, kTile, 0, st, a, f);
  return cudaErrorInvalidValue;
}

// The kernel for the dimension class D (kmv_simt_fwd_*.cu hold the instances).
template <int D>
cudaError_t fwd_launch_d(const KmvArgs& a, const SimtFwd& f, dim3 grid, cudaStream_t st) {
  switch (f.mp) {
    case 1: return fwd_launch_mp<D, 1>(a, f, grid, st);
    case 2: return fwd_launch_mp<D, 2>(a, f, grid, st);
    case 4: return fwd_launch_mp<D, 4>(a, f, grid, st);
    case 8: return fwd_launch_mp<D, 8>(a, f, grid, st);
    case 16: return fwd_launch_mp<D, 16>(a, f, grid, st);
    case 32:
      if constexpr (fwd_most_columns(D) >= 32) return fwd_launch_mp<D, 32>(a, f, grid, st);
      return cudaErrorInvalidValue;
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace kmv

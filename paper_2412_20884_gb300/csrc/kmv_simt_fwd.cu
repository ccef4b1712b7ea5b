// Plain FP32 forward product: the work split, the dispatch over dimensions and
// column widths, and the combine kernel (the product kernel is in
// kmv_simt_fwd.cuh).
#include <algorithm>

#include "kmv_simt_fwd.cuh"

namespace kmv {

extern template cudaError_t fwd_launch_d<1>(const KmvArgs&, const SimtFwd&, dim3, cudaStream_t);
extern template cudaError_t fwd_launch_d<2>(const KmvArgs&, const SimtFwd&, dim3, cudaStream_t);
extern template cudaError_t fwd_launch_d<3>(const KmvArgs&, const SimtFwd&, dim3, cudaStream_t);
extern template cudaError_t fwd_launch_d<4>(const KmvArgs&, const SimtFwd&, dim3, cudaStream_t);
extern template cudaError_t fwd_launch_d<6>(const KmvArgs&, const SimtFwd&, dim3, cudaStream_t);
extern template cudaError_t fwd_launch_d<8>(const KmvArgs&, const SimtFwd&, dim3, cudaStream_t);
extern template cudaError_t fwd_launch_d<12>(const KmvArgs&, const SimtFwd&, dim3, cudaStream_t);
extern template cudaError_t fwd_launch_d<16>(const KmvArgs&, const SimtFwd&, dim3, cudaStream_t);
extern template cudaError_t fwd_launch_d<24>(const KmvArgs&, const SimtFwd&, dim3, cudaStream_t);
extern template cudaError_t fwd_launch_d<32>(const KmvArgs&, const SimtFwd&, dim3, cudaStream_t);
extern template cudaError_t fwd_launch_d<48>(const KmvArgs&, const SimtFwd&, dim3, cudaStream_t);
extern template cudaError_t fwd_launch_d<64>(const KmvArgs&, const SimtFwd&, dim3, cudaStream_t);

// Adds the units' sums and writes Y, 128 rows and kCombineCols columns at a time.
constexpr int kCombineCols = 2;
__global__ void __launch_bounds__(kTile) fwd_simt_combine_kernel(KmvArgs a, SimtFwd f) {
  __shared__ double as2[2];
  const int item = blockIdx.x, c = blockIdx.y;
  const int b = a.L.item_inst[item];
  const int s = b * a.chains + c;
  if (a.sys_active && !a.sys_active[s]) return;
  load_alpha_s2(a, s, as2);
  const int64_t i = a.L.item_row0[item] + threadIdx.x;
  const int64_t o0 = a.L.offsets[b], o1 = a.L.offsets[b + 1];
  const bool valid = i < o1;
  const SimtUnits U(f, o1 - o0);
  __syncthreads();
  const double ai = valid && a.amp ? as2[0] * (double)a.amp[(int64_t)c * a.n_total + i] : as2[0];
  for (int c0 = blockIdx.z * kCombineCols; c0 < a.m; c0 += gridDim.z * kCombineCols) {
    const int mc = min(kCombineCols, a.m - c0);
    if (valid)
      for (int q = 0; q < mc; ++q)
        simt_put_y(a, s, c, i, c0 + q, ai, as2[1], simt_part_sum(a, f, U, c, c0 + q, i),
                   a.V[((int64_t)c * a.n_total + i) * a.m + c0 + q]);
  }
}

namespace {

constexpr int kDims[] = {1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64};
int dim_class(int d) {
  for (int v : kDims)
    if (d <= v) return v;
  return 0;
}

// Columns per CTA: the width with the least time over all chunks (above 32 dimensions
// with their number: `row_ctas` CTAs per chunk count as one wave up to two per SM, so that
// a small set is split over more CTAs: N = 1000, d = 64, m = 64 takes 54 us, 99 us with the
// widest chunk).  Per row and pair a
// chunk takes (2 D + mp + 6) / 4 clocks of the SM's FMA pipe (6: the exponential and
// the loop around it) and its R rows share (D + mp) clocks of shared-memory loads.
int fwd_width(int D, int m, double row_ctas, int num_sms) {
  int best = 1;
  double cost = -1.0;
  for (int mp = D > 32 ? std::min(16, pow2ceil(m)) : 1; mp <= fwd_most_columns(D); mp *= 2) {
    const double fma = (2.0 * D + mp + 6.0) / 4.0, lds = (double)(D + mp) / fwd_rows(D, mp);
    const double nz = (m + mp - 1) / mp;
    const double c = (D > 32 ? std::max(1.0, nz * row_ctas / (2.0 * num_sms)) : nz) * std::max(fma, lds);
    if (cost < 0.0 || c < cost) {
      cost = c;
      best = mp;
    }
  }
  return best;
}

// Chunks of whole J tiles of a small product: the FP32 sums start anew at each, so
// the count is part of the result's rounding.  1 from two CTAs (of 128 rows and
// kMaxMPFwd columns) per SM up, else about two per SM with at least two J tiles (of
// the largest instance, max_rows) per chunk.
int forward_jsplit(int n_items, int chains, int m, int64_t max_rows, int num_sms) {
  const int mp = m >= kMaxMPFwd ? kMaxMPFwd : pow2ceil(m);
  const int64_t ctas = (int64_t)n_items * chains * ((m + mp - 1) / mp);
  if (ctas <= 0 || ctas >= 2 * (int64_t)num_sms) return 1;
  int64_t js = std::min<int64_t>(kMaxJSplit, (2 * (int64_t)num_sms) / ctas);
  js = std::min<int64_t>(js, ((max_rows + kJT - 1) / kJT) / 2);
  return (int)std::max<int64_t>(1, js);
}

}  // namespace

// Rows per thread and the number of J units.  Units end at multiples of 512 columns
// of a chunk, where the FP32 sums are folded anyway, so the split changes the result
// only in the FP64 sums' last bits.
// One CTA of one-row threads per 128 rows took 2.18 ms at N = 20,000, d = 8, m = 16 (one
// to two CTAs per SM); four rows and units of 512 columns and up take 0.46 ms, with
// 0.03 ms for their sum.  The wide variant starts where its finest split fills every SM
// twice: at 2048 rows (d = 1, m = 1) its four tiles of 512 rows would leave most of the
// chip idle, and the one-row variant takes 7.7 us there against 12 us with the sum of the
// J units in a kernel of its own (now by the last CTA of a tile to arrive, up to two
// columns; with more columns that CTA's serial share costs more than a launch).
SimtFwd simt_fwd_plan(const SimtTiles& T, int n_inst, int n_items, int chains, int64_t n_total, int64_t max_rows, int d, int m,
                      int num_sms, bool one_unit) {
  SimtFwd f{};
  const int D = dim_class(d);
  f.n_inst = n_inst;
  f.js = forward_jsplit(n_items, chains, m, max_rows, num_sms);
  f.mp = fwd_width(D, m, (double)n_items * chains * f.js, num_sms);
  f.nz = (m + f.mp - 1) / f.mp;
  const int64_t n_jt = (max_rows + kJT - 1) / kJT, per = (n_jt + f.js - 1) / f.js;
  const int64_t fpc = std::max<int64_t>(1, (per * kJT + kFoldTiles * kTile - 1) / (kFoldTiles * kTile));
  const int R = fwd_rows(D, f.mp);
  const int64_t wide = (int64_t)(R == 4 ? T.n4 : R == 2 ? T.n2 : n_items) * chains * f.nz;
  // the wide variant once its finest split gives every SM two CTAs
  const bool big = R > 1 && wide * f.js * fpc >= 2 * (int64_t)num_sms;
  f.rows = big ? R : 1;
  f.tile_item = !big ? nullptr : R == 4 ? T.item4 : T.item2;
  f.n_tiles = !big ? n_items : R == 4 ? T.n4 : T.n2;
  const int64_t ctas = (int64_t)f.n_tiles * chains * f.nz * f.js;
  // about 8 CTAs per SM (two to four resident, so that the last wave is short), with at
  // most kSimtPartMax bytes of partial sums; a single unit (upc == 1 == js) needs none
  int64_t upc = std::min<int64_t>(fpc, std::max<int64_t>(1, (8 * (int64_t)num_sms + ctas - 1) / std::max<int64_t>(1, ctas)));
  const int64_t bytes = (int64_t)sizeof(double) * f.js * chains * m * std::max<int64_t>(1, n_total);
  while (upc > 1 && bytes * upc > kSimtPartMax) --upc;
  if (one_unit) upc = 1;
  f.folds = (int)((fpc + upc - 1) / upc);
  f.upc = (int)((fpc + f.folds - 1) / f.folds);
  f.max_units = f.js * f.upc;
  f.ticket = f.max_units > 1 && m <= 2;
  return f;
}

size_t simt_fwd_part_bytes(const SimtFwd& f, int chains, int64_t n_total, int m) {
  return f.max_units > 1 ? sizeof(double) * (size_t)f.max_units * chains * m * (size_t)n_total : 0;
}
size_t simt_fwd_counters(const SimtFwd& f, int chains) { return f.ticket ? (size_t)f.n_tiles * chains * f.nz : 0; }

cudaError_t launch_forward_simt(const KmvArgs& a, const SimtFwd& plan, int n_items, cudaStream_t st) {
  // the grid's z dimension (65,535) takes the column chunks in as many launches as they need
  const int z_most = std::max(1, 65535 / plan.max_units);
  for (int z0 = 0; z0 < plan.nz; z0 += z_most) {
    SimtFwd f = plan;
    f.z0 = z0;
    const dim3 grid(f.n_tiles, a.chains, std::min(z_most, f.nz - z0) * f.max_units);
    cudaError_t e = cudaErrorInvalidValue;
    switch (dim_class(a.d)) {
      case 1: e = fwd_launch_d<1>(a, f, grid, st); break;
      case 2: e = fwd_launch_d<2>(a, f, grid, st); break;
      case 3: e = fwd_launch_d<3>(a, f, grid, st); break;
      case 4: e = fwd_launch_d<4>(a, f, grid, st); break;
      case 6: e = fwd_launch_d<6>(a, f, grid, st); break;
      case 8: e = fwd_launch_d<8>(a, f, grid, st); break;
      case 12: e = fwd_launch_d<12>(a, f, grid, st); break;
      case 16: e = fwd_launch_d<16>(a, f, grid, st); break;
      case 24: e = fwd_launch_d<24>(a, f, grid, st); break;
      case 32: e = fwd_launch_d<32>(a, f, grid, st); break;
      case 48: e = fwd_launch_d<48>(a, f, grid, st); break;
      case 64: e = fwd_launch_d<64>(a, f, grid, st); break;
    }
    if (e != cudaSuccess) return e;
  }
  if (plan.max_units == 1 || plan.ticket) return cudaSuccess;
  const int gz = std::min(65535, (a.m + kCombineCols - 1) / kCombineCols);
  fwd_simt_combine_kernel<<<dim3(n_items, a.chains, gz), kTile, 0, st>>>(a, plan);
  return cudaGetLastError();
}

}  // namespace kmv

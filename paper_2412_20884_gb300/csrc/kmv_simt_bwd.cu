// Plain FP32 adjoint: the work split, the dispatch over dimensions and column
// widths, and the reductions of its partial sums (the kernel is in
// kmv_simt_bwd.cuh).
#include <algorithm>

#include "kmv_simt_bwd.cuh"

namespace kmv {

extern template cudaError_t bwd_launch_d<1, true>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
extern template cudaError_t bwd_launch_d<1, false>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
extern template cudaError_t bwd_launch_d<2, true>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
extern template cudaError_t bwd_launch_d<2, false>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
extern template cudaError_t bwd_launch_d<3, true>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
extern template cudaError_t bwd_launch_d<3, false>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
extern template cudaError_t bwd_launch_d<4, true>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
extern template cudaError_t bwd_launch_d<4, false>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
extern template cudaError_t bwd_launch_d<8, true>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
extern template cudaError_t bwd_launch_d<8, false>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
extern template cudaError_t bwd_launch_d<16, true>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
extern template cudaError_t bwd_launch_d<16, false>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
extern template cudaError_t bwd_launch_d<32, true>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
extern template cudaError_t bwd_launch_d<32, false>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
extern template cudaError_t bwd_launch_d<64, true>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
extern template cudaError_t bwd_launch_d<64, false>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);

int backward_mp(int m) { return m >= kMaxMPBwd ? kMaxMPBwd : pow2ceil(m); }

namespace {

constexpr int kDims[] = {1, 2, 3, 4, 8, 16, 32, 64};
int dim_class(int d) {
  for (int v : kDims)
    if (d <= v) return v;
  return 0;
}

// dL/dV = alpha amp sum_units part + sigma^2 G, 128 rows and kGvCols columns at a time.
constexpr int kGvCols = 2;
__global__ void __launch_bounds__(kTile) bwd_simt_combine_kernel(KmvArgs a, SimtBwd f) {
  __shared__ double as2[2];
  const int item = blockIdx.x, c = blockIdx.y;
  const int b = a.L.item_inst[item];
  const int s = b * a.chains + c;
  if (a.sys_active && !a.sys_active[s]) return;
  if (threadIdx.x < 2) as2[threadIdx.x] = exp(a.theta[(int64_t)s * a.n_theta + (threadIdx.x ? a.n_theta - 1 : 0)]);
  const int64_t i = a.L.item_row0[item] + threadIdx.x;
  const int64_t nb = a.L.offsets[b + 1] - a.L.offsets[b], len = (int64_t)f.folds * kFoldTiles * kTile;
  const int units = (int)((nb + len - 1) / len);
  __syncthreads();
  if (i >= a.L.offsets[b + 1]) return;
  const int64_t row = (int64_t)c * a.n_total + i;
  const double ai = as2[0] * (double)(a.amp ? a.amp[row] : 1.f);
  for (int c0 = blockIdx.z * kGvCols; c0 < a.m; c0 += gridDim.z * kGvCols) {
    for (int q = c0; q < min(a.m, c0 + kGvCols); ++q) {
      double sum = 0.0;
      for (int u = 0; u < units; ++u) sum += f.part[(((size_t)u * a.chains + c) * a.m + q) * (size_t)a.n_total + i];
      const int64_t idx = row * a.m + q;
      a.Y[idx] = (float)(ai * sum + as2[1] * (double)a.G[idx]);
    }
  }
}

// grad[s, p] = scale_p * sum over the instance's tiles, column chunks and units of
// partial[..., p]: a CTA per (system, entry), threads striding over the partials, then
// the fixed order of block_sum; a few partials in their own order, whatever the batch
// around the system (one thread's serial chain over 157 items measured 75 us).
constexpr int kGradThreads = 128;
__global__ void __launch_bounds__(kGradThreads) grad_finalize_kernel(DevLayout L, SimtBwd f, int chains, int n_theta,
                                                                     const double* theta, const double* partial,
                                                                     double* grad) {
  __shared__ double red[kGradThreads / 32];
  chain_trigger();
  chain_wait();
  const int s = blockIdx.x / n_theta, p = blockIdx.x - s * n_theta;
  const int b = s / chains, c = s - b * chains;
  const double* th = theta + (int64_t)s * n_theta;
  const int64_t nb = L.offsets[b + 1] - L.offsets[b], len = (int64_t)f.folds * kFoldTiles * kTile;
  const int units = (int)((nb + len - 1) / len);
  const int i0 = L.inst_item0[b], n_t = (L.inst_item0[b + 1] - i0 + f.rows - 1) / f.rows;
  const int n = n_t * f.nz * units, per_tile = f.nz * units;
  auto at = [&](int e) {
    const int t = e / per_tile, zu = e - t * per_tile, z = zu / units, u = zu - z * units;
    return partial[((((int64_t)(i0 + t * f.rows) * chains + c) * f.nz + z) * f.units + u) * n_theta + p];
  };
  double acc = 0.0;
  if (n <= 32) {
    if (threadIdx.x < 32) {
      const double v = (int)threadIdx.x < n ? at(threadIdx.x) : 0.0;
      for (int e = 0; e < n; ++e) acc += __shfl_sync(0xffffffffu, v, e);
    }
  } else {
#pragma unroll 4
    for (int e = threadIdx.x; e < n; e += kGradThreads) acc += at(e);
    acc = block_sum(acc, red);
  }
  if (threadIdx.x != 0) return;
  double scale = exp(p == n_theta - 1 ? th[n_theta - 1] : th[0]);
  if (p != 0 && p != n_theta - 1) scale = scale / kHalfLog2e;
  grad[(int64_t)s * n_theta + p] = scale * acc;
}

}  // namespace

// Rows per thread and the number of J units: the wide variant once its finest split
// (units of one fold) gives every SM two CTAs; then about 8 CTAs per SM, and with
// dL/dV at most kSimtPartMax bytes of partial sums (a single unit needs none).  N = 20,000, d = 8, m = 16: 4.38 ms with one row
// per thread and no units, 1.12 ms now, with 0.03 ms for the sums of dL/dV and theta.
SimtBwd simt_bwd_plan(const SimtTiles& T, int n_items, int chains, int64_t n_total, int64_t max_rows, int d, int m,
                      bool want_gv, int num_sms, bool one_unit) {
  SimtBwd f = simt_bwd_plan_plain(n_items, m);
  const int R = bwd_rows(dim_class(d), f.mp);
  const int64_t fpc = std::max<int64_t>(1, (max_rows + kFoldTiles * kTile - 1) / (kFoldTiles * kTile));
  const int64_t wide = (int64_t)(R == 4 ? T.n4 : R == 2 ? T.n2 : n_items) * chains * f.nz;
  if (R > 1 && wide * fpc >= 2 * (int64_t)num_sms) {
    f.rows = R;
    f.tile_item = R == 4 ? T.item4 : T.item2;
    f.n_tiles = R == 4 ? T.n4 : T.n2;
  }
  const int64_t ctas = (int64_t)f.n_tiles * chains * f.nz;
  int64_t units = std::min<int64_t>(fpc, std::max<int64_t>(1, (8 * (int64_t)num_sms + ctas - 1) / std::max<int64_t>(1, ctas)));
  units = std::min<int64_t>(units, std::max(1, 65535 / f.nz));
  const int64_t bytes = want_gv ? (int64_t)sizeof(double) * chains * m * std::max<int64_t>(1, n_total) : 0;
  while (units > 1 && bytes * units > kSimtPartMax) --units;
  if (one_unit) units = 1;
  f.folds = (int)((fpc + units - 1) / units);
  f.units = (int)((fpc + f.folds - 1) / f.folds);
  return f;
}

SimtBwd simt_bwd_plan_plain(int n_items, int m) {
  SimtBwd f{};
  f.n_tiles = n_items;
  f.rows = 1;
  f.chunk = backward_mp(m);
  f.mp = std::max(2, f.chunk);
  f.nz = (m + f.chunk - 1) / f.chunk;
  f.folds = 1 << 30;
  f.units = 1;
  return f;
}

size_t simt_bwd_partials(const SimtBwd& f, int n_items, int chains, int n_theta) {
  return (size_t)std::max(1, n_items) * chains * f.nz * f.units * n_theta;
}
size_t simt_bwd_part_bytes(const SimtBwd& f, int chains, int64_t n_total, int m) {
  return f.units > 1 ? sizeof(double) * (size_t)f.units * chains * m * (size_t)n_total : 0;
}

template <int D>
static cudaError_t bwd_by_ard(const KmvArgs& a, const SimtBwd& f, dim3 grid, cudaStream_t st) {
  return a.ard ? bwd_launch_d<D, true>(a, f, grid, st) : bwd_launch_d<D, false>(a, f, grid, st);
}

cudaError_t launch_backward_simt(const KmvArgs& a, const SimtBwd& f, int n_items, cudaStream_t st) {
  const dim3 grid(f.n_tiles, a.chains, f.nz * f.units);
  cudaError_t e = cudaErrorInvalidValue;
  switch (dim_class(a.d)) {
    case 1: e = bwd_by_ard<1>(a, f, grid, st); break;
    case 2: e = bwd_by_ard<2>(a, f, grid, st); break;
    case 3: e = bwd_by_ard<3>(a, f, grid, st); break;
    case 4: e = bwd_by_ard<4>(a, f, grid, st); break;
    case 8: e = bwd_by_ard<8>(a, f, grid, st); break;
    case 16: e = bwd_by_ard<16>(a, f, grid, st); break;
    case 32: e = bwd_by_ard<32>(a, f, grid, st); break;
    case 64: e = bwd_by_ard<64>(a, f, grid, st); break;
  }
  if (e != cudaSuccess || f.units == 1 || !a.Y) return e;
  const int gz = std::min(65535, (a.m + kGvCols - 1) / kGvCols);
  bwd_simt_combine_kernel<<<dim3(n_items, a.chains, gz), kTile, 0, st>>>(a, f);
  return cudaGetLastError();
}

cudaError_t launch_grad_finalize(const DevLayout& L, const SimtBwd& f, int n_inst, int chains, int n_theta,
                                 const double* theta, const double* partial, double* grad, bool chained,
                                 cudaStream_t st) {
  return launch_chained(chained, grad_finalize_kernel, dim3((unsigned)n_inst * chains * n_theta), kGradThreads, 0, st, L, f, chains, n_theta,
                        theta, partial, grad);
}

}  // namespace kmv

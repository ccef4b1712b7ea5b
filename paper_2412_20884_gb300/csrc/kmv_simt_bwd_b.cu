// Instances of the FP32 adjoint kernel (kmv_simt_bwd.cuh), split over files for build time.
#include "kmv_simt_bwd.cuh"

namespace kmv {
template cudaError_t bwd_launch_d<4, true>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
template cudaError_t bwd_launch_d<4, false>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
template cudaError_t bwd_launch_d<8, true>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
template cudaError_t bwd_launch_d<8, false>(const KmvArgs&, const SimtBwd&, dim3, cudaStream_t);
}  // namespace kmv

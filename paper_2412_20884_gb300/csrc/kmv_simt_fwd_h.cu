// Instances of the FP32 forward kernel (kmv_simt_fwd.cuh), split over files for build time.
#include "kmv_simt_fwd.cuh"

namespace kmv {
template cudaError_t fwd_launch_d<48>(const KmvArgs&, const SimtFwd&, dim3, cudaStream_t);
}  // namespace kmv

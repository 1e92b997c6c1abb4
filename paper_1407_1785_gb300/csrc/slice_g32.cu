// slice_g32.cu -- slice-SVT kernels with 32 lanes per vector pair.
#include "slice_kernel.cuh"

namespace tsvd {

cudaError_t launch_lanes_32(const SliceArgs& a, const SliceShape& sh, size_t smem, int threads,
                           bool xres, cudaStream_t st) {
  TSVD_CASE(32, 1, 1)
  TSVD_CASE(32, 2, 1)
  TSVD_CASE(32, 3, 1)
  TSVD_CASE(32, 4, 1)
  return cudaErrorInvalidValue;
}

}  // namespace tsvd

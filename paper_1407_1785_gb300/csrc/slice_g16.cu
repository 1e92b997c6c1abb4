// slice_g16.cu -- slice-SVT kernels with 16 lanes per vector pair.
#include "slice_kernel.cuh"

namespace tsvd {

cudaError_t launch_lanes_16(const SliceArgs& a, const SliceShape& sh, size_t smem, int threads,
                           bool xres, cudaStream_t st) {
  TSVD_CASE(16, 1, 1)
  TSVD_CASE(16, 2, 1)
  TSVD_CASE(16, 3, 1)
  TSVD_CASE(16, 4, 1)
  TSVD_CASE(16, 6, 1)
  TSVD_CASE(16, 8, 1)
  TSVD_CASE(16, 1, 2)
  TSVD_CASE(16, 2, 2)
  TSVD_CASE(16, 3, 2)
  TSVD_CASE(16, 4, 2)
  return cudaErrorInvalidValue;
}

}  // namespace tsvd

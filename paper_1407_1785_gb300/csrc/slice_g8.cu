// slice_g8.cu -- slice-SVT kernels with 4 or 8 lanes per vector pair.
#include "slice_kernel.cuh"

namespace tsvd {

cudaError_t launch_lanes_8(const SliceArgs& a, const SliceShape& sh, size_t smem, int threads,
                           bool xres, cudaStream_t st) {
  TSVD_CASE(4, 1, 1)
  TSVD_CASE(4, 2, 1)
  TSVD_CASE(8, 1, 1)
  TSVD_CASE(8, 2, 1)
  TSVD_CASE(8, 3, 1)
  TSVD_CASE(8, 4, 1)
  TSVD_CASE(8, 6, 1)
  TSVD_CASE(8, 8, 1)
  TSVD_CASE(8, 1, 2)
  TSVD_CASE(8, 2, 2)
  TSVD_CASE(8, 3, 2)
  TSVD_CASE(8, 4, 2)
  return cudaErrorInvalidValue;
}

}  // namespace tsvd

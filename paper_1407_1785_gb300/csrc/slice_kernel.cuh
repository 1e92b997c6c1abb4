// slice_kernel.cuh -- the slice-SVT kernel and its launch, instantiated by slice_g*.cu.
#pragma once
#include "slice_svt.cuh"

namespace tsvd {
namespace {

template <int G, int CPL, int NP, bool XRES>
__global__ void __maxnreg__(max_regs_for(CPL * NP, XRES))
    jacobi_svt_kernel(SliceArgs a, SliceShape sh) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ SliceShared ss;
  const int C = sh.C;
  const int crank = C > 1 ? (int)cg::this_cluster().block_rank() : 0;
  const int so = blockIdx.x / C;     // slice ordinal in this launch
  float* xbuf = C > 1 ? reinterpret_cast<float*>(static_cast<char*>(a.scratch) +
                                                 (size_t)so * sh.xbuf_floats * sizeof(float))
                      : nullptr;
  svt_slice<G, CPL, NP, XRES>(a, sh, so, crank, xbuf, smem_raw, ss);
}

template <int G, int CPL, int NP, bool XRES>
cudaError_t launch_gc(const SliceArgs& a, const SliceShape& sh, size_t smem, int threads,
                      cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(jacobi_svt_kernel<G, CPL, NP, XRES>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // the register budget can allow fewer threads than the warp cap: the kernel takes any
  // multiple of 32 (it runs a local round's pairs in as many trips as its groups need)
  cudaFuncAttributes fa;
  e = cudaFuncGetAttributes(&fa, jacobi_svt_kernel<G, CPL, NP, XRES>);
  if (e != cudaSuccess) return e;
  if (threads > fa.maxThreadsPerBlock) threads = fa.maxThreadsPerBlock / 32 * 32;
  if (threads < 32) return cudaErrorInvalidConfiguration;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.nslices * sh.C), 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)sh.C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, jacobi_svt_kernel<G, CPL, NP, XRES>, a, sh);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

// Past 3 chunks both forms have the same budget, and one instance serves them.
#define TSVD_CASE(G_, C_, N_)                                                  \
  if (sh.G == G_ && sh.cpl == C_ && sh.np == N_)                               \
    return xres ? launch_gc<G_, C_, N_, true>(a, sh, smem, threads, st)        \
                : launch_gc<G_, C_, N_, (C_ * N_ > 3)>(a, sh, smem, threads, st);

}  // namespace
}  // namespace tsvd

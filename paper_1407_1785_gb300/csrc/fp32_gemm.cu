// fp32_gemm.cu -- the batched complex product of Fourier slices in FP32 on the CUDA cores.
#include "tsvd_internal.h"

namespace tsvd {
namespace {

// C = op(A) op(B), batched, generic strides (see CGemm in tsvd_internal.h), on the CUDA cores.
// A CTA of 8 x 16 threads forms a 16 RP x 16 CN tile, a thread RP pairs of adjacent rows by CN
// columns, with packed FP32x2 FMAs over the two rows of a pair (A is staged planar, so a pair
// of real parts is one 64-bit load; the element of B is the same for both and is doubled in
// registers, in issue slots the half-rate FMAs leave free).  The next K tile is loaded into
// registers while the current one is multiplied, so one barrier per tile remains.  Bound by the
// FMA pipe and the tiles' padding; every product is summed over l in order, as
// acc + (-ai bi) + ar br and acc + ai br + ar bi, whatever the tile.
// Measured against scalar FMAs on 64 x 64 tiles, 4 x 4 outputs a thread (M x N x K, batch):
// 176 x 144 x 144, 51: 72 -> 43 us (34.5 TFLOP/s); 320 x 240 x 240, 31: 152 -> 107 us (43);
// 128 x 96 x 96, 20: 23 -> 11 us; 176 x 55 x 144, 51: 43 -> 23 us.
template <int RP, int CN>
__global__ void __launch_bounds__(128) cgemm_fp32_kernel(CGemm g) {
  constexpr int TM = 16 * RP, TN = 16 * CN, TK = 16;
  __shared__ __align__(16) float As[2][2][TK][TM + 2];   // buffer, re / im
  __shared__ __align__(16) float2 Bs[2][TK][TN + 1];
  if (g.kdev) {
    const int kk = *g.kdev;
    if (g.dynM) g.M = kk;
    if (g.dynN) g.N = kk;
    if (g.dynK) g.K = kk;
  }
  const int i0 = blockIdx.x * TM, j0 = blockIdx.y * TN;
  if (i0 >= g.M || j0 >= g.N) return;
  const int bz = blockIdx.z;
  const float2* A = g.a.p + (int64_t)(g.a.idx ? g.a.idx[bz] : bz) * g.a.bs;
  const float2* B = g.b.p + (int64_t)(g.b.idx ? g.b.idx[bz] : bz) * g.b.bs;
  float2* C = const_cast<float2*>(g.c.p) + (int64_t)(g.c.idx ? g.c.idx[bz] : bz) * g.c.bs;
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
  // staging: 16 neighbouring threads run along whichever index is contiguous in global memory
  const int l16 = tid & 15, grp = tid >> 4;
  const bool a_rows = g.a.s0 == 1, b_cols = g.b.s0 != 1;
  // load u of a thread: (row, l) = (l16 + 16 (u / 2), grp + 8 (u % 2)) along the rows, else
  // (grp + 8 u, l16); the same for B with columns
  const int64_t a_u = a_rows ? 16 * g.a.s0 : 8 * g.a.s0, a_h = a_rows ? 8 * g.a.s1 : 8 * g.a.s0;
  const int64_t b_u = b_cols ? 16 * g.b.s1 : 8 * g.b.s1, b_h = b_cols ? 8 * g.b.s0 : 8 * g.b.s1;
  const int am = a_rows ? l16 : grp, al = a_rows ? grp : l16;
  const int bn = b_cols ? l16 : grp, bl = b_cols ? grp : l16;
  const float2* pa = A + (i0 + am) * g.a.s0 + al * g.a.s1;
  const float2* pb = B + bl * g.b.s0 + (j0 + bn) * g.b.s1;
  float2 ra[2 * RP], rb[2 * CN];
  auto fetch = [&](int l0) {
#pragma unroll
    for (int u = 0; u < 2 * RP; ++u) {
      const int m = a_rows ? am + 16 * (u / 2) : am + 8 * u;
      const int l = a_rows ? al + 8 * (u & 1) : al;
      const int64_t o = a_rows ? (u / 2) * a_u + (u & 1) * a_h : u * a_u;
      ra[u] = i0 + m < g.M && l0 + l < g.K ? pa[o] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < 2 * CN; ++u) {
      const int n = b_cols ? bn + 16 * (u / 2) : bn + 8 * u;
      const int l = b_cols ? bl + 8 * (u & 1) : bl;
      const int64_t o = b_cols ? (u / 2) * b_u + (u & 1) * b_h : u * b_u;
      rb[u] = j0 + n < g.N && l0 + l < g.K ? pb[o] : make_float2(0.f, 0.f);
    }
    pa += TK * g.a.s1;
    pb += TK * g.b.s0;
  };
  const float sa = g.a.conj ? -1.f : 1.f, sb = g.b.conj ? -1.f : 1.f;
  auto stage = [&](int buf) {
#pragma unroll
    for (int u = 0; u < 2 * RP; ++u) {
      const int m = a_rows ? am + 16 * (u / 2) : am + 8 * u;
      const int l = a_rows ? al + 8 * (u & 1) : al;
      As[buf][0][l][m] = ra[u].x;
      As[buf][1][l][m] = sa * ra[u].y;
    }
#pragma unroll
    for (int u = 0; u < 2 * CN; ++u) {
      const int n = b_cols ? bn + 16 * (u / 2) : bn + 8 * u;
      const int l = b_cols ? bl + 8 * (u & 1) : bl;
      Bs[buf][l][n] = make_float2(rb[u].x, sb * rb[u].y);
    }
  };
  float2 accr[RP][CN], acci[RP][CN];
#pragma unroll
  for (int p = 0; p < RP; ++p)
#pragma unroll
    for (int c = 0; c < CN; ++c) accr[p][c] = acci[p][c] = make_float2(0.f, 0.f);
  fetch(0);
  stage(0);
  __syncthreads();
  int buf = 0;
  for (int l0 = 0; l0 < g.K; l0 += TK, buf ^= 1) {
    const bool more = l0 + TK < g.K;
    if (more) fetch(l0 + TK);
#pragma unroll 4
    for (int l = 0; l < TK; ++l) {
      float2 ar[RP], ai[RP];
#pragma unroll
      for (int p = 0; p < RP; ++p) {
        ar[p] = *reinterpret_cast<const float2*>(&As[buf][0][l][2 * tx + 16 * p]);
        ai[p] = *reinterpret_cast<const float2*>(&As[buf][1][l][2 * tx + 16 * p]);
      }
#pragma unroll
      for (int c = 0; c < CN; ++c) {
        const float2 b = Bs[buf][l][ty + 16 * c];
        const float2 br = make_float2(b.x, b.x), bi = make_float2(b.y, b.y);
        const float2 nb = make_float2(-b.y, -b.y);
#pragma unroll
        for (int p = 0; p < RP; ++p) {
          accr[p][c] = __ffma2_rn(ar[p], br, __ffma2_rn(ai[p], nb, accr[p][c]));
          acci[p][c] = __ffma2_rn(ar[p], bi, __ffma2_rn(ai[p], br, acci[p][c]));
        }
      }
    }
    if (more) stage(buf ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int c = 0; c < CN; ++c) {
    const int j = j0 + ty + 16 * c;
    if (j >= g.N) continue;
#pragma unroll
    for (int p = 0; p < RP; ++p) {
      const int i = i0 + 2 * tx + 16 * p;
      float2* o = C + i * g.c.s0 + j * g.c.s1;
      if (i < g.M) o[0] = make_float2(accr[p][c].x, acci[p][c].x);
      if (i + 1 < g.M) o[g.c.s0] = make_float2(accr[p][c].y, acci[p][c].y);
    }
  }
}

}  // namespace

// The tile of an FP32 product: the least work on the busiest SM, where a tile costs its RP x CN
// products a thread and about half of RP + CN + 2 more for its loads and its loop.  Small tiles
// win where large ones pad (144 = 3 x 48) or leave SMs idle, 64 x 64 elsewhere.
cudaError_t launch_cgemm_fp32(const CGemm& g, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return cudaSuccess;
  double best = 1e300;
  int brp = 4, bcn = 4;
  const int64_t sms = device_sm_count();
  for (int rp = 2; rp <= 4; ++rp)
    for (int cn = 1; cn <= 4; ++cn) {
      const int64_t tiles = (int64_t)((g.M + 16 * rp - 1) / (16 * rp)) *
                            ((g.N + 16 * cn - 1) / (16 * cn)) * g.batch;
      const double cost = (double)((tiles + sms - 1) / sms) * (rp * cn + 0.5 * (rp + cn) + 1);
      if (cost < best - 1e-9) {
        best = cost;
        brp = rp;
        bcn = cn;
      }
    }
  const dim3 grid((unsigned)((g.M + 16 * brp - 1) / (16 * brp)),
                  (unsigned)((g.N + 16 * bcn - 1) / (16 * bcn)), (unsigned)g.batch);
#define TSVD_TILE(R_, C_) \
  if (brp == R_ && bcn == C_) cgemm_fp32_kernel<R_, C_><<<grid, 128, 0, st>>>(g);
  TSVD_TILE(2, 1) TSVD_TILE(2, 2) TSVD_TILE(2, 3) TSVD_TILE(2, 4)
  TSVD_TILE(3, 1) TSVD_TILE(3, 2) TSVD_TILE(3, 3) TSVD_TILE(3, 4)
  TSVD_TILE(4, 1) TSVD_TILE(4, 2) TSVD_TILE(4, 3) TSVD_TILE(4, 4)
#undef TSVD_TILE
  return cudaGetLastError();
}

}  // namespace tsvd

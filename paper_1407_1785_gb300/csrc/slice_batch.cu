// slice_batch.cu -- the persistent batched launch: the slice SVTs and tube passes of every tensor
// of a batch in one kernel per ADMM iteration.
#include "slice_svt.cuh"
#include "tube_tile.cuh"

#include <cstring>

namespace tsvd {
namespace {

// ---------------------------------------------------------------------------------------------
// Persistent batched launch.  One launch per ADMM iteration runs, for every tensor of a batch,
// the slice SVTs of that iteration (Lemma of Sec. 4.1 per Fourier slice; the slices of all
// tensors are independent, eq. shrink2) and then the fused tube pass that follows them
// (completion: eq. proj and the dual update of Sec. 4; RPCA: eq. sparse / sparse2 and eq.
// dual of Sec. 5).  Work is taken from device queues:
//   1. cluster items: (tensor, slice) pairs of the tensors planned with C CTAs per slice, in
//      decreasing cost; crank 0 of a cluster takes the next one and shares it over DSMEM;
//   2. CTA items: slices of the small tensors planned with one CTA per slice, in decreasing
//      cost, taken by each CTA once the cluster items are gone;
//   3. tube tiles: (tensor, 32 tubes) in the order in which the tensors' slices finish.
// A tube tile of tensor t starts when t's slices of this iteration are all written: a per-tensor
// counter, raised after each slice, is waited on with a bounded wait (globaltimer, 2 s) that
// sets an error word instead of hanging.  Only taken items are waited on, and a taken item is
// held by a running CTA, so the waits always end.
// ---------------------------------------------------------------------------------------------
constexpr int kBatchG = 16;                               // lanes per vector pair
constexpr unsigned long long kBatchWaitNs = 2000000000ull; // bounded wait of a tube tile

struct BatchDesc {
  BatchTensor t;
  SliceShape sh;   // slice-SVT plan (sh.C = 1: CTA items, else cluster items)
  int rm;          // tube tile rows per thread (2, 4, 8)
  int pad;
};

struct BatchLaunch {
  const BatchDesc* desc;
  const int2* big;
  const int2* small;
  const int* tile_start;    // n + 1 prefix of tiles, in tile order
  const int* tile_tensor;   // tensor at each tile-order position
  int n, nbig, nsmall, ntiles;
  BatchIter it;
  float* xbuf;
  size_t xbuf_floats;
  int C;
};

__device__ __forceinline__ unsigned long long batch_clock() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned batch_ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Bounded wait (one thread): until *p >= target, polling with a short sleep; gives up after
// limit_ns of globaltimer time and returns false.  The persistent kernel's only wait.
__device__ bool wait_counter_geq(const unsigned* p, unsigned target, unsigned long long limit_ns) {
  const unsigned long long t0 = batch_clock();
  while (batch_ld_acquire(p) < target) {
    if (batch_clock() - t0 > limit_ns) return false;
    __nanosleep(256);
  }
  return true;
}

// The bounded wait on a counter nothing raises (tsvd_selftest_bounded_wait): must give up.
__global__ void wait_selftest_kernel(const unsigned* counter, unsigned long long limit_ns, int* err) {
  if (threadIdx.x == 0 && !wait_counter_geq(counter, 1u, limit_ns)) atomicExch(err, 1);
}

__device__ SliceArgs batch_slice_args(const BatchDesc& d, const BatchIter& it) {
  const BatchTensor& t = d.t;
  SliceArgs a{};
  a.ahat = t.spec_a;
  a.zhat = t.spec_b;
  a.slices = t.slices;
  a.nslices = t.nslices;
  a.n1 = t.n1;
  a.n2 = t.n2;
  a.N12 = t.g.N12;
  a.tau = (float)(t.scale / it.r);
  a.tol = it.tol;
  a.max_sweeps = it.max_sweeps;
  a.stat = t.stat;
  a.acc = t.acc;
  a.abs_stop = it.abs_stop;
  if (t.warm) {
    // V form from the previous iteration's V (cold every kWarmColdEvery iterations), rebuilt
    // in the U form from B itself
    const int nv = min(t.n1, t.n2);
    a.vout = t.vwarm;
    a.vstride = (int64_t)nv * nv;
    a.brb = t.spec_a;
    if (it.k % kWarmColdEvery != 0) {
      a.vin = t.vwarm;
      a.prerot = 1;
    }
  }
  return a;
}

// The tube pass of tensor t that follows iteration it.k (it.k < 0: the first pass); false
// when the tensor has none there.
__device__ bool batch_tube_args(const BatchDesc& d, const BatchIter& it, TubeArgs& a) {
  const BatchTensor& t = d.t;
  a = TubeArgs{};
  a.g = t.g;
  a.twid_h = t.twid_h;
  a.twid_f = t.twid_f;
  a.ratio = 1.f;
  const bool complete = t.kind == 1;
  if (it.k < 0) {
    a.in = t.in;
    a.spec_out = t.spec_a;
    if (complete) {
      a.mode = TUBE_COMPLETE;
      a.state = t.state;
      a.first = 1;
      a.write_out = it.iters == 1;
      a.out0 = t.out0;
    } else {
      a.mode = TUBE_FWD;
    }
    return true;
  }
  const int k = it.k;
  if (complete) {
    if (k + 1 < it.iters) {
      a.mode = TUBE_COMPLETE;
      a.in = t.in;
      a.state = t.state;
      a.spec_in = t.spec_b;
      a.spec_out = t.spec_a;
      a.ratio = (float)(it.r / it.r_next);
      a.write_out = k + 2 == it.iters;
      a.out0 = t.out0;
      return true;
    }
    if (t.out1) {
      a.mode = TUBE_INV;
      a.spec_in = t.spec_b;
      a.out0 = t.out1;
      return true;
    }
    return false;
  }
  a.mode = TUBE_RPCA;
  a.in = t.in;
  a.state = t.state;
  a.spec_in = t.spec_b;
  a.spec_out = t.spec_a;
  a.ratio = (float)(it.r / it.r_next);
  a.kappa = (float)((double)t.lambda / it.r);
  a.first = k == 0;
  a.last = k + 1 == it.iters;
  a.out0 = t.out0;
  a.out1 = t.out1;
  a.tube_sparse = t.tube_sparse;
  return true;
}

// Without cross_rounds: their resident vectors, inlined for every chunk count beside the tube
// tiles, spilled 1.8 KB a thread (0.7 without), and an iteration waits for its slowest slice.
// 15 iterations, ms: 4 tensors up to 144 x 176 x 30 and 96 x 128 x 100 34.5 -> 29.0; 6 up to
// 96 x 90 x 30 10.3 -> 9.5.
template <int CMAX>
__device__ void batch_slice(const SliceArgs& a, const SliceShape& sh, int so, int crank,
                            float* xbuf, unsigned char* smem_raw, SliceShared& ss) {
  switch (sh.cpl) {
    case 1: svt_slice<kBatchG, 1, 1, false>(a, sh, so, crank, xbuf, smem_raw, ss); break;
    case 2:
      if constexpr (CMAX >= 2) svt_slice<kBatchG, 2, 1, false>(a, sh, so, crank, xbuf, smem_raw, ss);
      break;
    case 3:
      if constexpr (CMAX >= 3) svt_slice<kBatchG, 3, 1, false>(a, sh, so, crank, xbuf, smem_raw, ss);
      break;
    case 4:
      if constexpr (CMAX >= 4) svt_slice<kBatchG, 4, 1, false>(a, sh, so, crank, xbuf, smem_raw, ss);
      break;
    case 6:
      if constexpr (CMAX >= 6) svt_slice<kBatchG, 6, 1, false>(a, sh, so, crank, xbuf, smem_raw, ss);
      break;
    case 8:
      if constexpr (CMAX >= 8) svt_slice<kBatchG, 8, 1, false>(a, sh, so, crank, xbuf, smem_raw, ss);
      break;
    default: break;
  }
}

template <int CMAX>
__global__ void __maxnreg__(max_regs_for(CMAX, false)) batch_iter_kernel(BatchLaunch L) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ SliceShared ss;
  __shared__ int s_item;
  const BatchIter& it = L.it;
  const int C = L.C;
  cg::cluster_group cluster = cg::this_cluster();
  const int crank = C > 1 ? (int)cluster.block_rank() : 0;
  float* xbuf = C > 1 ? L.xbuf + (size_t)(blockIdx.x / C) * L.xbuf_floats : nullptr;
  if (it.k >= 0) {
    // 1. cluster items (every CTA of a cluster takes the same number of turns)
    if (C > 1 && L.nbig > 0) {
      for (;;) {
        if (crank == 0 && threadIdx.x == 0) s_item = atomicAdd(&it.ctr[0], 1);
        cluster.sync();
        const int item = *cluster.map_shared_rank(&s_item, 0);
        cluster.sync();
        if (item >= L.nbig) break;
        const int2 w = L.big[item];
        const BatchDesc& d = L.desc[w.x];
        batch_slice<CMAX>(batch_slice_args(d, it), d.sh, w.y, crank, xbuf, smem_raw, ss);
        __threadfence();
        cluster.sync();   // every CTA of the cluster has written its columns of the slice
        if (crank == 0 && threadIdx.x == 0) atomicAdd(&it.done[w.x], 1u);
      }
    }
    // 2. single-CTA items
    for (;;) {
      if (threadIdx.x == 0) s_item = atomicAdd(&it.ctr[1], 1);
      __syncthreads();
      const int item = s_item;
      __syncthreads();
      if (item >= L.nsmall) break;
      const int2 w = L.small[item];
      const BatchDesc& d = L.desc[w.x];
      batch_slice<CMAX>(batch_slice_args(d, it), d.sh, w.y, 0, nullptr, smem_raw, ss);
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) atomicAdd(&it.done[w.x], 1u);
    }
    if (it.slices_only) return;
  }
  // 3. tube tiles (threads TILE_THREADS and up skip the tile work); the tile tables are
  // rebuilt only when the tensor changes
  int last_tix = -1;
  for (;;) {
    if (threadIdx.x == 0) s_item = atomicAdd(&it.ctr[2], 1);
    __syncthreads();
    const int item = s_item;
    __syncthreads();
    if (item >= L.ntiles) break;
    int lo = 0, hi = L.n - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) / 2;
      if (L.tile_start[mid] <= item) lo = mid;
      else hi = mid - 1;
    }
    const int tix = L.tile_tensor[lo];
    const BatchDesc& d = L.desc[tix];
    TubeArgs ta;
    if (!batch_tube_args(d, it, ta)) continue;
    if (it.k >= 0) {
      if (threadIdx.x == 0 &&
          !wait_counter_geq(&it.done[tix], (unsigned)(it.k + 1) * (unsigned)d.t.nslices,
                            kBatchWaitNs))
        atomicExch(it.err, 1);
      __syncthreads();
      __threadfence();
    }
    if (threadIdx.x < TILE_THREADS) {
      const int64_t t0 = (int64_t)(item - L.tile_start[lo]) * TT;
      const bool build = tix != last_tix;
      switch (d.rm) {
        case 2: tube_tile_body<2>(ta, t0, smem_raw, build); break;
        case 4: tube_tile_body<4>(ta, t0, smem_raw, build); break;
        default: tube_tile_body<8>(ta, t0, smem_raw, build); break;
      }
    }
    last_tix = tix;
  }
}

template <int CMAX>
cudaError_t batch_occupancy(const BatchPlan& p, int* clusters) {
  cudaError_t e = cudaFuncSetAttribute(batch_iter_kernel<CMAX>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem);
  if (e != cudaSuccess) return e;
  if (p.C == 1) {
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_iter_kernel<CMAX>, p.threads,
                                                      p.smem);
    *clusters = per_sm * device_sm_count();
    return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(p.C * device_sm_count()), 1, 1);
  cfg.blockDim = dim3((unsigned)p.threads, 1, 1);
  cfg.dynamicSmemBytes = p.smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)p.C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaOccupancyMaxActiveClusters(clusters, batch_iter_kernel<CMAX>, &cfg);
}

template <int CMAX>
cudaError_t batch_launch(const BatchPlan& p, const BatchLaunch& L, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(batch_iter_kernel<CMAX>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)p.grid, 1, 1);
  cfg.blockDim = dim3((unsigned)p.threads, 1, 1);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)p.C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, batch_iter_kernel<CMAX>, L);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

size_t align16(size_t x) { return (x + 15) / 16 * 16; }
}  // namespace

bool batch_plan(const BatchTensor* ts, int n, int C, int small_nv, BatchPlan& plan,
                std::vector<unsigned char>& table) {
  if (n <= 0 || (C != 1 && C != 2 && C != 4 && C != 8)) return false;
  plan = BatchPlan{};
  plan.C = C;
  plan.small_nv = small_nv < 0 ? 2 * C * kMinBlock : small_nv;
  plan.ntensors = n;
  std::vector<BatchDesc> desc((size_t)n);
  size_t smem = 0;
  int cmax = 1;
  for (int i = 0; i < n; ++i) {
    const BatchTensor& t = ts[i];
    BatchDesc& d = desc[(size_t)i];
    std::memset(&d, 0, sizeof d);
    d.t = t;
    const int nv = std::min(t.n1, t.n2);
    const SliceKnobs k1 = {1, kBatchG, 1, t.warm ? 1 : 0};
    const SliceKnobs kc = {C, kBatchG, 1, t.warm ? 1 : 0};
    size_t sm = 0;
    SliceShape sh;
    bool ok = false;
    if (C == 1 || nv < plan.small_nv) ok = plan_with_ctas(t.n1, t.n2, 1, k1, sh, sm);
    if (!ok && C > 1) ok = plan_with_ctas(t.n1, t.n2, C, kc, sh, sm);
    if (!ok || sh.G != kBatchG || sh.np != 1) return false;
    d.sh = sh;
    d.rm = tile_rm(t.g);
    if (d.rm == 0) return false;
    smem = std::max(smem, std::max(sm, tile_smem_bytes(t.g)));
    cmax = std::max(cmax, sh.cpl);
    if (sh.C > 1) plan.xbuf_floats = std::max(plan.xbuf_floats, sh.xbuf_floats);
  }
  plan.cmax = cmax <= 4 ? 4 : 8;   // (a 2-chunk instance would run at 80 registers and spill)
  plan.threads = max_warps_for(plan.cmax, false) * 32;
  if (plan.threads < TILE_THREADS) return false;
  plan.smem = smem;
  if (smem + kStaticSmemReserve > (size_t)max_optin_smem()) return false;
  // items in decreasing cost: m n^2 per slice, a cold start ~3x the sweeps of a warm one
  std::vector<double> cost((size_t)n);
  for (int i = 0; i < n; ++i) {
    const double m = std::max(ts[i].n1, ts[i].n2), nn = std::min(ts[i].n1, ts[i].n2);
    cost[(size_t)i] = m * nn * nn * (ts[i].warm ? 1.0 : 3.0);
  }
  std::vector<int2> big, small;
  for (int i = 0; i < n; ++i)
    for (int so = 0; so < ts[i].nslices; ++so)
      (desc[(size_t)i].sh.C > 1 ? big : small).push_back(make_int2(i, so));
  auto by_cost = [&](const int2& a, const int2& b) {
    if (cost[(size_t)a.x] != cost[(size_t)b.x]) return cost[(size_t)a.x] > cost[(size_t)b.x];
    return a.x != b.x ? a.x < b.x : a.y < b.y;
  };
  std::sort(big.begin(), big.end(), by_cost);
  std::sort(small.begin(), small.end(), by_cost);
  plan.nbig = (int)big.size();
  plan.nsmall = (int)small.size();
  // tube tiles: tensors in the order their last slice item is taken
  std::vector<int> last((size_t)n, -1), order((size_t)n);
  for (int j = 0; j < plan.nbig; ++j) last[(size_t)big[(size_t)j].x] = j;
  for (int j = 0; j < plan.nsmall; ++j) last[(size_t)small[(size_t)j].x] = plan.nbig + j;
  for (int i = 0; i < n; ++i) order[(size_t)i] = i;
  std::stable_sort(order.begin(), order.end(),
                   [&](int a, int b) { return last[(size_t)a] < last[(size_t)b]; });
  std::vector<int> tstart((size_t)n + 1, 0), ttensor((size_t)n);
  for (int j = 0; j < n; ++j) {
    const int i = order[(size_t)j];
    ttensor[(size_t)j] = i;
    tstart[(size_t)j + 1] = tstart[(size_t)j] + (int)((ts[i].g.N12 + TT - 1) / TT);
  }
  plan.ntiles = tstart[(size_t)n];
  // device table
  plan.off_desc = 0;
  plan.off_big = align16(sizeof(BatchDesc) * (size_t)n);
  plan.off_small = plan.off_big + align16(sizeof(int2) * big.size());
  plan.off_tstart = plan.off_small + align16(sizeof(int2) * small.size());
  plan.off_ttensor = plan.off_tstart + align16(sizeof(int) * ((size_t)n + 1));
  plan.table_bytes = plan.off_ttensor + align16(sizeof(int) * (size_t)n);
  table.assign(plan.table_bytes, 0);
  std::memcpy(table.data() + plan.off_desc, desc.data(), sizeof(BatchDesc) * (size_t)n);
  if (!big.empty()) std::memcpy(table.data() + plan.off_big, big.data(), sizeof(int2) * big.size());
  if (!small.empty())
    std::memcpy(table.data() + plan.off_small, small.data(), sizeof(int2) * small.size());
  std::memcpy(table.data() + plan.off_tstart, tstart.data(), sizeof(int) * ((size_t)n + 1));
  std::memcpy(table.data() + plan.off_ttensor, ttensor.data(), sizeof(int) * (size_t)n);
  // persistent grid: the clusters that fit on the device at once
  int clusters = 0;
  cudaError_t e = plan.cmax == 4 ? batch_occupancy<4>(plan, &clusters)
                                 : batch_occupancy<8>(plan, &clusters);
  if (e != cudaSuccess || clusters <= 0) {
    cudaGetLastError();
    clusters = std::max(1, device_sm_count() / C);
  }
  plan.grid = clusters * C;
  plan.scratch_bytes = C > 1 ? (size_t)clusters * plan.xbuf_floats * sizeof(float) : 0;
  return true;
}

cudaError_t launch_wait_selftest(const unsigned* counter, unsigned long long limit_ns, int* err,
                                 cudaStream_t st) {
  wait_selftest_kernel<<<1, 32, 0, st>>>(counter, limit_ns, err);
  return cudaGetLastError();
}

cudaError_t launch_batch_iteration(const BatchPlan& p, const void* table_dev, void* scratch,
                                   const BatchIter& it, cudaStream_t st) {
  const char* tb = static_cast<const char*>(table_dev);
  BatchLaunch L;
  L.desc = reinterpret_cast<const BatchDesc*>(tb + p.off_desc);
  L.big = reinterpret_cast<const int2*>(tb + p.off_big);
  L.small = reinterpret_cast<const int2*>(tb + p.off_small);
  L.tile_start = reinterpret_cast<const int*>(tb + p.off_tstart);
  L.tile_tensor = reinterpret_cast<const int*>(tb + p.off_ttensor);
  L.n = p.ntensors;
  L.nbig = p.nbig;
  L.nsmall = p.nsmall;
  L.ntiles = p.ntiles;
  L.it = it;
  L.xbuf = static_cast<float*>(scratch);
  L.xbuf_floats = p.xbuf_floats;
  L.C = p.C;
  if (p.C > 1 && p.nbig > 0 && !scratch) return cudaErrorInvalidValue;
  if (p.cmax == 4) return batch_launch<4>(p, L, st);
  return batch_launch<8>(p, L, st);
}

}  // namespace tsvd

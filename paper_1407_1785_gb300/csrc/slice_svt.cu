// slice_svt.cu -- plans and dispatch of the slice SVTs.
#include "slice_svt.cuh"

#include <cstring>

namespace tsvd {

int max_optin_smem() {
  static int max_optin = -1;
  if (max_optin < 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) !=
        cudaSuccess)
      max_optin = 227 * 1024;
  }
  return max_optin;
}

namespace {

// Lanes per pair and 4-entry chunks per lane for vectors of ld floats (a multiple of 4).
// `prefer` = 0 picks the narrowest group with at most 2 chunks per lane, else 16 lanes;
// `prefer` = 4, 8, 16 or 32 asks for that group width (more chunks per lane = more independent
// work per lane, fewer lanes = fewer shuffle levels and more pairs per warp).
bool pick_group(int ld, int prefer, int& G, int& cpl) {
  const int nchunk = ld / 4;
  const int opts[6] = {1, 2, 3, 4, 6, 8};
  auto fit = [&](int g) {
    const int need = (nchunk + g - 1) / g;
    if (g == 4 && need > 2) return false;
    for (int o : opts)
      if (need <= o) {
        G = g;
        cpl = o;
        return true;
      }
    return false;
  };
  if (prefer) return fit(prefer);
  const int Gs[2] = {4, 8};
  for (int gi = 0; gi < 2; ++gi)
    if ((nchunk + Gs[gi] - 1) / Gs[gi] <= 2) return fit(Gs[gi]);
  return fit(16);
}

}  // namespace

// The block schedule: which circle slot each CTA takes in each block round.  Every next pair
// joins two CTAs that hold one of its blocks each, and every CTA holds two blocks, so the next
// pairs are the edges of cycles over the CTAs; giving each CTA the edge it leaves a cycle by
// lets every CTA keep one block and trade the other.  The rotations and their order are those
// of the circle method, whichever CTA does them (in the block form a CTA that holds its y block
// first takes the pairs of a round in another order).  Worked out by the compiler: a plan is made
// for every candidate of every launch, and 9 slices of 32 x 32 lost 17 of their 215 us a t-SVT to
// this walk on the host.
struct BlockSchedule {
  unsigned char slot_of[2 * kMaxCtasPerSlice - 1][kMaxCtasPerSlice];
};

constexpr BlockSchedule fill_schedule(int C) {
  BlockSchedule sch = {};
  auto& slot_of = sch.slot_of;
  const int nb = 2 * C;
  int at[2 * kMaxCtasPerSlice] = {};   // CTA that holds a block
  for (int r = 0; r < nb - 1; ++r) {
    int bx[kMaxCtasPerSlice] = {}, by[kMaxCtasPerSlice] = {}, cta_of[kMaxCtasPerSlice] = {};
    for (int s = 0; s < C; ++s) {
      round_robin_pair(r, s, nb, bx[s], by[s]);
      cta_of[s] = r == 0 ? s : -1;
    }
    for (int c = 0; r > 0 && c < C; ++c) {
      bool has = false;
      for (int s = 0; s < C; ++s) has |= cta_of[s] == c;
      for (int cur = c; !has;) {   // walk the cycle through c
        int s = 0;
        while (cta_of[s] >= 0 || (at[bx[s]] != cur && at[by[s]] != cur)) ++s;
        cta_of[s] = cur;
        cur = at[bx[s]] == cur ? at[by[s]] : at[bx[s]];
        has = cur == c;
      }
    }
    for (int s = 0; s < C; ++s) {
      slot_of[r][cta_of[s]] = (unsigned char)s;
      at[bx[s]] = at[by[s]] = cta_of[s];
    }
  }
  return sch;
}

// What the exchange of svt_slice relies on: round 0 as loaded (slot c on CTA c), every slot of a
// round on one CTA, and every CTA with exactly one of its two blocks in the next round (the
// circle method itself brings every pair of blocks together once).
constexpr bool one_block_stays(const BlockSchedule& sch, int C) {
  const int nb = 2 * C;
  for (int c = 0; c < C; ++c)
    if (sch.slot_of[0][c] != c) return false;
  bool met[2 * kMaxCtasPerSlice][2 * kMaxCtasPerSlice] = {};
  for (int r = 0; r < nb - 1; ++r)
    for (int c = 0; c < C; ++c) {
      int bx = 0, by = 0, nx = 0, ny = 0;
      round_robin_pair(r, sch.slot_of[r][c], nb, bx, by);
      if (bx == by || met[bx][by] || met[by][bx]) return false;
      met[bx][by] = true;
      for (int d = 0; d < c; ++d)
        if (sch.slot_of[r][d] == sch.slot_of[r][c]) return false;
      if (r + 2 == nb) continue;
      round_robin_pair(r + 1, sch.slot_of[r + 1][c], nb, nx, ny);
      if ((bx == nx || bx == ny) == (by == nx || by == ny)) return false;
    }
  return true;
}

constexpr BlockSchedule kSchedules[4] = {fill_schedule(1), fill_schedule(2), fill_schedule(4),
                                         fill_schedule(8)};
static_assert(one_block_stays(kSchedules[0], 1) && one_block_stays(kSchedules[1], 2) &&
                  one_block_stays(kSchedules[2], 4) && one_block_stays(kSchedules[3], 8),
              "a CTA must keep one block from round to round");

static const BlockSchedule& block_schedule(int C) { return kSchedules[C == 8 ? 3 : C / 2]; }

bool plan_with_ctas(int n1, int n2, int C, const SliceKnobs& k, SliceShape& sh, size_t& smem) {
  const int max_optin = max_optin_smem();
  sh.rows = n1 < n2 ? 1 : 0;
  sh.nv = n1 < n2 ? n1 : n2;
  sh.len = n1 < n2 ? n2 : n1;
  sh.vform = k.vform ? 1 : 0;
  sh.block = k.block ? 1 : 0;
  sh.C = C;
  sh.nb = 2 * C;
  std::memcpy(sh.slot_of, block_schedule(C).slot_of, sizeof sh.slot_of);
  sh.bs = (sh.nv + sh.nb - 1) / sh.nb;
  if (sh.block) {
    // block form: rows of the vector's 4-entry chunks (and its V entries), no lane layout;
    // it runs in the 16-lane, 4-chunk kernel instance (its register budget), nl <= 128
    if (2 * sh.bs > 128 || k.ppg > 1) return false;
    sh.G = 16;
    sh.cpl = 4;
    sh.np = 1;
    sh.ld = 4 * ((sh.len + 3) / 4);
    sh.ldv = sh.vform ? 4 * ((sh.nv + 3) / 4) : 0;
    sh.nlp = 2 * sh.bs + 1;
  } else {
    // lanes and chunks for the vector's own 4-entry chunks (the row pitch is made odd below;
    // sizing the chunks from an odd pitch instead padded e.g. a 128-entry vector to 192)
    if (!pick_group(4 * ((sh.len + 3) / 4), k.lanes, sh.G, sh.cpl)) return false;
    // rows padded so that the vector part is exactly G * cpl chunks and the V part a multiple
    // of G chunks: every lane's chunks lie inside the row and the rotation needs no tests
    sh.ld = 4 * sh.G * sh.cpl;
    sh.ldv = sh.vform ? 4 * (((sh.nv + 3) / 4 + sh.G - 1) / sh.G * sh.G) : 0;
    sh.np = k.ppg == 2 ? 2 : 1;
    if (k.ppg != 0 && k.ppg != 1 && k.ppg != 2) return false;
    if (sh.np == 2 && (sh.G == 4 || sh.cpl > 4)) return false;   // register budget
    if (sh.G == 32 && (sh.np == 2 || sh.cpl > 4)) return false;   // no such kernel instances
    sh.nlp = 0;
  }
  sh.rowp = sh.ld + sh.ldv;
  if (((sh.rowp / 4) & 1) == 0) sh.rowp += 4;   // pitch / 4 odd
  sh.kcap = C > 1 ? 2 * sh.bs * sh.rowp / sh.ld : 2 * sh.bs;
  sh.xbuf_floats = C > 1 ? (size_t)2 * sh.nb * 2 * sh.bs * sh.rowp : 0;
  for (int nc = kNC; nc >= 1; nc >>= 1) {
    sh.nc = nc;
    smem = slice_smem_bytes(sh);
    if (smem + kStaticSmemReserve <= (size_t)max_optin) return true;
  }
  return false;
}

namespace {

// CTAs per slice: the fewest waves of one CTA per SM, weighted by the work of one CTA
// (1/C), without blocks thinner than kMinBlock vectors; the smallest C on ties.  k.ctas = -1:
// the fewest CTAs that hold the slice (for launches that share the GPU with others).
bool plan_slice(int n1, int n2, int nslices, const SliceKnobs& k, SliceShape& sh,
                size_t& smem) {
  const int nv = n1 < n2 ? n1 : n2;
  const int cands[4] = {1, 2, 4, 8};
  if (k.ctas == -1) {
    SliceKnobs k1 = k;
    for (int C : cands) {
      k1.ctas = C;
      if (plan_with_ctas(n1, n2, C, k1, sh, smem)) return true;
    }
    return false;
  }
  const int force = k.ctas;
  double best = 1e300;
  bool found = false;
  for (int C : cands) {
    if (force && C != force) continue;
    if (!force && C > 1 && nv < 2 * C * kMinBlock) continue;
    SliceShape t;
    size_t sm;
    if (!plan_with_ctas(n1, n2, C, k, t, sm)) continue;
    const int sms = device_sm_count();
    const int waves = (nslices * C + sms - 1) / sms;
    const double cost = (double)waves / C;
    if (cost < best - 1e-12) {
      best = cost;
      sh = t;
      smem = sm;
      found = true;
    }
  }
  if (!found && !force) {
    // slices too large for the thin-block rule: take the smallest C that fits
    for (int C : cands) {
      SliceShape t;
      size_t sm;
      if (plan_with_ctas(n1, n2, C, k, t, sm)) {
        sh = t;
        smem = sm;
        return true;
      }
    }
  }
  return found;
}

size_t scratch_for(const SliceShape& sh, int64_t N12, int nslices) {
  (void)N12;
  if (sh.C <= 1) return 0;
  return (size_t)nslices * sh.xbuf_floats * sizeof(float);
}

}  // namespace

bool jacobi_svt_supported(int n1, int n2) {
  SliceShape sh;
  size_t smem;
  const SliceKnobs k = {0, 0, 0, 0};
  return n1 >= 1 && n2 >= 1 && plan_slice(n1, n2, 1, k, sh, smem);
}

bool jacobi_svt_plan_ok(int n1, int n2, int nslices, const SliceKnobs& k) {
  SliceShape sh;
  size_t smem;
  return n1 >= 1 && n2 >= 1 && plan_slice(n1, n2, nslices, k, sh, smem);
}

size_t jacobi_svt_scratch_bytes(int n1, int n2, int nslices, const SliceKnobs& k) {
  SliceShape sh;
  size_t smem;
  if (!plan_slice(n1, n2, nslices, k, sh, smem)) return 0;
  return scratch_for(sh, (int64_t)n1 * n2, nslices);
}

int jacobi_svt_ctas_per_slice(int n1, int n2, int nslices, const SliceKnobs& k) {
  SliceShape sh;
  size_t smem;
  if (!plan_slice(n1, n2, nslices, k, sh, smem)) return 0;
  return sh.C;
}

cudaError_t launch_jacobi_svt(const SliceArgs& a, cudaStream_t st) {
  if (a.nslices <= 0) return cudaSuccess;
  SliceShape sh;
  size_t smem;
  if (!plan_slice(a.n1, a.n2, a.nslices, a.knobs, sh, smem)) return cudaErrorInvalidValue;
  if (sh.C > 1 && (a.scratch == nullptr || a.scratch_bytes < scratch_for(sh, a.N12, a.nslices)))
    return cudaErrorInvalidValue;
  if (a.wout && a.wout_stride < (int64_t)a.n1 * a.n2) return cudaErrorInvalidValue;
  if ((a.vin || a.vout) && (!sh.vform || a.vstride < (int64_t)sh.nv * sh.nv))
    return cudaErrorInvalidValue;
  const int per_warp = 32 / sh.G * sh.np;     // pairs a warp has in flight
  const int chunks = sh.cpl * sh.np;
  // enough groups for all pairs of a local round in as few passes as fit, balanced
  auto passes_of = [&](bool x) {
    const int most = max_warps_for(chunks, x) * per_warp;
    return (sh.bs + most - 1) / most;
  };
  auto warps_of = [&](bool x) {
    // block form: a warp per 4 local vectors (the Gram tiles and update chunks spread over them)
    const int per_pass = passes_of(x) * per_warp;
    const int n = sh.block ? (2 * sh.bs + 3) / 4 : (sh.bs + per_pass - 1) / per_pass;
    return std::min(std::max(n, kMinWarps), max_warps_for(chunks, x));
  };
  auto waves_of = [&](bool x) {
    const int by_regs = 65536 / (max_regs_for(chunks, x) * warps_of(x) * 32);
    const int by_smem = (int)(kSmSmem / (smem + kStaticSmemReserve));
    const int64_t held = (int64_t)device_sm_count() * std::max(1, std::min(by_regs, by_smem));
    return ((int64_t)a.nslices * sh.C + held - 1) / held;
  };
  // Which instance (up to 3 chunks; others have one): the one with x in registers, unless its
  // 16 warps need two passes a round where 24 (18 at 3 chunks) need one, its registers cost a
  // wave of CTAs, or there are no cross rounds (C = 1) and the other does not spill (3 chunks).
  // A t-SVT without / with x in registers, us: two passes, 101 slices of 70 x 90, C = 1: 960 /
  // 1195; 126 of 80 x 100, 32 lanes, C = 2: 1734 / 1984; a wave, 126 of 80 x 100, 16 lanes,
  // C = 2: 1071 / 1440; 51 of 96 x 128, 32 lanes, C = 8: 1079 / 1485; 3 chunks, 32 of 61 x 75, 8
  // lanes, C = 1: 598 / 635.  Else 126 of 61 x 75, 16 lanes, C = 4: 750 / 687; 51 of 61 x 75,
  // 32 lanes, C = 1: 957 / 895; three passes against two, 126 of 96 x 128, 32 lanes, C = 1:
  // 2319 / 2234.
  const bool xres = sh.block || chunks > 3 ||
                    !(passes_of(true) >= 2 * passes_of(false) || (sh.C == 1 && chunks == 3) ||
                      (a.nslices * sh.C > device_sm_count() && waves_of(false) < waves_of(true)));
  const int threads = warps_of(xres) * 32;
  if (sh.G == 32) return launch_lanes_32(a, sh, smem, threads, xres, st);
  if (sh.G == 16) return launch_lanes_16(a, sh, smem, threads, xres, st);
  return launch_lanes_8(a, sh, smem, threads, xres, st);
}

}  // namespace tsvd

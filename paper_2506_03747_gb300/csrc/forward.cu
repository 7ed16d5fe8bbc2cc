// Forward transient kernel: the (scan point, surface point) pair sum of the
// generalised Eq. 1 of Shi et al. (arXiv 2506.03747), accumulated as a
// per-scan-point histogram over time bins, with the Gaussian jitter of
// Eq. 16/17 fused into the write-out, or as the differentiable Gaussian splat.
//
// Layout and schedule (GB300, sm_103a):
//  * One CTA tile = 32 scan points; lane l of every warp owns scan point l of
//    the tile, so the shared histogram [bin][32] gives every lane its own bank
//    and the shared atomics of a warp never conflict.
//  * Surface points are packed in pairs (64 B, see PointPair). One producer warp
//    stages the groups of 16 pairs that the tile may bin into shared memory by
//    1-D TMA bulk copies, a few slots ahead on mbarriers; the other warps read the
//    same slot (broadcast loads) and split its pairs; each lane evaluates the two
//    points of a pair for its scan point with packed FP32x2 arithmetic
//    (__ffma2_rn & co.).
//  * Work units (scan tile, bin window, point block): a first kernel lists those
//    that the bounds leave, and a persistent grid takes the list in contiguous
//    ranges of equal weight, the rest of a long list in claimed chunks. A CTA
//    flushes its partial histogram into the zeroed output with vectorised global
//    reductions whenever its (tile, window) changes. The jitter convolution is
//    linear, so it is applied to each partial histogram during the flush.
#include "forward_core.cuh"
#include "pack_core.cuh"

#include <algorithm>

namespace nlos {

// Standalone launch: a persistent grid (one CTA per SM) over the live-unit list
// or, without one, over chunks of all units claimed from a counter in the scene
// scratch.
template <int SCAN, int COS, int MODE>
__global__ void __launch_bounds__(1024, 1)
    fwd_kernel(const __grid_constant__ FwdArgs a, const __grid_constant__ MomTab mt,
               const __grid_constant__ OccSet occ) {
  extern __shared__ __align__(128) unsigned char smem[];
  FwdSmem sm;
  const size_t hist_bytes = (MODE == MODE_SPLAT_MOM) ? (size_t)kMoments * kMomRows * kTile * 4
                                                     : (size_t)a.bw * kTile * 4;
  sm.hist = reinterpret_cast<float*>(smem);
  sm.stage = reinterpret_cast<PointPair*>(smem + hist_bytes);
  sm.bars = reinterpret_cast<uint64_t*>(sm.stage + (size_t)a.stages * a.ppb);
  sm.units = reinterpret_cast<unsigned long long*>(sm.bars + 2 * a.stages);
  sm.lane_units = sm.units + a.stages + 1;
  sm.rows = reinterpret_cast<uint32_t*>(sm.lane_units + 32);
  sm.fill = sm.rows + kRowWords;
  sm.occ = sm.fill + kMaxRangedStages;
  if (threadIdx.x == 0) {
    for (uint32_t i = 0; i < a.stages; ++i) {
      mbar_init(&sm.bars[i], 1);                                 // full
      mbar_init(&sm.bars[a.stages + i], (blockDim.x >> 5) - 1);  // empty (consumer warps)
    }
    fence_mbar_init();
  }
  __syncthreads();
  FwdCount cnt;
  uint32_t it = 0;
  (void)fwd_run_ws<SCAN, COS, MODE, MODE == MODE_SPLAT_MOM ? 2 : kFwdUnroll, true>(a, 0, 0, sm, (int)a.stages, cnt, &mt, it,
                                                      a.next_chunk, a.chunk, a.units, 0, &occ);
  if (MODE == MODE_NEAREST_COUNT && cnt.boundary) atomicAdd(a.boundary, cnt.boundary);
  // the count is warp-uniform: one lane adds it, 64 pairs per warp iteration
  if ((threadIdx.x & 31) == 0 && cnt.full) atomicAdd(a.pairs_full, cnt.full * 64ull);
  if ((threadIdx.x & 31) == 0 && cnt.tested) atomicAdd(a.pairs_tested, cnt.tested * 64ull);
}

// Zeroes n floats from a 16-byte aligned p, by the whole grid.
__device__ __forceinline__ void zero_floats(float* p, size_t n) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x, nt = (size_t)gridDim.x * blockDim.x;
  float4* p4 = reinterpret_cast<float4*>(p);
  for (size_t i = t; i < n / 4; i += nt) p4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  for (size_t i = n / 4 * 4 + t; i < n; i += nt) p[i] = 0.f;
}

constexpr uint32_t kRunWeight = 10;  // a tile change in groups of work (3 to 14 thousand cycles)
constexpr int kListThreads = 1024;  // (of fewer blocks than 128 a tile: 256)

// The live units of a pass, for the forward's ranges and chunk claims: one CTA
// per (tile, window) tests the point blocks against the bounds (unit_live),
// then the groups of the live ones (the warps take them in turn: the live blocks
// of a tile are neighbours, mostly of one warp), and appends the
// units that have any with the histogram rows they can touch. Entries of one
// (tile, window) are contiguous (a CTA's blocks at a time), so a range of the list
// rarely spans many tiles; the order of the runs does not matter. Each entry
// holds the weight of the list before it (both come from one atomic, so they
// ascend together). The same launch zeroes the output that the forward adds to
// (of a list in several passes, a memory set does).
template <int SCAN, int COS, int MODE>
__global__ void __launch_bounds__(kListThreads)
    unit_list_kernel(const __grid_constant__ FwdArgs a, ListEntry* __restrict__ list,
                     unsigned long long* __restrict__ n_live) {
  __shared__ uint32_t s_units[32], s_groups[32], s_n;
  __shared__ uint32_t s_blk[kListThreads], s_rows[kListThreads], s_mask[kListThreads];
  __shared__ unsigned long long s_base;
  if (a.list_zeroes) {
    zero_floats(a.tau, (size_t)a.S * a.B);
    if (MODE == MODE_SPLAT_MOM) zero_floats(a.far_mass, a.S);
  }
  const unsigned long long tw = a.list_tw0 + blockIdx.x;
  const float margin = window_margin<MODE>(a);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const TileBound tile = a.tiles[(uint32_t)(tw / a.n_win)];
  const int w0 = window_start(a, (uint32_t)(tw % a.n_win));
  const float lim = (float)window_bins(a, w0);
  for (uint32_t b0 = 0; b0 < a.n_blk; b0 += blockDim.x) {
    const uint32_t blk = b0 + threadIdx.x;
    const unsigned long long unit = tw * a.n_blk + blk;
    float ulo = 0.f, uhi = 0.f;
    const bool maybe =
        blk < a.n_blk && (a.ppb == 2 * kSubPairs
                              ? unit_live_halves<SCAN, COS>(a, unit, margin, ulo, uhi)
                              : unit_live<SCAN, COS>(a, unit, margin, ulo, uhi));
    const uint32_t found = __ballot_sync(0xffffffffu, maybe);
    if (lane == 0) s_units[warp] = (uint32_t)__popc(found);
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t sum = 0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        const uint32_t c = s_units[w];
        s_units[w] = sum;
        sum += c;
      }
      s_n = sum;
    }
    __syncthreads();
    if (maybe) {
      const uint32_t at = s_units[warp] + __popc(found & ((1u << lane) - 1u));
      s_blk[at] = blk;
      s_rows[at] = unit_rows(ulo, uhi, margin, a.bw);
    }
    __syncthreads();
    const uint32_t n = s_n;
    for (uint32_t i = warp; i < n; i += blockDim.x >> 5) {
      const uint32_t g = block_groups<SCAN, COS>(a, tile, s_blk[i], w0, lim, margin);
      if (lane == 0) s_mask[i] = g;
    }
    __syncthreads();
    // thread i takes the i-th of them
    const uint32_t groups = threadIdx.x < n ? s_mask[threadIdx.x] : 0u;
    const uint32_t mask = __ballot_sync(0xffffffffu, groups != 0u);
    uint32_t upto = (uint32_t)__popc(groups);  // inclusive sum over the lanes
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, upto, o);
      if (lane >= o) upto += v;
    }
    if (lane == 31) {
      s_units[warp] = (uint32_t)__popc(mask);
      s_groups[warp] = upto;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t units = 0, sum = 0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        const uint32_t u = s_units[w], g = s_groups[w];
        s_units[w] = units;
        s_groups[w] = sum;
        units += u;
        sum += g;
      }
      // (a run's weight is more than any weight within it, so entries ascend)
      const unsigned long long weight = ((sum + kRunWeight) >> a.list_shift) + 1u;
      s_base = units ? atomicAdd(n_live, units | (weight << 32)) : 0ull;
    }
    __syncthreads();
    if (groups != 0u) {
      const uint32_t pos = (uint32_t)s_base + s_units[warp] + __popc(mask & ((1u << lane) - 1u));
      const uint32_t before = (uint32_t)(s_base >> 32) +
                              ((s_groups[warp] + upto - (uint32_t)__popc(groups)) >> a.list_shift);
      list[pos] = ListEntry{(uint32_t)(tw * a.n_blk + s_blk[threadIdx.x]), s_rows[threadIdx.x],
                            groups, before};
    }
    __syncthreads();
  }
}

// Moment form, after the forward: the transients for which the weight kept
// beyond the splat's cut could exceed 1e-5 of their own peak (far_mass pairs
// beyond the ends, at most 1.6e-8 of their peak each) are summed again tap by
// tap. One warp per transient, bound by reading tau once from L2; the sums
// again are rare (a scan corner whose window holds only tails).
template <int SCAN, int COS>
__global__ void __launch_bounds__(256) splat_tail_kernel(const __grid_constant__ FwdArgs a) {
  const int lane = threadIdx.x & 31;
  const uint32_t warps = gridDim.x * (blockDim.x >> 5);
  for (uint32_t si = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); si < a.S; si += warps) {
    const ScanPoint sp = a.scan[si];
    const float far = a.far_mass[sp.row];
    if (far == 0.f) continue;
    float* row = a.tau + (size_t)sp.row * a.B;
    float peak = 0.f;
    for (uint32_t b = lane; b < a.B; b += 32) peak = fmaxf(peak, row[b]);
    for (int o = 16; o > 0; o >>= 1) peak = fmaxf(peak, __shfl_xor_sync(0xffffffffu, peak, o));
    if (!(far * a.norm * 1.6e-8f > 1e-5f * peak)) continue;
    for (uint32_t b = lane; b < a.B; b += 32) row[b] = 0.f;
    __syncwarp();
    for (uint32_t i = lane; i < a.n_pairs; i += 32) {
      PointPair q;
      load_pair(a.pairs + i, q);
      float2 u, w, cn;
      pair_eval2<SCAN, COS>(q, make_float2(-sp.sx, -sp.sx), make_float2(-sp.sy, -sp.sy),
                            make_float2(sp.off, sp.off), make_float2(a.kbin, a.kbin), u, w, cn);
      for (int h = 0; h < 2; ++h) {
        const float uh = h ? u.y : u.x, wh = h ? w.y : w.x;
        if (!facing<COS>(h ? cn.y : cn.x) || !(uh > -a.reach && uh < (float)a.B + a.reach)) continue;
        const int lo = max(0, (int)(floorf(uh - 0.5f - a.reach) + 1.0f));
        const int hi = min((int)a.B - 1, (int)(ceilf(uh - 0.5f + a.reach) - 1.0f));
        for (int b = lo; b <= hi; ++b) {
          const float x = (float)b + 0.5f - uh;
          red_add_global(row + b, wh * a.norm * expf(-x * x * a.inv2s2));
        }
      }
    }
  }
}

// Per-pair table (debug/parity): the same pack and pair_eval2 arithmetic on
// the points 2k, 2k + 1 of the caller's order (the forward packs them in a
// spatial order) for scan point s_begin + i; u relative to bin 0, w as
// accumulated.
struct PairTableArgs {
  const float* raw;
  unsigned int* err;
  uint32_t n_pairs, P;
  int scan_mode, cos_mode;
  PackConst pc;
};

template <int SCAN, int COS>
__global__ void pair_table_kernel(const PairTableArgs t, const ScanPoint* scan, uint64_t s_begin,
                                  uint64_t s_count, float kbin, float* u_out, float* w_out) {
  const uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t n_pairs = t.n_pairs, P = t.P;
  if (idx >= s_count * n_pairs) return;
  const uint64_t i = idx / n_pairs;
  const uint32_t k = (uint32_t)(idx % n_pairs);
  const ScanPoint sp = scan[s_begin + i];
  const PointPair q = pack_pair_value(t.raw, P, k, t.scan_mode, t.cos_mode, t.pc, t.err, nullptr);
  float2 u, w, cn;
  pair_eval2<SCAN, COS>(q, make_float2(-sp.sx, -sp.sx), make_float2(-sp.sy, -sp.sy),
                        make_float2(sp.off, sp.off), make_float2(kbin, kbin), u, w, cn);
  if (!facing<COS>(cn.x)) w.x = 0.f;
  if (!facing<COS>(cn.y)) w.y = 0.f;
  const uint64_t p0 = 2ull * k;
  if (u_out) {
    u_out[i * P + p0] = u.x;
    if (p0 + 1 < P) u_out[i * P + p0 + 1] = u.y;
  }
  if (w_out) {
    w_out[i * P + p0] = w.x;
    if (p0 + 1 < P) w_out[i * P + p0 + 1] = w.y;
  }
}

// ---------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------
namespace {

using FwdFn = void (*)(FwdArgs, MomTab, OccSet);
using TailFn = void (*)(FwdArgs);

TailFn pick_tail(int scan, int cos) {
  if (scan == NLOS_CONFOCAL) {
    if (cos == NLOS_COS_NONE) return splat_tail_kernel<NLOS_CONFOCAL, NLOS_COS_NONE>;
    if (cos == NLOS_COS_OBJECT) return splat_tail_kernel<NLOS_CONFOCAL, NLOS_COS_OBJECT>;
    return splat_tail_kernel<NLOS_CONFOCAL, NLOS_COS_OBJECT_WALL>;
  }
  if (cos == NLOS_COS_NONE) return splat_tail_kernel<NLOS_NONCONFOCAL, NLOS_COS_NONE>;
  if (cos == NLOS_COS_OBJECT) return splat_tail_kernel<NLOS_NONCONFOCAL, NLOS_COS_OBJECT>;
  return splat_tail_kernel<NLOS_NONCONFOCAL, NLOS_COS_OBJECT_WALL>;
}
using ListFn = void (*)(FwdArgs, ListEntry*, unsigned long long*);

template <int SCAN, int COS>
ListFn pick_list_mode(int mode) {
  switch (mode) {
    case MODE_NEAREST: return unit_list_kernel<SCAN, COS, MODE_NEAREST>;
    case MODE_NEAREST_OCC: return unit_list_kernel<SCAN, COS, MODE_NEAREST_OCC>;
    case MODE_SPLAT_MOM: return unit_list_kernel<SCAN, COS, MODE_SPLAT_MOM>;
    case MODE_SPLAT: return unit_list_kernel<SCAN, COS, MODE_SPLAT>;
    default: return nullptr;  // the boundary count evaluates every unit
  }
}

ListFn pick_list(int scan, int cos, int mode) {
  if (scan == NLOS_CONFOCAL) {
    if (cos == NLOS_COS_NONE) return pick_list_mode<NLOS_CONFOCAL, NLOS_COS_NONE>(mode);
    if (cos == NLOS_COS_OBJECT) return pick_list_mode<NLOS_CONFOCAL, NLOS_COS_OBJECT>(mode);
    return pick_list_mode<NLOS_CONFOCAL, NLOS_COS_OBJECT_WALL>(mode);
  }
  if (cos == NLOS_COS_NONE) return pick_list_mode<NLOS_NONCONFOCAL, NLOS_COS_NONE>(mode);
  if (cos == NLOS_COS_OBJECT) return pick_list_mode<NLOS_NONCONFOCAL, NLOS_COS_OBJECT>(mode);
  return pick_list_mode<NLOS_NONCONFOCAL, NLOS_COS_OBJECT_WALL>(mode);
}

template <int SCAN, int COS>
FwdFn pick_mode(int mode) {
  switch (mode) {
    case MODE_NEAREST: return fwd_kernel<SCAN, COS, MODE_NEAREST>;
    case MODE_NEAREST_COUNT: return fwd_kernel<SCAN, COS, MODE_NEAREST_COUNT>;
    case MODE_NEAREST_OCC: return fwd_kernel<SCAN, COS, MODE_NEAREST_OCC>;
    case MODE_SPLAT_MOM: return fwd_kernel<SCAN, COS, MODE_SPLAT_MOM>;
    default: return fwd_kernel<SCAN, COS, MODE_SPLAT>;
  }
}

FwdFn pick(int scan, int cos, int mode) {
  if (scan == NLOS_CONFOCAL) {
    if (cos == NLOS_COS_NONE) return pick_mode<NLOS_CONFOCAL, NLOS_COS_NONE>(mode);
    if (cos == NLOS_COS_OBJECT) return pick_mode<NLOS_CONFOCAL, NLOS_COS_OBJECT>(mode);
    return pick_mode<NLOS_CONFOCAL, NLOS_COS_OBJECT_WALL>(mode);
  }
  if (cos == NLOS_COS_NONE) return pick_mode<NLOS_NONCONFOCAL, NLOS_COS_NONE>(mode);
  if (cos == NLOS_COS_OBJECT) return pick_mode<NLOS_NONCONFOCAL, NLOS_COS_OBJECT>(mode);
  return pick_mode<NLOS_NONCONFOCAL, NLOS_COS_OBJECT_WALL>(mode);
}

}  // namespace

// D_n[i] = K^(n)(X_i) / (n! q^n) for the Gaussian K(x) = exp(-x^2/(2 s^2)) / (s sqrt(2 pi)):
// K^(n)(x) = (-1)^n He_n(x/s) K(x) / s^n with the probabilists' Hermite
// polynomials He_0 = 1, He_1 = t, He_{n+1} = t He_n - n He_{n-1} (FP64).
void moment_table(double s, MomTab& mt) {
  mt.J = (int)std::ceil(6.0 * s) + 1;
  mt.q = moment_rows_per_bin(s);
  for (int i = 0; i < (2 * mt.J + 1) * mt.q; ++i) {
    const double x = 0.5 - (i - mt.J * mt.q + 0.5) / mt.q, t = x / s;
    const double k = std::exp(-0.5 * t * t) / (s * std::sqrt(2.0 * 3.14159265358979323846));
    double he[kMomTerms];
    he[0] = 1.0;
    he[1] = t;
    for (int n = 1; n + 1 < kMomTerms; ++n) he[n + 1] = t * he[n] - n * he[n - 1];
    double scale = 1.0;  // n! (q s)^n
    for (int n = 0; n < kMomTerms; ++n) {
      if (n >= 1) scale *= n * mt.q * s;
      mt.d[i][n] = (float)(((n & 1) ? -1.0 : 1.0) * he[n] * k / scale);
    }
  }
}

int jitter_radius(double sigma) {
  if (!(sigma > 0.0)) return 0;
  return (int)std::ceil(2.0 * sigma);
}

// What every forward of a scene takes, resolved once: the launch's arguments
// and shape, and the live-unit list's memory (resolving it on each call, with a
// list from the stream-ordered pool and three memsets, made the smallest scene's
// pass 32 us of host calls). Only occluders change it (the kernel's mode).
struct FwdPlan {
  FwdArgs a{};
  MomTab mt{};
  int mode = -1;
  FwdFn fn = nullptr;
  ListFn list_fn = nullptr;  // null: chunks of all units are claimed
  size_t smem = 0;
  unsigned grid = 0;
  ListEntry* list = nullptr;  // [pass_runs * n_blk], or null
  uint64_t pass_runs = 0;     // (tile, window) runs of a pass over the list
};

namespace {

int forward_mode(const SceneImpl& sc) {
  const Geometry& g = sc.g;
  return g.bin_mode == NLOS_BIN_SPLAT ? (forward_moments(g.sigma, g.P, g.B) ? MODE_SPLAT_MOM
                                                                                : MODE_SPLAT)
         : sc.params.boundary_eps > 0.f ? MODE_NEAREST_COUNT
         : sc.occ.n > 0                 ? MODE_NEAREST_OCC
                                        : MODE_NEAREST;
}

// Kernels of the plan's mode, allowed all of the shared memory an SM has.
cudaError_t plan_mode(FwdPlan& p, const SceneImpl& sc, int mode) {
  const Geometry& g = sc.g;
  p.mode = mode;
  p.fn = pick(g.scan_mode, g.cos_mode, mode);
  p.list_fn = p.list ? pick_list(g.scan_mode, g.cos_mode, mode) : nullptr;
  int optin = 0, per_sm = 0;
  cudaFuncAttributes fa{};
  cudaError_t e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, sc.device);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, p.fn);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(p.fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             optin - (int)fa.sharedSizeBytes);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, p.fn, 1024, p.smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  p.grid = (unsigned)std::min<unsigned long long>((unsigned long long)sc.num_sms * per_sm, p.a.units);
  // chunks of units claimed by the CTAs where there is no list: about
  // NLOS_FWD_CHUNKS_PER_CTA per CTA, but at least 8 units (a chunk mostly ends
  // in a tile change, whose flush is worth amortising) and at most 64 (finer
  // claims even out the cost of units, which the bounds do not predict), and
  // never so large that some CTA would get none. Measured on the union (32768
  // units: 8 beats 6.7 per chunk) and heightfield (524288 units: 64 beats 108).
  const unsigned long long per_cta =
      p.a.units / ((unsigned long long)p.grid * NLOS_FWD_CHUNKS_PER_CTA);
  p.a.chunk = std::min<unsigned long long>(
      std::min<unsigned long long>(std::max<unsigned long long>(per_cta, 8), 64),
      std::max<unsigned long long>(1, p.a.units / p.grid));
  return cudaSuccess;
}

}  // namespace

void forward_plan_destroy(FwdPlan* p) {
  if (!p) return;
  if (p->list) cudaFree(p->list);
  if (p->a.far_mass) cudaFree(p->a.far_mass);
  delete p;
}

cudaError_t forward_plan_create(SceneImpl& sc) {
  const Geometry& g = sc.g;
  if (g.P == 0 || g.S == 0) return cudaSuccess;
  FwdPlan* p = sc.fwd_plan = new FwdPlan();
  FwdArgs& a = p->a;
  a.pairs = sc.pairs;
  a.scan = sc.scan_fwd;
  a.err = &sc.scratch->err;
  a.boundary = &sc.scratch->boundary_pairs;
  a.pairs_full = &sc.scratch->pairs_full;
  a.pairs_tested = &sc.scratch->pairs_tested;
  a.bounds = sc.bounds;
  a.groups = sc.groups;
  a.tiles = sc.tiles;
  a.next_chunk = &sc.scratch->next_chunk;
  a.n_pairs = (uint32_t)((g.P + 1) / 2);
  a.S = (uint32_t)g.S;
  a.B = g.B;
  a.kbin = (float)((g.scan_mode == NLOS_CONFOCAL ? 2.0 : 1.0) / g.cdt);
  const int mode = forward_mode(sc);
  const bool moments = mode == MODE_SPLAT_MOM;
  if (moments) moment_table(g.sigma, p->mt);
  a.eps = sc.params.boundary_eps;
  if (g.bin_mode == NLOS_BIN_SPLAT) {
    const double s = g.sigma;
    a.inv2s2 = (float)(1.0 / (2.0 * s * s));
    a.norm = (float)(1.0 / (s * std::sqrt(2.0 * 3.14159265358979323846)));
    a.reach = (float)(6.0 * s);
    a.qstep = (float)std::exp(-1.0 / (s * s));
    a.R = 0;
    a.taps[0] = 1.0f;  // the flush writes the histogram unchanged
  } else {
    a.R = jitter_taps(g.sigma, a.taps, kMaxTaps);
    a.R = (a.R - 1) / 2;
    a.replicate = sc.params.jitter_padding == 1;
    if (a.replicate) jitter_tails(a.taps, a.R, a.tail);
  }

  // shared memory: histogram [bw][32] floats + the staged slots + barriers
  int optin = 0;
  cudaError_t e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, sc.device);
  if (e != cudaSuccess) return e;
  // pairs per staged block: NLOS_FWD_PPB, halved while the histogram of a
  // full window (up to 1024 bins) would not fit beside the stages
  a.ppb = NLOS_FWD_PPB;
  a.stages = NLOS_FWD_STAGES;
  while (a.ppb > 256 && (size_t)std::min(g.B, 1024u) * kTile * 4 +
                                a.stages * (size_t)a.ppb * sizeof(PointPair) + 256 >
                            (size_t)optin)
    a.ppb /= 2;
  if (moments) {
    a.ppb = kPairsPerBlock;
    a.stages = 2;
  }
  const uint32_t n_tiles = (uint32_t)((g.S + kTile - 1) / kTile);
  // staged blocks, then full + empty barriers and what each slot holds
  auto stage_bytes = [&]() {
    return a.stages * (size_t)a.ppb * sizeof(PointPair) + 24 * a.stages + 64 + 8 * 32 +
           4 * kRowWords + 4 * kMaxRangedStages + 4 * a.stages * kOccGroups;
  };
  if (moments) {
    // windows of at most kMomRows rows over the bins and J beyond each end
    a.halo = p->mt.J;
    const uint32_t max_bw = (uint32_t)(kMomRows / p->mt.q), bins = g.B + 2u * (uint32_t)p->mt.J;
    a.n_win = (bins + max_bw - 1) / max_bw;
    a.bw = (bins + a.n_win - 1) / a.n_win;
  } else {
    // (256 bytes for the kernel's static shared memory)
    const uint32_t max_bw =
        (uint32_t)(((size_t)optin - 256 - stage_bytes()) / (kTile * 4)) & ~3u;
    a.n_win = (g.B + max_bw - 1) / max_bw;
    a.bw = ((g.B + a.n_win - 1) / a.n_win + 3) & ~3u;
  }
  a.ppb = block_pairs(a.ppb, n_tiles, a.n_win, a.n_pairs, (uint64_t)sc.num_sms);
  p->smem = (moments ? (size_t)kMoments * kMomRows : (size_t)a.bw) * kTile * 4 + stage_bytes();
  a.n_blk = (a.n_pairs + a.ppb - 1) / a.ppb;
  a.units = (unsigned long long)n_tiles * a.n_win * a.n_blk;
  if (moments) {
    e = cudaMalloc(reinterpret_cast<void**>(&a.far_mass), sizeof(float) * g.S);
    if (e != cudaSuccess) {
      a.far_mass = nullptr;
      return e;
    }
  }
  // With block bounds, a first kernel lists the live units and the forward
  // claims chunks of that list: a chunk then holds NLOS_FWD_LIST_MIN.. units
  // that all carry work (mostly of one tile), instead of a fixed run of
  // units of which most may be culled, so tile changes (flush, zeroing,
  // barriers) are fewer per unit of work. Without memory for it the producers
  // test the units themselves.
  p->pass_runs = list_pass_runs(a.units / a.n_blk, a.n_blk);
  if (NLOS_FWD_CULL && mode != MODE_NEAREST_COUNT && a.units < (1ull << 32) &&
      cudaMalloc(reinterpret_cast<void**>(&p->list),
                 sizeof(ListEntry) * p->pass_runs * a.n_blk) != cudaSuccess) {
    p->list = nullptr;
    (void)cudaGetLastError();
  }
  a.unit_list = p->list;
  while (((a.units * (a.ppb / kGroupPairs)) >> a.list_shift) >= (1ull << 31)) ++a.list_shift;
  a.n_live = &sc.scratch->n_live;
  a.list_chunks_per_cta = NLOS_FWD_LIST_CHUNKS_PER_CTA;
  a.list_min_chunk = NLOS_FWD_LIST_MIN;
  a.list_max_chunk = NLOS_FWD_LIST_MAX;
  // a moment flush costs as much as several units, so its list goes out in
  // one range per CTA (static 60 / 85 / 100%: 0.72 / 0.69 / 0.66 ms on the
  // 64 x 64 scan of 65,536 points at sigma = 3.2, 0.17 / 0.19 / 0.13 ms on the 32 x 32
  // scan of 16,384 points at sigma = 1.6)
  a.list_static_pct = moments ? NLOS_FWD_MOM_STATIC : NLOS_FWD_LIST_STATIC;
  return plan_mode(*p, sc, mode);
}

cudaError_t launch_forward(const SceneImpl& sc, float* tau, cudaStream_t st) {
  const Geometry& g = sc.g;
  FwdPlan* p = sc.fwd_plan;
  cudaError_t e = cudaSuccess;
  if (p && p->mode != forward_mode(sc) &&
      (e = plan_mode(*p, sc, forward_mode(sc))) != cudaSuccess)
    return e;
  const uint64_t runs = p ? p->a.units / p->a.n_blk : 0;
  const bool listed = p && p->list_fn;
  const bool one_pass = listed && p->pass_runs == runs;  // whose list kernel zeroes the output
  if (e == cudaSuccess && !one_pass) e = cudaMemsetAsync(tau, 0, sizeof(float) * g.S * g.B, st);
  if (e == cudaSuccess && !one_pass && p && p->a.far_mass)
    e = cudaMemsetAsync(p->a.far_mass, 0, sizeof(float) * g.S, st);
  if (e != cudaSuccess || !p) return e;
  FwdArgs a = p->a;
  a.tau = tau;
  a.list_zeroes = one_pass ? 1u : 0u;
  static_assert(offsetof(SceneScratch, n_live) == offsetof(SceneScratch, next_chunk) + 8,
                "zeroed together");
  // (the first pass finds its counters zeroed with the call's scratch)
  for (uint64_t r = 0; r < (listed ? runs : 1); r += p->pass_runs) {
    if (listed) {
      a.list_tw0 = r;
      if (r > 0 && (e = cudaMemsetAsync(a.next_chunk, 0, 2 * sizeof(unsigned long long), st)) !=
                       cudaSuccess)
        return e;
      p->list_fn<<<(unsigned)std::min(p->pass_runs, runs - r), a.n_blk < 128 ? 256 : kListThreads,
                   0, st>>>(a, p->list, &sc.scratch->n_live);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    p->fn<<<p->grid, 1024, p->smem, st>>>(a, p->mt, sc.occ);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (p->mode == MODE_SPLAT_MOM) {
    const unsigned blocks = (unsigned)std::min<uint64_t>((g.S + 7) / 8, (uint64_t)sc.num_sms * 8);
    pick_tail(g.scan_mode, g.cos_mode)<<<blocks, 256, 0, st>>>(a);
    e = cudaGetLastError();
  }
  return e;
}

cudaError_t launch_pair_table(const SceneImpl& sc, uint64_t s_begin, uint64_t s_count, float* u,
                              float* w, cudaStream_t st) {
  const Geometry& g = sc.g;
  const uint32_t n_pairs = (uint32_t)((g.P + 1) / 2);
  const uint64_t total = s_count * n_pairs;
  if (total == 0) return cudaSuccess;
  const float kbin = (float)((g.scan_mode == NLOS_CONFOCAL ? 2.0 : 1.0) / g.cdt);
  const unsigned blocks = (unsigned)((total + 255) / 256);
  PairTableArgs t{sc.raw_points, &sc.scratch->err, n_pairs, (uint32_t)g.P, g.scan_mode,
                  g.cos_mode, pack_const(sc.params.laser_x, sc.params.laser_y, 1.0 / g.cdt)};
#define NLOS_PT(SC, CO) \
  pair_table_kernel<SC, CO><<<blocks, 256, 0, st>>>(t, sc.scan, s_begin, s_count, kbin, u, w)
  if (g.scan_mode == NLOS_CONFOCAL) {
    if (g.cos_mode == NLOS_COS_NONE) NLOS_PT(NLOS_CONFOCAL, NLOS_COS_NONE);
    else if (g.cos_mode == NLOS_COS_OBJECT) NLOS_PT(NLOS_CONFOCAL, NLOS_COS_OBJECT);
    else NLOS_PT(NLOS_CONFOCAL, NLOS_COS_OBJECT_WALL);
  } else {
    if (g.cos_mode == NLOS_COS_NONE) NLOS_PT(NLOS_NONCONFOCAL, NLOS_COS_NONE);
    else if (g.cos_mode == NLOS_COS_OBJECT) NLOS_PT(NLOS_NONCONFOCAL, NLOS_COS_OBJECT);
    else NLOS_PT(NLOS_NONCONFOCAL, NLOS_COS_OBJECT_WALL);
  }
#undef NLOS_PT
  return cudaGetLastError();
}

}  // namespace nlos

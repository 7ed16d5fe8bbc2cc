// Spatial ordering of a scene's surface points, packing in that order, and
// the per-block bounds the forward kernel uses to skip (tile, block) units
// that cannot reach the acquisition window or face no spot of the tile.
//
// Ordering: a counting sort by the Morton index of a 32 x 32 x 32 grid of
// cells over the points' bounding box (cells in Z-order, points of a cell in
// arbitrary order), so that a packed block of 512 points covers a small part
// of the surface. The sum over points does not depend on the order; only the
// FP32 rounding of the histogram accumulation does.
//
// Two launches on one stream, without host synchronisation (the step routines
// are in order_core.cuh, shared with the serving kernel):
//   order_kernel, a cooperative launch whose CTAs meet at three grid barriers:
//     1. box: the points' bounding box (order-preserving integer atomics),
//     2. cell: each point's cell and the cell counts,
//     3. scan: exclusive prefix sums of the counts within slices of 1024 cells,
//     4. scatter: perm[slot] = point, the slot from the cell's cursor and the
//        slices before it;
//   pack_bounds_kernel: pack (pack_pair through perm), group and sub-block bounds
//     (one CTA per sub-block), and the counts and box words set up for the next
//     ordering.
// The steps are short whatever the point count, so what they cost is launches
// and latency: as six kernels 45 us for 262,144 points and 32 us for 40,001.
// The barriers need every CTA resident, which a cooperative launch promises on
// the context's SMs. On a stream of a green context, which may have only some of
// them, and where the launch is refused, the same four steps are four launches of
// their own.
#include "common.cuh"
#include "order_core.cuh"
#include "device_util.cuh"
#include "pack_core.cuh"

#include <cuda.h>

#include <algorithm>
#include <cmath>
#include <vector>

namespace nlos {

namespace {

// Words behind the counts: the box (6), the grid barrier, padding, slice totals.
constexpr uint32_t kBarrierWord = 6;
static_assert(kOrderCells / kSliceCells == 32 && kBarrierWord < kOrderBoxWords, "ordering scratch");

// All CTAs of the (cooperative) grid arrive before any leaves; the word counts
// the arrivals of a launch's barriers from zero. Bounded: false after about a
// second (the error is in *err).
__device__ __forceinline__ bool grid_barrier(uint32_t* word, unsigned int* err) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const uint32_t target = (atomicAdd(word, 1u) / gridDim.x + 1u) * gridDim.x;
    int ok = 1;
    const long long t0 = clock64();
    while ((int32_t)(*(volatile uint32_t*)word - target) < 0)
      if (clock64() - t0 > kWaitCycles) {
        atomicOr(err, kErrWaitTimeout);
        ok = 0;
        break;
      }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

constexpr int kOrderThreads = 512;

// GRID: all steps with grid barriers between them (a cooperative launch); else
// the one step `step`.
template <bool GRID>
__global__ void __launch_bounds__(kOrderThreads, 2)
    order_kernel(const float* __restrict__ raw, uint64_t P, int scan_mode, int cos_mode,
                 const PackConst pc, uint16_t* cell, uint32_t* counts, uint32_t* perm,
                 unsigned int* err, int step) {
  __shared__ uint32_t red[kOrderThreads / 32 * 6];
  __shared__ uint32_t base[kOrderCells / kSliceCells];
  uint32_t* box = counts + kOrderCells;
  uint32_t* totals = box + kOrderBoxWords;
  const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (GRID || step == 0) box_range(raw, 0, P, t, stride, box, red);
  if (GRID && !grid_barrier(box + kBarrierWord, err)) return;
  if (GRID || step == 1)
    cell_range(raw, 0, P, t, stride, box, cell, counts, scan_mode, cos_mode, pc);
  if (GRID && !grid_barrier(box + kBarrierWord, err)) return;
  // a warp scans 64 cells of a slice, then the 16 warp totals are scanned
  for (uint32_t sl = GRID || step == 2 ? blockIdx.x : kOrderCells;
       sl < kOrderCells / kSliceCells; sl += gridDim.x) {
    uint32_t* seg = counts + sl * kSliceCells + w * 64;
    const uint32_t v0 = seg[lane], v1 = seg[32 + lane];
    const uint32_t x0 = inclusive_scan(v0);
    const uint32_t x1 = inclusive_scan(v1) + __shfl_sync(0xffffffffu, x0, 31);
    if (lane == 31) red[w] = x1;
    __syncthreads();
    if (w == 0) {
      const uint32_t v = lane < kOrderThreads / 32 ? red[lane] : 0u;
      const uint32_t x = inclusive_scan(v);
      red[lane] = x - v;
      if (lane == 31) totals[sl] = x;
    }
    __syncthreads();
    seg[lane] = red[w] + x0 - v0;
    seg[32 + lane] = red[w] + x1 - v1;
    __syncthreads();
  }
  if (GRID && !grid_barrier(box + kBarrierWord, err)) return;
  if (!GRID && step != 3) return;
  if (w == 0) {
    const uint32_t v = *(volatile uint32_t*)&totals[lane];
    base[lane] = inclusive_scan(v) - v;
  }
  __syncthreads();
  scatter_range(cell, 0, P, t, stride, counts, perm, base, P);
}

// One CTA of kSubPairs threads per sub-block: thread k packs pair k of the
// sub-block, and the CTA reduces the bounds of its 2 kSubPairs points (the
// quantities of block_bound_warp, read off the packed record: the same
// laser-leg offsets, and liveness from the packed weight factor).
__global__ void __launch_bounds__(kSubPairs) pack_bounds_kernel(
    const float* __restrict__ raw, uint64_t P, int scan_mode, int cos_mode, const PackConst pc,
    const uint32_t* __restrict__ perm, PointPair* pairs, unsigned int* err,
    BlockBound* bounds, BlockBound* groups, uint32_t* counts, const __grid_constant__ OccSet occ) {
  static_assert(kSubPairs % 32 == 0 && kSubPairs <= 1024, "one thread per pair of a sub-block");
  __shared__ float red[kSubPairs / 32][15];
  // the counts, the box words and the barrier for the next ordering
  for (uint32_t i = blockIdx.x * kSubPairs + threadIdx.x; i < kOrderCells + kOrderBoxWords;
       i += gridDim.x * kSubPairs)
    counts[i] = i >= kOrderCells && i < kOrderCells + 3 ? 0xffffffffu : 0u;
  const uint64_t n_pairs = (P + 1) / 2;
  const uint64_t k = (uint64_t)blockIdx.x * kSubPairs + threadIdx.x;
  // only the laser leg of a non-confocal scan is tested here
  const OccSet* o = (occ.n > 0 && scan_mode == NLOS_NONCONFOCAL) ? &occ : nullptr;
  float lo[7], hi[7], live = 0.f;
  for (int c = 0; c < 7; ++c) {
    lo[c] = 3.0e38f;
    hi[c] = -3.0e38f;
  }
  if (k < n_pairs) {
    float rv[2][8];
    const PointPair pp = pack_pair_value(raw, P, k, scan_mode, cos_mode, pc, err, perm, o, rv);
    pairs[k] = pp;
    // the bounds from the packed record and the raw values already loaded:
    // the laser-leg offset as packed, and "can carry weight" as a nonzero
    // packed weight factor (zero for albedo or area 0, a point facing away
    // from the laser, or one hidden from it)
    for (int h = 0; h < 2 && 2 * k + h < P; ++h) {
      const float* r = rv[h];
      const float kq = h ? pp.kq.y : pp.kq.x, na = h ? pp.na.y : pp.na.x;
      const float nb = h ? pp.nb.y : pp.nb.x, nc = h ? pp.nc.y : pp.nc.x;
      const float v[7] = {r[0], r[1], r[2], r[3], r[4], r[5], h ? pp.uoff.y : pp.uoff.x};
      for (int c = 0; c < 7; ++c) {
        lo[c] = fminf(lo[c], v[c]);
        hi[c] = fmaxf(hi[c], v[c]);
      }
      if (kq != 0.f || na != 0.f || nb != 0.f || nc != 0.f) live = 1.f;
    }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // half a warp is one group
  static_assert(kGroupPairs == 16, "one group per half warp");
  bound_warp_reduce<16>(lo, hi, live);
  if ((lane & 15) == 0 && k < n_pairs) groups[k / kGroupPairs] = bound_record(lo, hi, live);
  bound_combine(lo, hi, live, 16);
  if (lane == 0) {
    for (int c = 0; c < 7; ++c) {
      red[warp][c] = lo[c];
      red[warp][7 + c] = hi[c];
    }
    red[warp][14] = live;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kSubPairs / 32; ++w) {
      for (int c = 0; c < 7; ++c) {
        lo[c] = fminf(lo[c], red[w][c]);
        hi[c] = fmaxf(hi[c], red[w][7 + c]);
      }
      live = fmaxf(live, red[w][14]);
    }
    bounds[blockIdx.x] = bound_record(lo, hi, live);
  }
}

// Whether a stream belongs to a green context (or the driver does not say).
bool partitioned(cudaStream_t st) {
  using StreamGetCtx = decltype(&cuStreamGetCtx_v2);
  static const StreamGetCtx stream_ctx = [] {
    void* q = nullptr;
    cudaDriverEntryPointQueryResult r = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuStreamGetCtx", &q, 13000, cudaEnableDefault, &r) ==
            cudaSuccess &&
        r == cudaDriverEntryPointSuccess)
      return reinterpret_cast<StreamGetCtx>(q);
    (void)cudaGetLastError();
    return StreamGetCtx(nullptr);
  }();
  CUcontext ctx = nullptr;
  CUgreenCtx green = nullptr;
  return !stream_ctx || stream_ctx(st, &ctx, &green) != CUDA_SUCCESS || green;
}

}  // namespace

cudaError_t init_order(SceneImpl& s, cudaStream_t st) {
  if (s.g.P == 0) return cudaSuccess;
  uint32_t* box = s.cells + kOrderCells;
  cudaError_t e = cudaMemsetAsync(s.cells, 0, sizeof(uint32_t) * kOrderWords, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(box, 0xff, 3 * sizeof(uint32_t), st);
  // (a valid order even if an ordering gave up at a barrier)
  if (e == cudaSuccess) e = cudaMemsetAsync(s.perm, 0, sizeof(uint32_t) * s.g.P, st);
  return e;
}

cudaError_t launch_order_pack(SceneImpl& s, cudaStream_t st) {
  const Geometry& g = s.g;
  const uint64_t P = g.P;
  if (P == 0) return cudaSuccess;
  uint32_t* counts = s.cells;
  const PackConst pc = pack_const(s.params.laser_x, s.params.laser_y, 1.0 / g.cdt);
  // one wave, at least a CTA a slice
  const uint64_t want =
      std::max<uint64_t>((P + kOrderThreads - 1) / kOrderThreads, kOrderCells / kSliceCells);
  const unsigned grid = (unsigned)std::min<uint64_t>(want, 2ull * (unsigned)s.num_sms);
  unsigned int* err = &s.scratch->err;
  cudaError_t e = cudaErrorCooperativeLaunchTooLarge;
  if (!partitioned(st)) {
    uint64_t n = P;
    int scan_mode = g.scan_mode, cos_mode = g.cos_mode, step = 0;
    void* args[] = {&s.raw_points, &n, &scan_mode, &cos_mode, const_cast<PackConst*>(&pc),
                    &s.cell, &counts, &s.perm, &err, &step};
    e = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(&order_kernel<true>), dim3(grid),
                                    dim3(kOrderThreads), args, 0, st);
  }
  if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
    (void)cudaGetLastError();
    e = cudaSuccess;
    for (int step = 0; step < 4 && e == cudaSuccess; ++step) {
      order_kernel<false><<<grid, kOrderThreads, 0, st>>>(s.raw_points, P, g.scan_mode, g.cos_mode,
                                                          pc, s.cell, counts, s.perm, err, step);
      e = cudaGetLastError();
    }
  }
  if (e != cudaSuccess) return e;
  const uint64_t n_pairs = (P + 1) / 2;
  const uint64_t n_sub = (n_pairs + kSubPairs - 1) / kSubPairs;
  pack_bounds_kernel<<<(unsigned)n_sub, kSubPairs, 0, st>>>(
      s.raw_points, P, g.scan_mode, g.cos_mode, pc, s.perm, s.pairs, &s.scratch->err,
      s.bounds, s.groups, counts, s.occ);
  return cudaGetLastError();
}

void tile_bounds_host(const ScanPoint* sp, uint64_t S, std::vector<TileBound>& out) {
  const uint64_t n = (S + kTile - 1) / kTile;
  out.assign(n, TileBound{});
  for (uint64_t t = 0; t < n; ++t) {
    TileBound b{3.0e38f, -3.0e38f, 3.0e38f, -3.0e38f, 3.0e38f, -3.0e38f, 0.f, 0.f};
    for (uint64_t s = t * kTile; s < std::min(S, (t + 1) * kTile); ++s) {
      b.sx0 = std::min(b.sx0, sp[s].sx);
      b.sx1 = std::max(b.sx1, sp[s].sx);
      b.sy0 = std::min(b.sy0, sp[s].sy);
      b.sy1 = std::max(b.sy1, sp[s].sy);
      b.off0 = std::min(b.off0, sp[s].off);
      b.off1 = std::max(b.off1, sp[s].off);
    }
    out[t] = b;
  }
}

}  // namespace nlos

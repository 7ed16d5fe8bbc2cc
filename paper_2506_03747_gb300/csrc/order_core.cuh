// Device steps of the spatial ordering of surface points (a counting sort by
// the Morton index of a 32 x 32 x 32 grid of cells over the points' bounding
// box), written as CTA-wide routines over a range of points so that both the
// standalone kernels (order.cu) and the persistent serving kernel (one range
// per work item) run them:
//   box_range      bounding box (order-preserving integer min/max atomics),
//   cell_range     each point's cell and the cell counts,
//   scan_cells     exclusive prefix sum of the counts (one CTA of 1024 threads),
//   scatter_range  perm[slot] = point, the slot from the cell's cursor.
#pragma once

#include "common.cuh"
#include "pack_core.cuh"

namespace nlos {

// float -> unsigned with the same order
__host__ __device__ inline uint32_t ord_bits(float f) {
  uint32_t b;
  memcpy(&b, &f, 4);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__host__ __device__ inline float ord_float(uint32_t u) {
  const uint32_t b = (u & 0x80000000u) ? (u & 0x7fffffffu) : ~u;
  float f;
  memcpy(&f, &b, 4);
  return f;
}

__host__ __device__ inline uint32_t spread5(uint32_t v) {
  uint32_t o = 0;
  for (int b = 0; b < 5; ++b) o |= ((v >> b) & 1u) << (3 * b);
  return o;
}

__host__ __device__ inline uint32_t cell_of(float x, float y, float z, const float* lo,
                                            const float* inv) {
  const float v[3] = {x, y, z};
  uint32_t q[3];
  for (int c = 0; c < 3; ++c) {
    const float t = (v[c] - lo[c]) * inv[c];
    q[c] = t > 0.f ? (uint32_t)fminf(t, 31.f) : 0u;
  }
  return spread5(q[0]) | (spread5(q[1]) << 1) | (spread5(q[2]) << 2);
}

__host__ __device__ inline void box_scale(const float* lo, const float* hi, float* inv) {
  for (int c = 0; c < 3; ++c) {
    const float ext = hi[c] - lo[c];
    inv[c] = ext > 0.f ? 32.0f / ext : 0.f;
  }
}

// Words of the ordering scratch after the kOrderCells counts: min x, y, z and
// max x, y, z as ord_bits (initialised to all ones / zero), then padding.
constexpr uint32_t kOrderBoxWords = 8;

// Points [b, e), thread t0 of a grid-stride of `stride` threads; red: shared
// scratch of 6 words per warp of the CTA. All threads of the CTA call it.
__device__ __forceinline__ void box_range(const float* __restrict__ raw, uint64_t b, uint64_t e,
                                          uint64_t t0, uint64_t stride, uint32_t* box,
                                          uint32_t* red) {
  uint32_t mn[3] = {0xffffffffu, 0xffffffffu, 0xffffffffu}, mx[3] = {0u, 0u, 0u};
  for (uint64_t i = b + t0; i < e; i += stride) {
    for (int c = 0; c < 3; ++c) {
      const uint32_t u = ord_bits(raw[8 * i + c]);
      mn[c] = min(mn[c], u);
      mx[c] = max(mx[c], u);
    }
  }
  for (int o = 16; o > 0; o >>= 1)
    for (int c = 0; c < 3; ++c) {
      mn[c] = min(mn[c], __shfl_xor_sync(0xffffffffu, mn[c], o));
      mx[c] = max(mx[c], __shfl_xor_sync(0xffffffffu, mx[c], o));
    }
  // CTA reduction first: one global atomic per CTA and word (same-address
  // atomics from every warp serialise)
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0)
    for (int c = 0; c < 3; ++c) {
      red[w * 6 + c] = mn[c];
      red[w * 6 + 3 + c] = mx[c];
    }
  __syncthreads();
  if (threadIdx.x < 6) {
    const int c = threadIdx.x;
    uint32_t v = red[c];
    for (int j = 1; j < (int)(blockDim.x >> 5); ++j)
      v = c < 3 ? min(v, red[j * 6 + c]) : max(v, red[j * 6 + c]);
    if (c < 3) atomicMin(&box[c], v);
    else atomicMax(&box[c], v);
  }
  __syncthreads();
}

// Can a point carry weight? False only where its packed weight factor is zero:
// albedo or area 0, or (non-confocal scans with object cosines) facing away
// from the laser spot, by the arithmetic of pack_pair_value.
__device__ __forceinline__ bool point_live(const float4& r0, const float4& r1, int scan_mode,
                                           int cos_mode, const PackConst& pc) {
  bool live = r1.z * r1.w != 0.f;
  if (scan_mode == NLOS_NONCONFOCAL && cos_mode != NLOS_COS_NONE) {
    const LaserLeg g = laser_leg(r0.x, r0.y, r0.z, pc);
    live = live && -fmaf(r0.w, g.vx, fmaf(r1.x, g.vy, r1.y * r0.z)) > 0.f;
  }
  return live;
}

// Points that carry no weight go to the last cells (kDeadCells of them, so
// that their counters are not one address), so that whole blocks of them are
// ruled out by their bounds.
constexpr uint32_t kDeadCells = 64;

__device__ __forceinline__ void cell_range(const float* __restrict__ raw, uint64_t b, uint64_t e,
                                           uint64_t t0, uint64_t stride, const uint32_t* box,
                                           uint16_t* cell, uint32_t* counts, int scan_mode,
                                           int cos_mode, const PackConst& pc) {
  float lo[3], hi[3], inv[3];
  for (int c = 0; c < 3; ++c) {
    lo[c] = ord_float(box[c]);
    hi[c] = ord_float(box[3 + c]);
  }
  box_scale(lo, hi, inv);
  for (uint64_t i = b + t0; i < e; i += stride) {
    float r[8];
    load_point(raw + 8 * i, r);
    const float4 r0 = make_float4(r[0], r[1], r[2], r[3]), r1 = make_float4(r[4], r[5], r[6], r[7]);
    const uint32_t k = point_live(r0, r1, scan_mode, cos_mode, pc)
                           ? cell_of(r0.x, r0.y, r0.z, lo, inv)
                           : kOrderCells - kDeadCells + (uint32_t)(i / 32 % kDeadCells);
    cell[i] = (uint16_t)k;
    // one atomic per distinct cell of the warp: points given in grid or scan
    // order put a warp's 32 points in one or two cells, whose counter the
    // lanes would otherwise increment one after the other
    const unsigned peers = __match_any_sync(__activemask(), k);
    if ((threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&counts[k], (uint32_t)__popc(peers));
  }
}

// Inclusive prefix sum over a warp.
__device__ __forceinline__ uint32_t inclusive_scan(uint32_t x) {
  const int lane = threadIdx.x & 31;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// counts[c] <- sum of counts[0..c). One CTA of exactly 1024 threads: warp w
// scans cells [w * 1024, (w + 1) * 1024) 32 at a time (coalesced loads,
// shuffle scans), then the 32 warp totals are scanned; wsum: 32 shared words.
__device__ __forceinline__ void scan_cells(uint32_t* counts, uint32_t* wsum) {
  constexpr int kPerWarp = kOrderCells / 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t* seg = counts + (size_t)w * kPerWarp;
  uint32_t carry = 0;
  for (int j = 0; j < kPerWarp; j += 32) {
    const uint32_t v = seg[j + lane];
    const uint32_t x = inclusive_scan(v);
    seg[j + lane] = carry + x - v;  // exclusive within the warp's segment
    carry += __shfl_sync(0xffffffffu, x, 31);
  }
  if (lane == 0) wsum[w] = carry;
  __syncthreads();
  if (w == 0) {
    const uint32_t v = wsum[lane];
    wsum[lane] = inclusive_scan(v) - v;
  }
  __syncthreads();
  const uint32_t base = wsum[w];
  for (int j = lane; j < kPerWarp; j += 32) seg[j] += base;
  __syncthreads();
}

// The lanes of one cell take consecutive slots from one atomic on its cursor.
// base (nullable): added to the cursors of each kSliceCells cells.
constexpr uint32_t kSliceCells = 1024;
__device__ __forceinline__ void scatter_range(const uint16_t* cell, uint64_t b, uint64_t e,
                                              uint64_t t0, uint64_t stride, uint32_t* cursor,
                                              uint32_t* perm, const uint32_t* base_of = nullptr,
                                              uint64_t limit = ~0ull) {
  const uint32_t lane = threadIdx.x & 31;
  for (uint64_t i = b + t0; i < e; i += stride) {
    const uint32_t k = cell[i];
    const unsigned peers = __match_any_sync(__activemask(), k);
    const int leader = __ffs(peers) - 1;
    uint32_t base = 0;
    if ((int)lane == leader) base = atomicAdd(&cursor[k], (uint32_t)__popc(peers));
    base = __shfl_sync(peers, base, leader);
    const uint32_t slot = base + (uint32_t)__popc(peers & ((1u << lane) - 1u)) +
                          (base_of ? base_of[k / kSliceCells] : 0u);
    if (slot < limit) perm[slot] = (uint32_t)i;
  }
}

}  // namespace nlos

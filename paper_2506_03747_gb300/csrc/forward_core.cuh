// Device core of the forward transient: the (scan point, surface point)
// pair sum of the generalised Eq. 1 of Shi et al. (arXiv 2506.03747),
// accumulated per scan point as a histogram over time bins, with the Gaussian
// jitter of Eq. 16/17 fused into the write-out, or as the differentiable
// Gaussian splat. Shared by the standalone forward kernel (forward.cu) and
// the persistent serving kernel (serve.cu), so both run identical arithmetic.
//
// Layout and schedule (GB300, sm_103a):
//  * One tile = 32 scan points; lane l of every warp owns scan point l of the
//    tile, so the shared histogram [bin][32] gives every lane its own bank and
//    the shared atomics of a warp never conflict.
//  * Surface points are packed in pairs (64 B, PointPair) and staged into
//    shared memory by 1-D TMA bulk copies, into a few slots on mbarriers. All
//    consumer warps of the CTA read the same slot (broadcast loads) and split
//    its pairs; each lane evaluates the two points of a pair for its scan
//    point with packed FP32x2 arithmetic (__ffma2_rn & co.).
//  * A work unit is (scan tile, bin window, point block). A CTA flushes its
//    partial histogram into the zeroed output with vectorised global reductions
//    whenever its (tile, window) changes; the jitter convolution is linear, so
//    it is applied to each partial histogram during the flush.
#pragma once

#include "common.cuh"
#include "device_util.cuh"
#include "rules.h"

#include <cmath>

namespace nlos {

constexpr float kMagic = 12582912.0f;       // 1.5 * 2^23: floor via round-down add
constexpr int kMagicBits = 0x4B400000;      // bit pattern of kMagic
constexpr int kMaxTaps = 129;               // fused jitter: R <= 64
constexpr int kPairsPerBlock = 256;         // serving kernel: 16 KB per staged block
#ifndef NLOS_FWD_PPB
#define NLOS_FWD_PPB 512                    // standalone forward: pairs per staged block
#endif
#ifndef NLOS_FWD_SQRT_RCP
#define NLOS_FWD_SQRT_RCP 1                 // r from sqrt.approx, weights from one rcp.approx
#endif
#ifndef NLOS_FWD_CULL
#define NLOS_FWD_CULL 1                     // skip (tile, block) units the bounds rule out
#endif
#ifndef NLOS_FWD_EARLY
#define NLOS_FWD_EARLY 0                    // warp-uniform early out before the square roots
#endif
#ifndef NLOS_FWD_VOTE
#define NLOS_FWD_VOTE 0                     // 2: warp-uniform skip before the reductions
#endif
#ifndef NLOS_FWD_CHUNKS_PER_CTA
#define NLOS_FWD_CHUNKS_PER_CTA 32          // standalone forward: claimed chunks per CTA (mean)
#endif
#ifndef NLOS_FWD_LIST_CHUNKS_PER_CTA
#define NLOS_FWD_LIST_CHUNKS_PER_CTA 6      // live-unit list: chunks per CTA (mean)
#endif
#ifndef NLOS_FWD_LIST_MIN
#define NLOS_FWD_LIST_MIN 2                 // live-unit list: entries per chunk, at least
#endif
#ifndef NLOS_FWD_LIST_STATIC
#define NLOS_FWD_LIST_STATIC 75             // live-unit list: percent in static ranges per CTA
#endif
#ifndef NLOS_FWD_LIST_MAX
#define NLOS_FWD_LIST_MAX 32                // ... and at most
#endif
#ifndef NLOS_FWD_MOM_STATIC
#define NLOS_FWD_MOM_STATIC 100             // the same for the moment form, whose flushes cost more
#endif
#ifndef NLOS_FWD_STAGES
#define NLOS_FWD_STAGES 3                   // staged blocks in flight (warp-specialised)
#endif
#ifndef NLOS_FWD_UNROLL
#define NLOS_FWD_UNROLL 4                   // standalone forward: unroll of the pair loop
#endif

constexpr int kFwdUnroll = NLOS_FWD_UNROLL;  // (#pragma unroll takes no macro)

enum { MODE_NEAREST = 0, MODE_NEAREST_COUNT = 1, MODE_SPLAT = 2, MODE_SPLAT_MOM = 3,
       MODE_NEAREST_OCC = 4 /* NEAREST with the occluder visibility test */ };

// Moment form of the splat (standalone forward and adjoint): the bins are cut
// into q rows each (q a power of two), and with v = u q, row = floor(v) and
// c = 1/2 - (v - row), a pair adds w c^n, n < kMoments, to its row's moments;
// at flush time
//   tau[b] = sum_n sum_r D_n[r - q b + q J] M_n[r],
//   D_n[i] = K^(n)(X_i) / (n! q^n),  X_i = 1/2 - (i - q J + 1/2) / q,
// the Taylor expansion of the Gaussian K about the row's centre. q makes half
// a row at most 0.16 sigma (0.2 sigma, one row a bin, from sigma = 2.5 up), so
// that six moments leave a truncation error of at most 3.5e-7 of the kernel's
// peak (1.3e-6 at sigma = 2.5, 3.1e-7 at 3.2). The shared histogram of each
// moment has kMomRows rows: a window of kMomRows / q bins, and a flush writes
// the bins up to J beyond its window. The windows reach J = ceil(6 sigma) + 1
// bins beyond [0, B), and a bin takes all of the J bins around it, so up to
// 1.5e-8 of the peak of a pair beyond the splat's cut at |x| = 6 sigma. Where
// that could show, in a transient that holds little but the cut tails of
// pairs beyond its ends, splat_tail_kernel sums the taps instead. A pair costs six shared reductions at
// any sigma, against 12 sigma of its taps: a 32 x 32 scan of 16,384 points at
// sigma = 1.6 takes 0.139 ms against 2.63 ms pair by pair (forward_moments says
// where the taps remain the better form). Fewer moments on
// finer rows (five at 0.1 sigma, four at 0.05) reduce less a pair but cut the
// windows into more: 0.74 and 0.79 ms against 0.68 ms (64 x 64 scan, 65,536
// points, sigma = 3.2).
constexpr int kMoments = 6;       // of the forward
constexpr int kMomTerms = 8;      // terms of the table (the adjoint takes them all)
constexpr int kMomRows = 256;
constexpr uint32_t kMomStride = kMomRows * 32 * 4;  // bytes between moment histograms
struct __align__(16) MomTab {
  int J, q;
  float d[kMomTaps][kMomTerms];  // D_n[i] as d[i][n]
};

// Fills mt for the unit-area Gaussian of standard deviation s bins (host).
void moment_table(double s, MomTab& mt);

// Per-thread counters of one forward run, added to the scene scratch at exit.
struct FwdCount {
  unsigned long long boundary = 0;  // pairs within eps of a bin edge (count mode)
  unsigned long long full = 0;      // warp iterations past the early out (x 64 pairs)
  unsigned long long tested = 0;    // warp iterations of staged units (x 64 pairs)
};

// A live unit: its number, the histogram rows it can touch (unit_rows), its live
// groups (unit_groups), and the weight of the list before it.
struct __align__(16) ListEntry {
  uint32_t unit, rows, groups, before;
};

struct FwdArgs {
  const PointPair* pairs;
  const ScanPoint* scan;
  float* tau;
  unsigned int* err;
  unsigned long long* boundary;
  unsigned long long* pairs_full;  // pairs past the early out (scene scratch)
  unsigned long long* pairs_tested;  // pairs of staged units (scene scratch)
  const BlockBound* bounds;   // [ceil(n_pairs / kSubPairs)] or null (no unit culling)
  const BlockBound* groups;   // [ceil(n_pairs / kGroupPairs)], with bounds
  const TileBound* tiles;     // [ceil(S / kTile)]
  unsigned long long* next_chunk;  // standalone launch: chunk counter (zeroed per pass)
  unsigned long long units;   // standalone launch: total units
  unsigned long long chunk;   // standalone launch: units per claimed chunk
  // standalone launch with a unit list (unit_list_kernel): *n_live packs its
  // entries (low word) and their weight (high word: live groups >> list_shift);
  // chunks of the list are claimed instead of chunks of units (null: no list)
  const ListEntry* unit_list;
  const unsigned long long* n_live;
  uint32_t list_shift;
  uint32_t list_chunks_per_cta;  // list chunks per CTA (mean), of the claimed part
  uint32_t list_min_chunk, list_max_chunk;  // list entries per chunk, clamped
  uint32_t list_static_pct;  // the list's first part (percent of weight) in one range per CTA
  uint32_t n_pairs, S, B, bw, n_win, n_blk, ppb;
  int halo;          // bins the windows reach beyond [0, B) on each side (moment form: J)
  uint32_t stages;   // staged point blocks (standalone warp-specialised kernel)
  float kbin;        // bins per metre of the scanned leg
  int R;             // jitter radius (NEAREST); 0 = none
  float eps;         // boundary-count tolerance (MODE_NEAREST_COUNT)
  float inv2s2;      // splat: 1 / (2 sigma^2)
  float norm;        // splat: 1 / (sigma sqrt(2 pi))
  float reach;       // splat: 6 sigma
  float qstep;       // splat: exp(-1 / sigma^2)
  float* far_mass;   // moment form: [S] weight of the pairs beyond a transient's ends (zeroed)
  float taps[kMaxTaps];
  int replicate;     // jitter with the edge bins continued outside the window
  float tail[kMaxTaps / 2 + 1];  // replicate corrections (jitter_tails)
  // the list's kernel: first (tile, window) of the pass, and whether it zeroes the
  // output (of a list in one pass)
  unsigned long long list_tw0;
  uint32_t list_zeroes;
};

struct bool2_t {
  bool x, y;
};

// Path-bin coordinate u and weight w of the two points of a pair for one scan
// spot (sx, sy, 0) with bin offset off (FP32x2: component i = point i).
//   r^2 = (px - sx)^2 + (py - sy)^2 + pz^2,   u = r * kbin + off (+ uoff)
//   cn  = na * (px - sx) + nb * (py - sy) + nc   (object cosine numerator
//         n.(spot - x), prescaled; from the offsets, so nothing cancels)
// Weight by scan and cosine mode (per-point factors folded in at packing):
//   confocal    NONE: kq / r^4        OBJECT: (cn / r^3)^2   WALL: (cn / r^4)^2
//   non-confocal NONE: kq / r^2       OBJECT: cn / r^3       WALL: cn / r^4
// Split in two: pair_geom2 (r^2 and cn: differences and FMAs only) and
// pair_finish2 (square root, u and the weight), so that the caller can skip
// the second part when no lane of the warp can bin either point.
__device__ __forceinline__ void pair_geom2(const PointPair& q, float2 nsx, float2 nsy, float2& r2,
                                           float2& cn) {
  const float2 dx = __fadd2_rn(q.px, nsx);
  const float2 dy = __fadd2_rn(q.py, nsy);
  r2 = __ffma2_rn(dx, dx, q.pz2);
  r2 = __ffma2_rn(dy, dy, r2);
  cn = __ffma2_rn(q.na, dx, q.nc);
  cn = __ffma2_rn(q.nb, dy, cn);
}

// u is formed relative to bin 0 of the transient; callers move it to the
// window by an exact subtraction of the window's first bin (an integer below
// 2^24: in the float for the splat forms, in the integer bin for the binned
// ones), so the bins and splat taps of a pair do not depend on how the bins
// are windowed.
template <int SCAN, int COS>
__device__ __forceinline__ void pair_finish2(const PointPair& q, float2 r2, float2 cn, float2 off,
                                             float2 kbin, float2& u, float2& w) {
  const float2 o = (SCAN == NLOS_CONFOCAL) ? off : __fadd2_rn(off, q.uoff);
#if NLOS_FWD_SQRT_RCP
  // r from the hardware square root; the weight's inverse powers of r from a
  // single reciprocal of r^2k, so no approximation error is raised to a power
  const float2 r = make_float2(sqrt_approx(r2.x), sqrt_approx(r2.y));
  u = __ffma2_rn(r, kbin, o);
  if (SCAN == NLOS_CONFOCAL) {
    if (COS == NLOS_COS_NONE) {
      const float2 d = __fmul2_rn(r2, r2);
      w = __fmul2_rn(q.kq, make_float2(rcp_approx(d.x), rcp_approx(d.y)));
    } else if (COS == NLOS_COS_OBJECT) {
      const float2 d = __fmul2_rn(__fmul2_rn(r2, r2), r2);
      w = __fmul2_rn(__fmul2_rn(cn, cn), make_float2(rcp_approx(d.x), rcp_approx(d.y)));
    } else {
      const float2 d2 = __fmul2_rn(r2, r2);
      const float2 d = __fmul2_rn(d2, d2);
      w = __fmul2_rn(__fmul2_rn(cn, cn), make_float2(rcp_approx(d.x), rcp_approx(d.y)));
    }
  } else {
    if (COS == NLOS_COS_NONE) {
      w = __fmul2_rn(q.kq, make_float2(rcp_approx(r2.x), rcp_approx(r2.y)));
    } else if (COS == NLOS_COS_OBJECT) {
      const float2 d = __fmul2_rn(r2, r);
      w = __fmul2_rn(cn, make_float2(rcp_approx(d.x), rcp_approx(d.y)));
    } else {
      const float2 d = __fmul2_rn(r2, r2);
      w = __fmul2_rn(cn, make_float2(rcp_approx(d.x), rcp_approx(d.y)));
    }
  }
#else
  float2 ri = make_float2(rsqrt_approx(r2.x), rsqrt_approx(r2.y));
  // one Newton step on 1/r (e = 1 - r2 ri^2, ri += ri e / 2): the hardware
  // estimate's few-ulp error would otherwise grow to ~1e-6 in the r^-6 weight
  float2 r = __fmul2_rn(r2, ri);
  const float2 e = __ffma2_rn(make_float2(-r.x, -r.y), ri, make_float2(1.0f, 1.0f));
  ri = __ffma2_rn(__fmul2_rn(ri, make_float2(0.5f, 0.5f)), e, ri);
  r = __fmul2_rn(r2, ri);
  u = __ffma2_rn(r, kbin, o);
  float2 ri2 = __fmul2_rn(ri, ri);
  if (SCAN == NLOS_CONFOCAL) {
    if (COS == NLOS_COS_NONE) {
      w = __fmul2_rn(__fmul2_rn(q.kq, ri2), ri2);
    } else if (COS == NLOS_COS_OBJECT) {
      float2 t = __fmul2_rn(cn, __fmul2_rn(ri2, ri));
      w = __fmul2_rn(t, t);
    } else {
      float2 t = __fmul2_rn(cn, __fmul2_rn(ri2, ri2));
      w = __fmul2_rn(t, t);
    }
  } else {
    if (COS == NLOS_COS_NONE) {
      w = __fmul2_rn(q.kq, ri2);
    } else if (COS == NLOS_COS_OBJECT) {
      w = __fmul2_rn(cn, __fmul2_rn(ri2, ri));
    } else {
      w = __fmul2_rn(cn, __fmul2_rn(ri2, ri2));
    }
  }
#endif
}

template <int SCAN, int COS>
__device__ __forceinline__ void pair_eval2(const PointPair& q, float2 nsx, float2 nsy, float2 off,
                                           float2 kbin, float2& u, float2& w, float2& cn) {
  float2 r2;
  pair_geom2(q, nsx, nsy, r2, cn);
  pair_finish2<SCAN, COS>(q, r2, cn, off, kbin, u, w);
}

// Early-out test on r^2, before any square root: can the point land in
// [-margin, lim + margin) bins of the window for this lane? Conservative
// (margin >= 1 bin against a rounding error of ~1e-3 bin); the exact bin
// test follows for the points that pass.
//   confocal:     r in [r_lo, r_hi) with per-lane bounds (r2lo, r2hi = squares)
//   non-confocal: r_lo/hi = base_lo/hi - uoff / kbin (per point and lane)
template <int SCAN>
__device__ __forceinline__ bool2_t may_bin2(const PointPair& q, float2 r2, float2 r2lo, float2 r2hi,
                                            float2 ikbin_neg) {
  if (SCAN == NLOS_CONFOCAL) {
    return bool2_t{r2.x >= r2lo.x && r2.x < r2hi.x, r2.y >= r2lo.y && r2.y < r2hi.y};
  } else {
    // here r2lo / r2hi hold base_lo / base_hi (in metres, per lane)
    const float2 rlo = __ffma2_rn(q.uoff, ikbin_neg, r2lo);
    const float2 rhi = __ffma2_rn(q.uoff, ikbin_neg, r2hi);
    const float2 lo2 = __fmul2_rn(rlo, rlo);
    const float2 hi2 = __fmul2_rn(rhi, rhi);
    return bool2_t{rhi.x > 0.f && r2.x < hi2.x && (rlo.x <= 0.f || r2.x >= lo2.x),
                   rhi.y > 0.f && r2.y < hi2.y && (rlo.y <= 0.f || r2.y >= lo2.y)};
  }
}

__device__ __forceinline__ void load_pair(const PointPair* p, PointPair& q) {
  const float4* v = reinterpret_cast<const float4*>(p);
  float4 a = v[0], b = v[1], c = v[2], d = v[3];
  q.px = make_float2(a.x, a.y);
  q.py = make_float2(a.z, a.w);
  q.pz2 = make_float2(b.x, b.y);
  q.kq = make_float2(b.z, b.w);
  q.na = make_float2(c.x, c.y);
  q.nb = make_float2(c.z, c.w);
  q.nc = make_float2(d.x, d.y);
  q.uoff = make_float2(d.z, d.w);
}

template <int COS>
__device__ __forceinline__ bool facing(float cn) {
  return COS == NLOS_COS_NONE ? true : (cn > 0.0f);
}

// First bin of window `win`, and its bins: the windows tile [-halo, B + halo).
__device__ __forceinline__ int window_start(const FwdArgs& a, uint32_t win) {
  return (int)(win * a.bw) - a.halo;
}
__device__ __forceinline__ int window_bins(const FwdArgs& a, int w0) {
  return min((int)a.bw, (int)a.B + a.halo - w0);
}

// One point's Gaussian splat into this lane's histogram column (bins of the
// window with |b + 1/2 - u| < 6 sigma), taps by the recurrence
// K_{b+1} = K_b * rho_b, rho_{b+1} = rho_b * exp(-1/sigma^2), restarted from a
// direct evaluation every 8 taps: the recurrence's rounding error grows with
// the square of the number of steps (about 1e-4 after 90 taps in FP32).
__device__ __forceinline__ void splat_one(uint32_t col_addr, float u, float w, int lim,
                                          const FwdArgs& a) {
  float lo_f = floorf(u - 0.5f - a.reach) + 1.0f;
  float hi_f = ceilf(u - 0.5f + a.reach) - 1.0f;
  int lo = max(0, (int)lo_f);
  int hi = min(lim - 1, (int)hi_f);
  if (lo > hi) return;
  const float wn = w * a.norm;
  uint32_t addr = col_addr + (uint32_t)lo * (kTile * 4);
  float K = 0.f, rho = 0.f;
  for (int b = lo; b <= hi; ++b) {
    if (((b - lo) & 7) == 0) {
      const float x = (float)b + 0.5f - u;
      K = wn * expf(-x * x * a.inv2s2);
      rho = expf(-(2.0f * x + 1.0f) * a.inv2s2);
    }
    red_add_shared(addr, K);
    K *= rho;
    rho *= a.qstep;
    addr += kTile * 4;
  }
}

struct FwdSmem {
  float* hist;                 // [bw][32]
  PointPair* stage;            // [stages][ppb]
  uint64_t* bars;              // full[stages] then empty[stages] (initialised by the caller)
  unsigned long long* units;   // [stages]: the (tile, window) of each slot's pairs
  uint32_t* rows = nullptr;    // [kRowWords] or null: row tracking (see fwd_run_ws)
  uint32_t* fill = nullptr;    // [stages]: the pairs staged in each slot
  uint32_t* occ = nullptr;     // [stages][kOccGroups]: occluders of each group (MODE_NEAREST_OCC)
  unsigned long long* lane_units = nullptr;  // [32]: the producer lanes' units | groups << 32 (list)
};
// rows: 32 words for the producer's lanes, then one per slot (up to 8 stages)
constexpr int kMaxRangedStages = 8;
constexpr int kRowWords = 32 + kMaxRangedStages;

constexpr uint32_t kOccGroups = NLOS_FWD_PPB / kGroupPairs;  // groups of a slot

constexpr unsigned long long kNoUnit = ~0ull;  // end of a run (in FwdSmem::units)

// Scan-point state of the (tile, window) a CTA is working on; lane l of every
// warp holds scan point l of the tile.
struct TileState {
  long long tw = -1;
  int w0 = 0;   // first bin of the current window
  int lim = 0;  // its bins
  float2 sx2, sy2, nsx2, nsy2;
  float2 off2;          // bin offset of the scan point, relative to bin 0
  float2 nw02;          // -(first bin of the window)
  uint32_t binbase = kMagicBits;  // bit pattern of kMagic + first bin of the window
  float2 r2lo2, r2hi2;  // early-out bounds (see may_bin2)
};

// Bins beyond the window edges that still matter: 1 for the histogram modes
// (edge pairs of the boundary count) and the moment form (whose windows hold
// the halo themselves), the splat reach + 1 for its taps.
template <int MODE>
__device__ __forceinline__ float window_margin(const FwdArgs& a) {
  return MODE == MODE_SPLAT ? a.reach + 1.0f : 1.0f;
}

__device__ __forceinline__ void load_tile(const FwdArgs& a, long long tw, int lane,
                                          TileState& ts, bool confocal, float margin) {
  const uint32_t tile = (uint32_t)(tw / a.n_win);
  ts.tw = tw;
  ts.w0 = window_start(a, (uint32_t)(tw % a.n_win));
  ts.lim = window_bins(a, ts.w0);
  const uint32_t s = tile * kTile + lane;
  if (s < a.S) {
    const ScanPoint sp = a.scan[s];
    ts.sx2 = make_float2(sp.sx, sp.sx);
    ts.sy2 = make_float2(sp.sy, sp.sy);
    ts.nsx2 = make_float2(-sp.sx, -sp.sx);
    ts.nsy2 = make_float2(-sp.sy, -sp.sy);
    ts.off2 = make_float2(sp.off, sp.off);
    ts.nw02 = make_float2(-(float)ts.w0, -(float)ts.w0);
    ts.binbase = (uint32_t)(kMagicBits + ts.w0);
    const float o = sp.off - (float)ts.w0;
    // r range of u in [-margin, lim + margin): r = (u - o) / kbin
    const float ik = 1.0f / a.kbin;
    const float rlo = (-margin - o) * ik, rhi = ((float)ts.lim + margin - o) * ik;
    float lo, hi;
    if (confocal) {
      lo = rlo > 0.f ? rlo * rlo : 0.f;
      hi = rhi > 0.f ? rhi * rhi : -1.f;
    } else {
      lo = rlo;  // the point's uoff / kbin is subtracted in may_bin2
      hi = rhi;
    }
    ts.r2lo2 = make_float2(lo, lo);
    ts.r2hi2 = make_float2(hi, hi);
  } else {
    ts.sx2 = ts.sy2 = ts.nsx2 = ts.nsy2 = make_float2(0.f, 0.f);
    ts.off2 = make_float2(-1e30f, -1e30f);  // u -> -inf: never binned
    ts.nw02 = make_float2(0.f, 0.f);
    ts.binbase = (uint32_t)(kMagicBits + ts.w0);
    ts.r2lo2 = make_float2(1.f, 1.f);      // empty r ranges
    ts.r2hi2 = make_float2(-1.f, -1.f);
  }
}

// Four output bins o0..o0+3 of one column: each histogram row read once
// (4 + 2R loads into registers), the taps unrolled at compile time.
template <int R>
__device__ __forceinline__ void conv_quad(const FwdArgs& a, const float* hist, int r0, int bw, int c,
                                          float v[4]) {
  float h[4 + 2 * R];
#pragma unroll
  for (int k = 0; k < 4 + 2 * R; ++k) {
    const int b = r0 - R + k;
    h[k] = (b >= 0 && b < bw) ? hist[b * kTile + c] : 0.f;
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    float acc = 0.f;
#pragma unroll
    for (int j = -R; j <= R; ++j) acc = fmaf(a.taps[j + R], h[e - j + R], acc);
    v[e] = acc;
  }
}

// Any radius (taps loop at run time).
__device__ __forceinline__ void conv_quad_any(const FwdArgs& a, const float* hist, int r0, int bw,
                                              int c, int R, float v[4]) {
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int bc = r0 + e;  // histogram row of the centre tap
    float acc = 0.f;
    for (int j = -R; j <= R; ++j) {
      const int b = bc - j;
      if (b >= 0 && b < bw) acc = fmaf(a.taps[j + R], hist[b * kTile + c], acc);
    }
    v[e] = acc;
  }
}

template <int R>
__device__ __forceinline__ void flush_quads(const FwdArgs& a, const float* hist, int lo, int nq,
                                            int w0, int R_rt, uint32_t s, int c, int warp_rel,
                                            int n_warps) {
  for (int qi = warp_rel; qi < nq; qi += n_warps) {
    const int o0 = lo + 4 * qi;
    float v[4];
    if (R >= 0) conv_quad<(R >= 0 ? R : 0)>(a, hist, o0 - w0, (int)a.bw, c, v);
    else conv_quad_any(a, hist, o0 - w0, (int)a.bw, c, R_rt, v);
    if (a.replicate) {
      // the taps beyond the first / last bin read that bin (linear, so each
      // partial histogram adds its own share); only the windows holding it
      const int last = (int)a.B - 1;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int o = o0 + e;
        if (w0 == 0 && o < R_rt) v[e] = fmaf(a.tail[o], hist[c], v[e]);
        if (last - w0 < (int)a.bw && last - o >= 0 && last - o < R_rt)
          v[e] = fmaf(a.tail[last - o], hist[(last - w0) * kTile + c], v[e]);
      }
    }
    if (s < a.S && (v[0] != 0.f || v[1] != 0.f || v[2] != 0.f || v[3] != 0.f)) {
      float* dst = a.tau + (size_t)s * a.B + o0;
      if ((a.B & 3u) == 0u) {
        red_add_global_v4(dst, make_float4(v[0], v[1], v[2], v[3]));
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (o0 + e < (int)a.B && o0 + e >= 0) red_add_global(dst + e, v[e]);
      }
    }
  }
}

// Flush the partial histogram of (tile, window) tw into tau (jittered for
// NEAREST): out[o] = sum_j taps[j + R] * hist[o - w0 - j], zero outside the
// window; four consecutive bins per thread, one vector reduction each. Runs
// on the warps [w_first, w_first + n_warps) of the CTA. Radii up to 16 use
// a compile-time unrolled convolution.
// Only histogram rows [rlo, rhi) may be nonzero, so only the output bins
// they reach are written.
template <int MODE>
__device__ __forceinline__ void flush_tile(const FwdArgs& a, long long tw, const float* hist,
                                           int warp_rel, int n_warps, int rlo, int rhi) {
  const uint32_t tile = (uint32_t)(tw / a.n_win);
  const int w0 = window_start(a, (uint32_t)(tw % a.n_win));
  const int R = (MODE == MODE_SPLAT) ? 0 : a.R;
  if (rhi <= rlo) return;
  const int lo = max(0, w0 + rlo - R) & ~3;
  const int hi = min((int)a.B, w0 + rhi + R);
  if (hi <= lo) return;
  const int nq = (hi - lo + 3) >> 2;  // quads of output bins
  const int c = threadIdx.x & 31;
  // the transient (output row) of the lane's scan point; none for the padding
  // lanes of a ragged last tile
  const uint32_t si = tile * kTile + c;
  const uint32_t s = si < a.S ? a.scan[si].row : 0xFFFFFFFFu;
#define NLOS_FLUSH_R(RR) \
  case RR:               \
    flush_quads<RR>(a, hist, lo, nq, w0, R, s, c, warp_rel, n_warps); \
    break;
  switch (R) {
    NLOS_FLUSH_R(0) NLOS_FLUSH_R(1) NLOS_FLUSH_R(2) NLOS_FLUSH_R(3) NLOS_FLUSH_R(4)
    NLOS_FLUSH_R(5) NLOS_FLUSH_R(6) NLOS_FLUSH_R(7) NLOS_FLUSH_R(8) NLOS_FLUSH_R(9)
    NLOS_FLUSH_R(10) NLOS_FLUSH_R(11) NLOS_FLUSH_R(12) NLOS_FLUSH_R(13) NLOS_FLUSH_R(14)
    NLOS_FLUSH_R(15) NLOS_FLUSH_R(16)
    default:
      flush_quads<-1>(a, hist, lo, nq, w0, R, s, c, warp_rel, n_warps);
  }
#undef NLOS_FLUSH_R
}

// red.shared.add.f32 [addr + k * kMomStride] of w c^k for the moments k <
// kMoments of one point, predicated on row < rows and a facing cosine.
template <int K>
__device__ __forceinline__ void red_moment(uint32_t addr, float wk, uint32_t ok) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n @p red.shared.add.f32 [%0+%3], %1;\n}\n" ::"r"(addr),
      "f"(wk), "r"(ok), "n"(K * kMomStride)
      : "memory");
}

template <int COS>
__device__ __forceinline__ void red_moments(uint32_t addr, float w, float c, uint32_t row,
                                            uint32_t rows, float cn) {
  static_assert(kMoments == 6, "red_moments is written out for six moments");
  const uint32_t ok = (row < rows && (COS == NLOS_COS_NONE || cn > 0.0f)) ? 1u : 0u;
  float wk = w;
  red_moment<0>(addr, wk, ok);
  wk *= c;
  red_moment<1>(addr, wk, ok);
  wk *= c;
  red_moment<2>(addr, wk, ok);
  wk *= c;
  red_moment<3>(addr, wk, ok);
  wk *= c;
  red_moment<4>(addr, wk, ok);
  wk *= c;
  red_moment<5>(addr, wk, ok);
}

// Visibility of the point S + d from the spot S = (sx, sy, 0) (the detector
// leg of a pair; A = |d|^2 > 0, d.z > 0): false when the segment runs
// strictly inside an occluder for more than o.eta of its length. Spheres: the
// chord in units of A (no division), from |S + t d - c|^2 < r^2; boxes: the
// slab intervals of t, with reciprocal estimates. The threshold is far above
// the FP32 rounding of the chord except for near-tangent segments, which the
// parity tests treat like pairs near a bin edge. Only the occluders of `mask`
// (those the segments to the point's group can meet, occ_bounds_mask) are tested.
__device__ __forceinline__ bool occ_seen(const OccSet& o, uint32_t mask, float sx, float sy,
                                         float dx, float dy, float dz, float A) {
  for (; mask; mask &= mask - 1) {
    const int k = __ffs(mask) - 1;
    const float4 p = o.occ[2 * k], q = o.occ[2 * k + 1];
    if (p.w == 0.f) {
      const float fx = sx - p.x, fy = sy - p.y;
      const float B = fmaf(fx, dx, fmaf(fy, dy, -p.z * dz));
      const float C = fmaf(fx, fx, fmaf(fy, fy, fmaf(p.z, p.z, -q.x * q.x)));
      const float disc = fmaf(B, B, -A * C);
      if (disc > 0.f) {
        const float sq = sqrt_approx(disc);
        const float t0 = fmaxf(-B - sq, 0.f), t1 = fminf(-B + sq, A);
        if (t1 - t0 > o.eta * A) return false;
      }
    } else {
      float t0 = 0.f, t1 = 1.f;
      bool miss = false;
      if (dx != 0.f) {
        const float r = rcp_approx(dx);
        const float ta = (p.x - sx) * r, tb = (q.x - sx) * r;
        t0 = fmaxf(t0, fminf(ta, tb));
        t1 = fminf(t1, fmaxf(ta, tb));
      } else {
        miss = !(p.x < sx && sx < q.x);
      }
      if (dy != 0.f) {
        const float r = rcp_approx(dy);
        const float ta = (p.y - sy) * r, tb = (q.y - sy) * r;
        t0 = fmaxf(t0, fminf(ta, tb));
        t1 = fminf(t1, fmaxf(ta, tb));
      } else {
        miss = miss || !(p.y < sy && sy < q.y);
      }
      const float rz = rcp_approx(dz);  // the spot is at z = 0, dz > 0
      t0 = fmaxf(t0, p.z * rz);
      t1 = fminf(t1, q.z * rz);
      if (!miss && t1 - t0 > o.eta) return false;
    }
  }
  return true;
}

// This warp's share of the n pairs of a slot: evaluate both points of a pair for
// the lane's scan point and add their weights to the lane's histogram column
// (or splat them).
template <int SCAN, int COS, int MODE, int UNROLL>
__device__ __forceinline__ void compute_block(const FwdArgs& a, const PointPair* blkp, uint32_t n,
                                              int warp_rel, int n_warps, const TileState& ts,
                                              uint32_t col_addr, FwdCount& cnt,
                                              int mom_q = 1, const OccSet* occ = nullptr,
                                              const uint32_t* occ_groups = nullptr,
                                              uint32_t rot = 0) {
  const float2 kbin2 = make_float2(a.kbin, a.kbin);
  const float2 magic2 = make_float2(kMagic, kMagic);
  const float2 ikbin_neg = make_float2(-1.0f / a.kbin, -1.0f / a.kbin);
  // a contiguous run of pairs per warp: neighbouring points, so the warps'
  // shared reductions meet different histogram rows at any one time; the
  // short last run rotates over the warps from block to block (rot)
  const uint32_t per = (n + (uint32_t)n_warps - 1u) / (uint32_t)n_warps;
  const uint32_t run = ((uint32_t)warp_rel + rot) % (uint32_t)n_warps;
  const uint32_t i_begin = min(n, run * per), i_end = min(n, i_begin + per);
  // iterations of this warp (counted once per block, not per iteration)
  const uint32_t n_it = i_end - i_begin;
  cnt.tested += n_it;
#if !NLOS_FWD_EARLY
  cnt.full += n_it;
#endif
#pragma unroll UNROLL
  for (uint32_t i = i_begin; i < i_end; ++i) {
    PointPair q;
    load_pair(blkp + i, q);
    float2 r2, cn;
    pair_geom2(q, ts.nsx2, ts.nsy2, r2, cn);
#if NLOS_FWD_EARLY
    // warp-uniform early out: for most (tile, point) combinations of a
    // scene no lane can bin either point (outside the window or facing away).
    // Not in the boundary-count mode, which counts every pair near a bin
    // edge of the whole transient (facing or not) in the first window's pass.
    if (MODE != MODE_NEAREST_COUNT) {
      const bool2_t m = may_bin2<SCAN>(q, r2, ts.r2lo2, ts.r2hi2, ikbin_neg);
      if (!__any_sync(0xffffffffu, (m.x && facing<COS>(cn.x)) || (m.y && facing<COS>(cn.y))))
        continue;
    }
    ++cnt.full;
#endif
    float2 u, w;
    pair_finish2<SCAN, COS>(q, r2, cn, ts.off2, kbin2, u, w);
    if (MODE == MODE_SPLAT) {
      // window-relative u (exact: w0 is an integer < 2^24)
      u = __fadd2_rn(u, ts.nw02);
      if (facing<COS>(cn.x)) splat_one(col_addr, u.x, w.x, ts.lim, a);
      if (facing<COS>(cn.y)) splat_one(col_addr, u.y, w.y, ts.lim, a);
    } else if (MODE == MODE_SPLAT_MOM) {
      const float2 v = __fmul2_rn(u, make_float2((float)mom_q, (float)mom_q));  // exact
      const float2 t = __fadd2_rd(v, magic2);                          // kMagic + floor(v)
      const float2 fl = __fadd2_rn(t, make_float2(-kMagic, -kMagic));  // floor(v), exact
      const float2 fr = __fadd2_rn(v, make_float2(-fl.x, -fl.y));      // v - floor(v), exact
      const float2 c = __fadd2_rn(make_float2(0.5f, 0.5f), make_float2(-fr.x, -fr.y));
      const uint32_t ra = (uint32_t)(__float_as_int(t.x) - kMagicBits - ts.w0 * mom_q);
      const uint32_t rb = (uint32_t)(__float_as_int(t.y) - kMagicBits - ts.w0 * mom_q);
      const uint32_t rows = (uint32_t)(ts.lim * mom_q);
      red_moments<COS>(col_addr + ra * (kTile * 4), w.x, c.x, ra, rows, cn.x);
      red_moments<COS>(col_addr + rb * (kTile * 4), w.y, c.y, rb, rows, cn.y);
    } else {
      // kMagic + floor(u), exactly; the window's first bin comes off the
      // integer (floor(u) - w0 = floor(u - w0) for an integer w0)
      const float2 t = __fadd2_rd(u, magic2);
      uint32_t ba = (uint32_t)__float_as_int(t.x) - ts.binbase;
      uint32_t bb = (uint32_t)__float_as_int(t.y) - ts.binbase;
      if (MODE == MODE_NEAREST_OCC) {
        // visibility only for pairs that would be binned; a hidden pair's bin
        // is moved out of range, so its reduction is predicated off
        const float sx = ts.sx2.x, sy = ts.sy2.x;
        const uint32_t occ_mask = occ_groups[i / kGroupPairs];
        if (ba < (uint32_t)ts.lim && facing<COS>(cn.x) &&
            !occ_seen(*occ, occ_mask, sx, sy, q.px.x - sx, q.py.x - sy, sqrt_approx(q.pz2.x),
                      r2.x))
          ba = 0xFFFFFFFFu;
        if (bb < (uint32_t)ts.lim && facing<COS>(cn.y) &&
            !occ_seen(*occ, occ_mask, sx, sy, q.px.y - sx, q.py.y - sy, sqrt_approx(q.pz2.y),
                      r2.y))
          bb = 0xFFFFFFFFu;
      }
      const uint32_t aa = col_addr + ba * (kTile * 4);
      const uint32_t ab = col_addr + bb * (kTile * 4);
      // the in-window and facing test and the reduction in one predicated
      // block (shared f32 reductions are a compare-and-swap loop here)
#if NLOS_FWD_VOTE == 2
      // preceded by one warp-uniform test: most pairs of a tile fall outside
      // the window or face away together
      const bool oka = ba < (uint32_t)ts.lim && facing<COS>(cn.x);
      const bool okb = bb < (uint32_t)ts.lim && facing<COS>(cn.y);
#endif
#if NLOS_FWD_VOTE == 2
      if (__any_sync(0xffffffffu, oka || okb)) {
        if (COS == NLOS_COS_NONE) {
          red_add_shared_if_bin(aa, w.x, ba, (uint32_t)ts.lim);
          red_add_shared_if_bin(ab, w.y, bb, (uint32_t)ts.lim);
        } else {
          red_add_shared_if_bin_cos(aa, w.x, ba, (uint32_t)ts.lim, cn.x);
          red_add_shared_if_bin_cos(ab, w.y, bb, (uint32_t)ts.lim, cn.y);
        }
      }
#else
      if (COS == NLOS_COS_NONE) {
        red_add_shared_if_bin(aa, w.x, ba, (uint32_t)ts.lim);
        red_add_shared_if_bin(ab, w.y, bb, (uint32_t)ts.lim);
      } else {
        red_add_shared_if_bin_cos(aa, w.x, ba, (uint32_t)ts.lim, cn.x);
        red_add_shared_if_bin_cos(ab, w.y, bb, (uint32_t)ts.lim, cn.y);
      }
#endif
      if (MODE == MODE_NEAREST_COUNT && ts.w0 == 0) {
        // pairs with u within eps of a bin edge m in [0, B] (u is global here)
        const float2 fl = __fadd2_rn(t, make_float2(-kMagic, -kMagic));
        const float fa = u.x - fl.x, fb = u.y - fl.y;
        const bool na = (fa < a.eps && fl.x >= 0.f && fl.x <= (float)a.B) ||
                        (1.0f - fa < a.eps && fl.x + 1.0f >= 0.f && fl.x + 1.0f <= (float)a.B);
        const bool nb = (fb < a.eps && fl.y >= 0.f && fl.y <= (float)a.B) ||
                        (1.0f - fb < a.eps && fl.y + 1.0f >= 0.f && fl.y + 1.0f <= (float)a.B);
        // the odd slot of the last pair may be padding (pz2 huge): its u is
        // never near a valid edge
        cnt.boundary += (unsigned)na + (unsigned)nb;
      }
    }
  }
}

// Moment flush: the bins o within J of the window's bins [blo, bhi) that may
// hold anything, tau[o] += sum_n sum_r D_n[r - q (o - w0) + q J] M_n[r]. A warp
// takes four consecutive bins at a time (lane = scan point) and, for each row
// phase, walks the rows k of that phase with the taps of the four bins in
// registers: bin e meets row k with tap m - e, m = k - o' + J, so each step
// loads one row and one new tap of each moment for 24 FMAs. (With each bin
// loading its own rows, four shared loads for the same 24 FMAs, the flushes
// were the larger part of a splat forward.)
__device__ __forceinline__ void flush_tile_mom(const FwdArgs& a, const MomTab& mt, long long tw,
                                               const float* hist, int warp_rel, int n_warps,
                                               int blo, int bhi) {
  const uint32_t tile = (uint32_t)(tw / a.n_win);
  const int w0 = window_start(a, (uint32_t)(tw % a.n_win));
  const int J = mt.J, q = mt.q;
  const int lo = max(0, w0 + blo - J) & ~3;
  const int hi = bhi > blo ? min((int)a.B, w0 + bhi + J) : lo;
  const int c = threadIdx.x & 31;
  // the transient (output row) of the lane's scan point; none for the padding
  // lanes of a ragged last tile
  const uint32_t si = tile * kTile + c;
  const uint32_t s = si < a.S ? a.scan[si].row : 0xFFFFFFFFu;
  for (int o0 = lo + 4 * warp_rel; o0 < hi; o0 += 4 * n_warps) {
    const int rel = o0 - w0;  // window-relative first bin
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    const int k0 = max(blo, rel - J), k1 = min(bhi, rel + 3 + J + 1);
    for (int ph = 0; ph < q; ++ph) {
      float tap[4][kMoments];
      // taps of bins 1..3 before the first row
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int m = k0 - 1 - rel + J - e;  // becomes bin e + 1's tap at row k0
#pragma unroll
        for (int n = 0; n < kMoments; ++n)
          tap[e][n] = (e < 3 && m >= 0 && m <= 2 * J) ? mt.d[ph + q * m][n] : 0.f;
      }
#pragma unroll 4
      for (int k = k0; k < k1; ++k) {
        const int m = k - rel + J;
        const float* h = hist + (size_t)(k * q + ph) * kTile + c;
#pragma unroll
        for (int n = 0; n < kMoments; ++n) {
#pragma unroll
          for (int e = 3; e > 0; --e) tap[e][n] = tap[e - 1][n];
          tap[0][n] = m <= 2 * J ? mt.d[ph + q * m][n] : 0.f;
          const float hn = h[n * kMomRows * kTile];
#pragma unroll
          for (int e = 0; e < 4; ++e) v[e] = fmaf(tap[e][n], hn, v[e]);
        }
      }
    }
    if (s < a.S && (v[0] != 0.f || v[1] != 0.f || v[2] != 0.f || v[3] != 0.f)) {
      float* dst = a.tau + (size_t)s * a.B + o0;
      if ((a.B & 3u) == 0u) {
        red_add_global_v4(dst, make_float4(v[0], v[1], v[2], v[3]));
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (o0 + e < (int)a.B) red_add_global(dst + e, v[e]);
      }
    }
  }
  // the weight of the pairs beyond either end of [0, B) (splat_tail_kernel)
  float far = 0.f;
  for (int bin = blo + warp_rel; bin < bhi; bin += n_warps)
    if (w0 + bin < 0 || w0 + bin >= (int)a.B)
      for (int ph = 0; ph < q; ++ph) far += hist[(bin * q + ph) * kTile + c];
  if (s < a.S && far != 0.f) red_add_global(a.far_mass + s, far);
}

// For three weights x at a time, the first of n list entries with at least x
// before it (n if none), by a whole warp: 32 probes a round.
__device__ __forceinline__ void list_lower_bounds(const ListEntry* list, uint32_t n,
                                                  const uint32_t x[3], uint32_t at[3]) {
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t lo[3] = {0u, 0u, 0u}, len[3] = {n, n, n};
  while (len[0] | len[1] | len[2]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const uint32_t step = (len[i] + 31u) / 32u, p = lane * step;
      const bool below = p < len[i] && list[lo[i] + p].before < x[i];
      const uint32_t m = __ballot_sync(0xffffffffu, below);
      // probes ascend: the answer lies in (last below, next probe]
      if (m == 0u) {
        len[i] = 0u;
      } else {
        const uint32_t last = (31u - (uint32_t)__clz((int)m)) * step;
        lo[i] += last + 1u;
        len[i] = min(step - 1u, len[i] - last - 1u);
      }
    }
  }
  for (int i = 0; i < 3; ++i) at[i] = lo[i];
}

// max of a * b over a in [a0, a1], b in [b0, b1]
__device__ __forceinline__ float imax(float a0, float a1, float b0, float b1) {
  return fmaxf(fmaxf(a0 * b0, a0 * b1), fmaxf(a1 * b0, a1 * b1));
}

// Can unit (tile, window, point block) bin anything? From the block's
// bounds and the tile's: the range of u over every (spot, point) of the
// unit (distance bounds between the spot box at z = 0 and the point box)
// against the window with `margin` bins on each side, the object cosine
// (upper bound of n.(spot - x) over the boxes) and whether any point carries
// weight. Conservative: a unit it keeps may still bin nothing.
// Bounds of point block blk: the union of its sub-blocks' bounds.
__device__ __forceinline__ BlockBound block_bound(const FwdArgs& a, uint32_t blk) {
  const uint32_t sub_per = max(1u, a.ppb / kSubPairs);
  const uint32_t sb0 = blk * a.ppb / kSubPairs;  // (a block smaller than a sub-block lies in one)
  const uint32_t n_sub = (a.n_pairs + kSubPairs - 1) / kSubPairs;
  BlockBound b = a.bounds[sb0];
  for (uint32_t j = 1; j < sub_per && sb0 + j < n_sub; ++j) {
    const BlockBound c = a.bounds[sb0 + j];
    b.x0 = fminf(b.x0, c.x0); b.x1 = fmaxf(b.x1, c.x1);
    b.y0 = fminf(b.y0, c.y0); b.y1 = fmaxf(b.y1, c.y1);
    b.z0 = fminf(b.z0, c.z0); b.z1 = fmaxf(b.z1, c.z1);
    b.nx0 = fminf(b.nx0, c.nx0); b.nx1 = fmaxf(b.nx1, c.nx1);
    b.ny0 = fminf(b.ny0, c.ny0); b.ny1 = fmaxf(b.ny1, c.ny1);
    b.nz0 = fminf(b.nz0, c.nz0); b.nz1 = fmaxf(b.nz1, c.nz1);
    b.uo0 = fminf(b.uo0, c.uo0); b.uo1 = fmaxf(b.uo1, c.uo1);
    b.live = fmaxf(b.live, c.live);
  }
  return b;
}

// Can a point inside the bounds b reach the window starting at bin w0 (lim
// bins) of a tile with spot bounds t (and face one of its spots)? ulo, uhi:
// the range of u over the two boxes, window-relative.
template <int SCAN, int COS>
__device__ __forceinline__ bool bounds_live(const FwdArgs& a, const TileBound& t,
                                            const BlockBound& b, int w0, float lim,
                                            float margin, float& ulo_out, float& uhi_out) {
  if (b.live == 0.f) return false;
  const float dx = fmaxf(0.f, fmaxf(b.x0 - t.sx1, t.sx0 - b.x1));
  const float dy = fmaxf(0.f, fmaxf(b.y0 - t.sy1, t.sy0 - b.y1));
  const float rmin = sqrtf(dx * dx + dy * dy + b.z0 * b.z0);
  const float fx = fmaxf(fabsf(b.x1 - t.sx0), fabsf(t.sx1 - b.x0));
  const float fy = fmaxf(fabsf(b.y1 - t.sy0), fabsf(t.sy1 - b.y0));
  const float rmax = sqrtf(fx * fx + fy * fy + b.z1 * b.z1);
  float ulo = fmaf(rmin, a.kbin, t.off0) - (float)w0;
  float uhi = fmaf(rmax, a.kbin, t.off1) - (float)w0;
  if (SCAN != NLOS_CONFOCAL) {
    ulo += b.uo0;
    uhi += b.uo1;
  }
  ulo_out = ulo;
  uhi_out = uhi;
  if (uhi < -margin || ulo >= lim + margin) return false;
  if (COS != NLOS_COS_NONE) {
    const float f = imax(b.nx0, b.nx1, t.sx0 - b.x1, t.sx1 - b.x0) +
                    imax(b.ny0, b.ny1, t.sy0 - b.y1, t.sy1 - b.y0) +
                    imax(b.nz0, b.nz1, -b.z1, -b.z0);
    if (f <= 0.f) return false;
  }
  return true;
}

template <int SCAN, int COS>
__device__ __forceinline__ bool unit_live(const FwdArgs& a, unsigned long long unit, float margin,
                                          float& ulo_out, float& uhi_out) {
  const unsigned long long tw = unit / a.n_blk;
  const uint32_t blk = (uint32_t)(unit - tw * a.n_blk);
  const uint32_t tile = (uint32_t)(tw / a.n_win);
  const int w0 = window_start(a, (uint32_t)(tw % a.n_win));
  const float lim = (float)window_bins(a, w0);
  const TileBound t = a.tiles[tile];
  const BlockBound b = block_bound(a, blk);
  return bounds_live<SCAN, COS>(a, t, b, w0, lim, margin, ulo_out, uhi_out);
}

// The same test on each sub-block of a unit of two: whether one is live, and
// the u range over the live ones.
template <int SCAN, int COS>
__device__ __forceinline__ bool unit_live_halves(const FwdArgs& a, unsigned long long unit,
                                                 float margin, float& ulo_out, float& uhi_out) {
  const unsigned long long tw = unit / a.n_blk;
  const uint32_t blk = (uint32_t)(unit - tw * a.n_blk);
  const uint32_t tile = (uint32_t)(tw / a.n_win);
  const int w0 = window_start(a, (uint32_t)(tw % a.n_win));
  const float lim = (float)window_bins(a, w0);
  const TileBound t = a.tiles[tile];
  const uint32_t sb0 = blk * 2u;
  const uint32_t n_sub = (a.n_pairs + kSubPairs - 1) / kSubPairs;
  float l0 = 0.f, h0 = 0.f, l1 = 0.f, h1 = 0.f;
  const bool live0 = bounds_live<SCAN, COS>(a, t, a.bounds[sb0], w0, lim, margin, l0, h0);
  const bool live1 = sb0 + 1 < n_sub &&
                     bounds_live<SCAN, COS>(a, t, a.bounds[sb0 + 1], w0, lim, margin, l1, h1);
  ulo_out = live0 ? (live1 ? fminf(l0, l1) : l0) : l1;
  uhi_out = live0 ? (live1 ? fmaxf(h0, h1) : h0) : h1;
  return live0 || live1;
}

// The groups of kGroupPairs pairs of a block that a tile may bin (bit g: pairs
// [16 g, 16 g + 16) of the block), one group a lane; the whole warp calls it.
template <int SCAN, int COS>
__device__ __forceinline__ uint32_t block_groups(const FwdArgs& a, const TileBound& t, uint32_t blk,
                                                 int w0, float lim, float margin) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t first = blk * a.ppb + lane * kGroupPairs;
  bool live = lane * kGroupPairs < a.ppb && first < a.n_pairs;
  if (live) {
    float ulo, uhi;
    live = bounds_live<SCAN, COS>(a, t, a.groups[first / kGroupPairs], w0, lim, margin, ulo, uhi);
  }
  return __ballot_sync(0xffffffffu, live);
}

// The same for a unit; cull: whether to test the bounds (else every group).
template <int SCAN, int COS>
__device__ __forceinline__ uint32_t unit_groups(const FwdArgs& a, unsigned long long unit,
                                                float margin, bool cull) {
  const unsigned long long tw = unit / a.n_blk;
  const uint32_t blk = (uint32_t)(unit - tw * a.n_blk);
  if (!cull) {
    const uint32_t at = (threadIdx.x & 31u) * kGroupPairs;
    return __ballot_sync(0xffffffffu, at < a.ppb && blk * a.ppb + at < a.n_pairs);
  }
  const int w0 = window_start(a, (uint32_t)(tw % a.n_win));
  return block_groups<SCAN, COS>(a, a.tiles[(uint32_t)(tw / a.n_win)], blk, w0,
                                 (float)window_bins(a, w0), margin);
}

// Occluders that can meet a segment from a spot of the tile t (z = 0) to a
// point inside the bounds b, as bits (conservative). A segment ending at depth
// z_p in [z0, z1] is at depth zeta at t = zeta / z_p, over the lateral box
// interpolated at t between the tile's spot box and the block's box; over
// the depths an occluder spans, t stays in [zeta_lo / z1, min(1, zeta_hi /
// z0)], and the box is linear in t, so its extremes sit at those two ends.
__device__ __forceinline__ uint32_t occ_bounds_mask(const TileBound& t, const BlockBound& b,
                                                    const OccSet& o) {
  const uint32_t all = o.n >= 32 ? 0xFFFFFFFFu : (1u << o.n) - 1u;
  if (!(b.z0 > 0.f)) return all;
  constexpr float pad = 1e-4f;  // metres, against rounding of the boxes
  uint32_t m = 0;
  for (int k = 0; k < o.n; ++k) {
    const float4 p = o.occ[2 * k], q = o.occ[2 * k + 1];
    const bool sph = p.w == 0.f;
    const float ox0 = (sph ? p.x - q.x : p.x) - pad, ox1 = (sph ? p.x + q.x : q.x) + pad;
    const float oy0 = (sph ? p.y - q.x : p.y) - pad, oy1 = (sph ? p.y + q.x : q.y) + pad;
    const float oz0 = (sph ? p.z - q.x : p.z) - pad, oz1 = (sph ? p.z + q.x : q.z) + pad;
    const float zlo = fmaxf(oz0, 0.f), zhi = fminf(oz1, b.z1);
    if (zlo > zhi) continue;
    const float tlo = zlo / b.z1, thi = fminf(1.f, zhi / b.z0);
    const float xmin = fminf(fmaf(tlo, b.x0 - t.sx0, t.sx0), fmaf(thi, b.x0 - t.sx0, t.sx0));
    const float xmax = fmaxf(fmaf(tlo, b.x1 - t.sx1, t.sx1), fmaf(thi, b.x1 - t.sx1, t.sx1));
    const float ymin = fminf(fmaf(tlo, b.y0 - t.sy0, t.sy0), fmaf(thi, b.y0 - t.sy0, t.sy0));
    const float ymax = fmaxf(fmaf(tlo, b.y1 - t.sy1, t.sy1), fmaf(thi, b.y1 - t.sy1, t.sy1));
    if (xmax < ox0 || xmin > ox1 || ymax < oy0 || ymin > oy1) continue;
    m |= 1u << k;
  }
  return m;
}

// Histogram rows a unit can touch, packed lo | hi << 16, from its u range
// (window-relative) widened by the mode's margin and two bins against
// rounding, clipped to [0, bw).
__device__ __forceinline__ uint32_t unit_rows(float ulo, float uhi, float margin, uint32_t bw) {
  const float m = ceilf(margin) + 2.f;
  const float lo = fmaxf(floorf(fmaxf(ulo, -1e6f)) - m, 0.f);
  const float hi = fminf(ceilf(fminf(uhi, 1e6f)) + m + 1.f, (float)bw);
  return lo < hi ? (uint32_t)lo | ((uint32_t)hi << 16) : 0u;
}

__device__ __forceinline__ void named_barrier(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Warp-specialised run of work units (tile, window, point block) of one job:
// warp 0 stages points with TMA bulk copies into `stages` slots, the other warps
// evaluate them. The bounds of each group of 16 pairs of a unit are tested, one
// group a lane (by the list's kernel, or here without a list), and the producer
// copies the groups that the tile may bin side by side, so a slot holds up to ppb pairs of one (tile, window), of as many units
// as it takes, and the consumers split them evenly. (Evaluating whole blocks,
// or halves of them, took 24% more pairs on the 64 x 64 union scene and 35%
// more on a ragged heightfield; skipping dead groups on the consumers' side
// left warps waiting for the few that had live ones.) The producer writes each
// slot's (tile, window) and pair count beside it (kNoUnit ends the run); the
// full barrier orders them before the consumers read them. Units come either from the range [u0, u1)
// (chunk_counter == nullptr) or in chunks of `chunk` units claimed from
// *chunk_counter until units_total is reached (or, with max_claims > 0, after
// that many claims), so that CTAs that meet cheap units (culled, or most
// pairs stopped by the early out) take more of them. Consumers
// flush their (tile, window) histogram whenever the tile changes and at the
// end. `it` carries the barrier phases across calls (the serving kernel runs
// one call per work item). UNROLL: unroll of the consumers' pair loop;
// RANGED: track the histogram rows each tile can touch (from the unit
// bounds) and flush and zero only those (both cost registers). Every wait is
// bounded; returns false if one gave up (the error is in *a.err).
template <int SCAN, int COS, int MODE, int UNROLL, bool RANGED>
__device__ bool fwd_run_ws(const FwdArgs& a, unsigned long long u0, unsigned long long u1,
                           const FwdSmem& sm, int stages, FwdCount& cnt, const MomTab* mt,
                           uint32_t& it, unsigned long long* chunk_counter = nullptr,
                           unsigned long long chunk = 0, unsigned long long units_total = 0,
                           uint32_t max_claims = 0, const OccSet* occ = nullptr) {
  const int mom_q = (MODE == MODE_SPLAT_MOM) ? mt->q : 1;
  __shared__ int s_abort;
  __shared__ uint32_t s_used;  // slots this call used (units + the end mark)
  __shared__ unsigned long long s_list_base;  // first entry of the list's claimed part
  // rows each lane's unit can touch (producer), and for each slot the rows
  // its tile's units so far can touch (consumers), in the caller's shared
  // memory (static arrays here would be repeated in every instantiation)
  uint32_t* const s_lane_rows = sm.rows;
  uint32_t* const s_slot_rows = sm.rows + 32;
  float* hist = sm.hist;
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const int warp = tid >> 5;
  const int ncw = (blockDim.x >> 5) - 1;  // consumer warps
  uint64_t* full = sm.bars;
  uint64_t* empty = sm.bars + stages;
  unsigned long long* unit_of = sm.units;
  if (tid == 0) {
    s_abort = 0;
    s_used = 0;
  }
  __syncthreads();
  const bool cull = NLOS_FWD_CULL && a.bounds != nullptr && MODE != MODE_NEAREST_COUNT;
  // bins tracked per tile (flush and zero only those)
  const bool ranged = RANGED && sm.rows != nullptr && cull && stages <= kMaxRangedStages;
  if (warp == 0) {
    // The whole warp walks the units 32 at a time: each lane tests one unit
    // against the bounds (unit_live), then lane 0 stages the live ones in
    // order. Chunk claims (lane 0) run one ahead of their use.
    const float margin = window_margin<MODE>(a);
    // list mode: chunks of the live-unit list, sized from its length
    const bool listed = a.unit_list != nullptr && chunk_counter != nullptr &&
                        sm.lane_units != nullptr;
    // the list's first list_static_pct percent (by weight, so that every CTA
    // gets as many live groups) goes to the CTAs in contiguous ranges (the
    // list holds each (tile, window)'s units together, so a CTA meets few tiles
    // there); the rest is claimed chunk by chunk (the claimed part's first entry
    // is kept in shared memory: it is read once per claim, and a register for it
    // spilled in the pair loop)
    unsigned long long s0 = 0, s1 = 0;  // the CTA's range
    if (lane == 0) s_list_base = 0;
    __syncwarp();
    if (listed) {
      const unsigned long long nl = *reinterpret_cast<const volatile unsigned long long*>(a.n_live);
      units_total = nl & 0xFFFFFFFFull;
      // chunks of a short list would hold too few units for the flush that
      // each costs: its whole weight goes out in the ranges (a ragged scan of
      // 1,500 live units: 66 against 76 us; a heightfield of 50,000 balances
      // better with claims, 1,062 against 1,257 us)
      const bool claimed = units_total * (100u - a.list_static_pct) / 100ull >=
                           4ull * gridDim.x * a.list_chunks_per_cta;
      const unsigned long long share = claimed ? (nl >> 32) * a.list_static_pct / 100ull : nl >> 32;
      const uint32_t x[3] = {(uint32_t)(share * blockIdx.x / gridDim.x),
                             (uint32_t)(share * (blockIdx.x + 1ull) / gridDim.x), (uint32_t)share};
      uint32_t at[3];
      list_lower_bounds(a.unit_list, (uint32_t)units_total, x, at);
      s0 = at[0];
      s1 = at[1];
      if (lane == 0) s_list_base = at[2];
      __syncwarp();
      chunk = (units_total - s_list_base) /
              ((unsigned long long)gridDim.x * a.list_chunks_per_cta);
      chunk = min(max(chunk, (unsigned long long)a.list_min_chunk),
                  (unsigned long long)a.list_max_chunk);
    }
    unsigned long long cur = u0, lim = u1, next = 0;
    bool have_next = false;  // a chunk claimed ahead of its use
    uint32_t claims = 0;
    auto claim = [&]() {
      unsigned long long c = 0;
      if (lane == 0) c = atomicAdd(chunk_counter, 1ull);
      ++claims;
      return __shfl_sync(0xffffffffu, c, 0);
    };
    if (chunk_counter) {
      const unsigned long long base = s_list_base;
      if (base > 0) {
        cur = s0;
        lim = s1;
      } else {
        const unsigned long long c = claim();
        cur = min(c * chunk, units_total);
        lim = min(cur + chunk, units_total);
      }
      if (cur < lim && (max_claims == 0 || claims < max_claims)) {
        next = claim();
        have_next = true;
      } else if (cur >= lim && base > 0) {
        // an empty static range: go straight to the claimed part
        const unsigned long long c = claim();
        cur = min(base + c * chunk, units_total);
        lim = min(cur + chunk, units_total);
        if (cur < lim && (max_claims == 0 || claims < max_claims)) {
          next = claim();
          have_next = true;
        }
      }
    }
    uint32_t k = 0;
    bool failed = false;
    unsigned long long run_tw = kNoUnit;  // (tile, window) of the last staged unit
    uint32_t run_rows = 0;   // union of the rows of its units so far
    unsigned long long slot_tw = kNoUnit; // of the open slot
    uint32_t fill = 0;       // pairs in the open slot (0: none is open)
    // hands the open slot to the consumers
    auto commit = [&]() {
      if (MODE == MODE_NEAREST_OCC) __syncwarp();  // (every lane wrote its groups' masks)
      if (lane == 0) {
        const int slot = (int)((it + k) % (uint32_t)stages);
        unit_of[slot] = slot_tw;
        sm.fill[slot] = fill;
        if (ranged) s_slot_rows[slot] = run_rows;
        mbar_arrive(&full[slot]);
      }
      ++k;
      fill = 0;
    };
    for (;;) {
      if (cur == lim && have_next) {
        cur = min(s_list_base + next * chunk, units_total);
        lim = min(cur + chunk, units_total);
        have_next = false;
        if (cur < lim && (max_claims == 0 || claims < max_claims)) {
          next = claim();
          have_next = true;
        }
      }
      if (cur >= lim) break;
      const uint32_t n = (uint32_t)min(32ull, lim - cur);
      bool live;
      if (listed) {
        // every list entry is live; its rows and groups were found with it
        live = lane < n;
        uint4 e = make_uint4(0u, 0u, 0u, 0u);
        if (live) e = reinterpret_cast<const uint4*>(a.unit_list)[cur + lane];
        sm.lane_units[lane] = e.x | ((unsigned long long)e.z << 32);
        if (ranged) s_lane_rows[lane] = e.y;
        __syncwarp();
      } else {
        float ulo = 0.f, uhi = 0.f;
        live = lane < n && (!cull || unit_live<SCAN, COS>(a, cur + lane, margin, ulo, uhi));
        if (ranged) {
          s_lane_rows[lane] = live ? unit_rows(ulo, uhi, margin, a.bw) : 0u;
          __syncwarp();
        }
      }
      uint32_t mask = __ballot_sync(0xffffffffu, live);
      // the groups of each unit that the tile may bin, packed densely: a slot
      // takes groups of as many units of one (tile, window) as fill it
      while (mask && !failed) {
        const int j = __ffs(mask) - 1;
        mask &= mask - 1;
        const unsigned long long unit = listed ? (sm.lane_units[j] & 0xFFFFFFFFull) : cur + j;
        uint32_t groups = listed ? (uint32_t)(sm.lane_units[j] >> 32)
                                 : unit_groups<SCAN, COS>(a, unit, margin, cull);
        if (groups == 0u) continue;
        const unsigned long long utw = unit / a.n_blk;
        if (fill > 0 && utw != slot_tw) commit();
        // each lane's group
        uint32_t group_occ = 0;
        if (MODE == MODE_NEAREST_OCC && ((groups >> lane) & 1u))
          group_occ = occ_bounds_mask(
              a.tiles[(uint32_t)(utw / a.n_win)],
              a.groups[((uint32_t)(unit - utw * a.n_blk) * a.ppb) / kGroupPairs + (uint32_t)lane], *occ);
        if (ranged) {
          const uint32_t ur = s_lane_rows[j];
          if (utw != run_tw) {
            run_tw = utw;
            run_rows = ur;
          } else {
            run_rows = min(run_rows & 0xFFFFu, ur & 0xFFFFu) |
                       (max(run_rows >> 16, ur >> 16) << 16);
          }
        }
        const uint32_t first = (uint32_t)(unit - utw * a.n_blk) * a.ppb;  // first pair of the block
        while (groups) {
          const uint32_t g = it + k;  // slot uses continue across calls
          const int slot = (int)(g % (uint32_t)stages);
          if (fill == 0) {  // open the next slot
            const uint32_t use = g / (uint32_t)stages;
            if (lane == 0 && use > 0 && !mbar_wait_bounded(&empty[slot], (use - 1) & 1)) {
              atomicOr(a.err, kErrWaitTimeout);
              s_abort = 1;
              failed = true;
            }
            failed = __shfl_sync(0xffffffffu, (int)failed, 0) != 0;
            if (failed) break;
            slot_tw = utw;
          }
          // the lowest groups that fit; only the last group of all is short
          const uint32_t room = a.ppb / kGroupPairs - fill / kGroupPairs;
          const uint32_t rank = (uint32_t)__popc(groups & ((1u << lane) - 1u));
          const bool take = ((groups >> lane) & 1u) && rank < room;
          const uint32_t taken = __ballot_sync(0xffffffffu, take);
          const uint32_t top = 31u - (uint32_t)__clz((int)taken);
          const uint32_t short_by =
              kGroupPairs - min(kGroupPairs, a.n_pairs - (first + top * kGroupPairs));
          const uint32_t added = (uint32_t)__popc(taken) * kGroupPairs - short_by;
          if (lane == 0) mbar_expect_tx(&full[slot], added * (uint32_t)sizeof(PointPair));
          __syncwarp();
          if (take) {
            const uint32_t p0 = first + (uint32_t)lane * kGroupPairs;
            if (MODE == MODE_NEAREST_OCC)
              sm.occ[slot * kOccGroups + fill / kGroupPairs + rank] = group_occ;
            fence_proxy_async_smem();
            bulk_g2s(sm.stage + (size_t)slot * a.ppb + fill + rank * kGroupPairs, a.pairs + p0,
                     min(kGroupPairs, a.n_pairs - p0) * (uint32_t)sizeof(PointPair), &full[slot]);
          }
          fill += added;
          groups &= ~taken;
          if (fill + kGroupPairs > a.ppb || short_by > 0) commit();
        }
      }
      if (failed) break;
      __syncwarp();
      cur += n;
    }
    if (fill > 0) commit();
    if (lane == 0) {
      if (!failed) {
        // end mark: no copy, a plain arrival completes the slot
        const uint32_t g = it + k;
        const int slot = (int)(g % (uint32_t)stages);
        const uint32_t use = g / (uint32_t)stages;
        if (use > 0 && !mbar_wait_bounded(&empty[slot], (use - 1) & 1)) {
          atomicOr(a.err, kErrWaitTimeout);
          s_abort = 1;
        } else {
          unit_of[slot] = kNoUnit;
          mbar_arrive(&full[slot]);
          ++k;
        }
      }
      // copies still in flight must land before the CTA exits or reuses the
      // stages: wait for the last use of every slot (bounded)
      for (uint32_t j = (k > (uint32_t)stages ? k - (uint32_t)stages : 0); j < k; ++j)
        (void)mbar_wait_bounded(&full[(it + j) % (uint32_t)stages],
                                ((it + j) / (uint32_t)stages) & 1);
      s_used = k;
    }
  } else {
    const int cw = warp - 1;
    const int nthr = ncw * 32;
    const uint32_t col_addr = smem_addr(hist) + (uint32_t)lane * 4u;
    TileState ts;
    uint32_t tile_rows = (uint32_t)a.bw << 16;  // rows of the current tile that may be nonzero
    for (uint32_t k = 0;; ++k) {
      const uint32_t g = it + k;
      const int slot = (int)(g % (uint32_t)stages);
      const uint32_t use = g / (uint32_t)stages;
      if (*(volatile int*)&s_abort != 0) break;
      if (!mbar_wait_bounded(&full[slot], use & 1)) {
        if (lane == 0) {
          atomicOr(a.err, kErrWaitTimeout);
          s_abort = 1;
        }
        break;
      }
      const unsigned long long tag = *(volatile unsigned long long*)&unit_of[slot];
      if (tag != kNoUnit) {
        const long long tw = (long long)tag;
        if (tw != ts.tw) {
          named_barrier(1, nthr);  // every consumer is done with the previous tile
          if (ts.tw >= 0) {
            if constexpr (MODE == MODE_SPLAT_MOM)
              flush_tile_mom(a, *mt, ts.tw, hist, cw, ncw, (int)(tile_rows & 0xFFFFu),
                             (int)(tile_rows >> 16));
            else flush_tile<MODE>(a, ts.tw, hist, cw, ncw, (int)(tile_rows & 0xFFFFu),
                                  (int)(tile_rows >> 16));
            named_barrier(1, nthr);
          }
          // zero what the previous tile may have written (everything the first
          // time: the buffer may hold another item's data)
          const uint32_t per_bin = (uint32_t)(mom_q * kTile);
          const uint32_t z0 = (ranged && ts.tw >= 0) ? (tile_rows & 0xFFFFu) * per_bin : 0u;
          const uint32_t z1 = ((ranged && ts.tw >= 0) ? (tile_rows >> 16) : a.bw) * per_bin;
          for (int n = 0; n < (MODE == MODE_SPLAT_MOM ? kMoments : 1); ++n)
            for (uint32_t i = z0 + tid - 32; i < z1; i += nthr) hist[n * kMomRows * kTile + i] = 0.f;
          load_tile(a, tw, lane, ts, SCAN == NLOS_CONFOCAL, window_margin<MODE>(a));
          named_barrier(1, nthr);
        }
        // the producer's running union for this tile, up to this unit
        if (ranged) tile_rows = s_slot_rows[slot];
        compute_block<SCAN, COS, MODE, UNROLL>(a, sm.stage + (size_t)slot * a.ppb,
                                               *(volatile uint32_t*)&sm.fill[slot], cw, ncw, ts,
                                               col_addr, cnt, mom_q, occ,
                                               sm.occ + slot * kOccGroups, g);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[slot]);
      if (tag == kNoUnit) break;
    }
    named_barrier(1, nthr);
    if (ts.tw >= 0) {
      if constexpr (MODE == MODE_SPLAT_MOM)
        flush_tile_mom(a, *mt, ts.tw, hist, cw, ncw, (int)(tile_rows & 0xFFFFu),
                       (int)(tile_rows >> 16));
      else flush_tile<MODE>(a, ts.tw, hist, cw, ncw, (int)(tile_rows & 0xFFFFu),
                            (int)(tile_rows >> 16));
    }
  }
  __syncthreads();
  it += s_used;
  return s_abort == 0;
}

}  // namespace nlos

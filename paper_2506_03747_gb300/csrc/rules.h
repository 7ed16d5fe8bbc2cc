// Host rules that choose between the forms of a kernel, from sizes alone
// (plain C++, so that they can be checked without a GPU).
#pragma once

#include <cmath>
#include <cstdint>

namespace nlos {

constexpr int kMomMaxJ = 60;
constexpr int kMomTaps = 144;  // (2J + 1) q at most: 121 at q = 1, 66, 92, 104, 144 at q = 2 .. 16

// Moment form of the splat: rows a bin (forward_core.cuh).
inline int moment_rows_per_bin(double sigma) {
  int q = 1;
  if (sigma < 2.5)
    while (0.5 / q > 0.16 * sigma) q *= 2;
  return q;
}

// Splat kernels whose taps fit the moment table (sigma up to 9.8 bins); wider
// ones run their taps pair by pair.
inline bool moments_fit(double sigma) { return (int)std::ceil(6.0 * sigma) + 1 <= kMomMaxJ; }

// Forward of a splat over B bins of P points: moments or taps. A pair costs six
// reductions against about 12 sigma, but finer rows cut a transient into more
// windows, each with its zeroing and its flush, whatever the number of points.
//  * two rows a bin and fewer (sigma from 1.5625): moments, 1.2 to 28 times faster
//    (0.9 at worst, 64 x 64 scan of 1,000 points over 1,024 bins: 224 / 205 us);
//  * four rows (from 0.78125): moments where P sigma^4 >= 8 B. Moments / taps, us:
//    32 x 32 scan, 8,000 points, 512 bins, sigma 0.8: 186 / 139, 1.0: 189 / 352;
//    64 x 64 scan, 4,000 points, 1,024 bins, sigma 1.0: 428 / 328, 1.5: 483 / 678;
//  * more rows: taps (64 x 64 scan, 16,000 points, 512 bins, sigma 0.35: 3,103 /
//    617, 0.7: 1,535 / 908; only very many points over few bins reverse it,
//    128 x 128 scan, 65,536 points, 256 bins, sigma 0.7: 6,246 / 8,192).
inline bool forward_moments(double sigma, uint64_t P, uint32_t B) {
  const int q = moment_rows_per_bin(sigma);
  if (!moments_fit(sigma) || q > 4) return false;
  return q <= 2 || (double)P * (sigma * sigma) * (sigma * sigma) >= 8.0 * B;
}

// The adjoint of the same: the moment tables cost S B q (2J + 1) products before
// the first pair, the taps of a pair 12 sigma gathers. From two rows a bin up the
// tables always pay (1.4 times and more); below, with enough points a bin.
// Moments / taps, us: 64 x 64 scan over 512 bins, sigma 0.35: 16,000 points 1,893 /
// 861, 100,000 4,337 / 5,052; sigma 0.7: 893 / 998 and 2,679 / 5,916; 64 x 64 scan
// over 1,024 bins, sigma 0.8: 1,000 points 428 / 238, 4,000 542 / 817. The taps
// form holds [B][32] floats in shared memory: beyond 832 bins one CTA fills an
// SM, and the line lies at a quarter of the points (48 x 48 scan, 32,000 points,
// 1,024 bins, sigma 0.35: 2,086 / 3,073).
constexpr uint32_t kAdjOneCtaBins = 832;
inline bool adjoint_moments(double sigma, uint64_t P, uint32_t B) {
  if (!moments_fit(sigma)) return false;
  const int q = moment_rows_per_bin(sigma);
  if (q <= 2) return true;
  if (q == 4) return 2 * P >= 3ull * B;
  return P >= (B > kAdjOneCtaBins ? 1ull : 4ull) * (uint64_t)q * B;
}

// Pairs of a staged block: `most`, halved while the scene has fewer units (tile,
// window, block) than SMs, so that more SMs take part (the 32 x 32 scan of 1,024
// points has 32 units of 1,024: 32.1 us a pass in one block, 22 us in blocks of 128
// points).
constexpr uint32_t kFwdMinPpb = 64;
inline uint32_t block_pairs(uint32_t most, uint64_t n_tiles, uint64_t n_win, uint64_t n_pairs,
                            uint64_t sms) {
  uint32_t ppb = most;
  while (ppb > kFwdMinPpb && n_tiles * n_win * ((n_pairs + ppb - 1) / ppb) < sms) ppb /= 2;
  return ppb;
}

// The forward's live-unit list is 16 bytes a unit and belongs to the scene, so it
// is bounded to 64 MiB: a longer one is made and worked off in passes of whole
// (tile, window) runs of n_blk units, as many as kListEntries hold and at least
// one. A pass costs its tail and two launches: 256 x 256 scan, 4,194,304 points,
// 512 bins: 92.4 ms in one pass of 134 MB, 92.6 in 2 passes, 96.3 in 8 of 16 MiB;
// 512 x 512 scan, 300,000 points: 4.27 ms in one pass, 4.45 in 3 of 16 MiB.
constexpr uint64_t kListEntries = 1ull << 22;
inline uint64_t list_pass_runs(uint64_t runs, uint64_t n_blk) {
  uint64_t most = kListEntries / n_blk;
  if (most < 1) most = 1;
  const uint64_t passes = (runs + most - 1) / most;
  return (runs + passes - 1) / passes;
}

}  // namespace nlos

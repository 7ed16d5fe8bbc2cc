// Detector model kernels of the GB300 NLOS simulator (arXiv 2506.03747):
//  * Gaussian timing jitter per transient (Eq. 16/17, Algorithm 1 step 2.3);
//  * per-transient FP64 energy, and the cube's maximum / FP64 sum and sum of
//    squares that set the noise scale;
//  * seeded Poisson photon + dark-count noise (Eq. 18/19, Algorithm 1 step 2.4)
//    from per-bin Philox4x32-10 counter streams.
// All three are HBM-streaming kernels: coalesced row-wise reads and writes,
// grids sized to the SM count.
#include "common.cuh"
#include "device_util.cuh"
#include "noise_core.cuh"
#include "reduce_core.cuh"

#include <algorithm>
#include <cmath>

namespace nlos {

// ---------------------------------------------------------------------------
// Jitter taps: sigma in bins, R = ceil(2 sigma), k = 2R + 1 (Eq. 17), sampled
// Gaussian exp(-j^2 / (2 sigma^2)) normalised to sum 1 (computed in FP64 on
// the host, stored FP32). sigma = 0 gives the identity (k = 1).
// ---------------------------------------------------------------------------
int jitter_taps(double sigma, float* taps, int max_taps) {
  const int R = jitter_radius(sigma);
  const int k = 2 * R + 1;
  if (k > max_taps) return -k;
  if (R == 0) {
    taps[0] = 1.0f;
    return 1;
  }
  static thread_local double t[4097];
  double sum = 0.0;
  for (int j = -R; j <= R; ++j) {
    t[j + R] = std::exp(-(double)j * (double)j / (2.0 * sigma * sigma));
    sum += t[j + R];
  }
  for (int j = 0; j < k; ++j) taps[j] = (float)(t[j] / sum);
  return k;
}

void jitter_tails(const float* taps, int R, float* tail) {
  double acc = 0.0;  // running sum from the outermost tap inwards
  for (int k = R - 1; k >= 0; --k) {
    acc += (double)taps[R + k + 1];
    tail[k] = (float)acc;
  }
}

constexpr int kJitterMaxTaps = 2049;  // R <= 1024 bins
constexpr int kJitterTile = 1024;     // output bins of a CTA at most (staged form)
constexpr int kJitterUnrolled = 16;   // radii with a compile-time unrolled form

template <int kTaps>
struct JitterArgs {
  const float* in;
  float* out;
  uint64_t traces;
  uint32_t B;
  int R;
  int replicate;  // 1: the edge bins continue outside the trace
  uint32_t tiles, len;  // runs of a trace and their length (a multiple of a thread's bins)
  float taps[kTaps];
};
using JitterShort = JitterArgs<2 * kJitterUnrolled + 1>;
using JitterLong = JitterArgs<kJitterMaxTaps>;

// Two forms, both HBM-bound (8 bytes a bin) once a thread computes several
// consecutive bins from one window of registers; one bin a thread, each with
// its own 2R + 1 shared loads, was bound by those loads (16,384 x 1024 bins,
// R = 7: 86 us; now 22.6 us, 5.9 TB/s).
//  * rows of 16-byte alignment: each thread takes 8 bins from the 8 + 2R
//    inputs around them, read straight from global memory (neighbouring
//    threads' overlap hits L1), so no barrier separates loads and stores;
//  * other rows (bin counts that are not multiples of 4, unaligned buffers)
//    and radii above 16: a run of the trace with its halo is staged in shared
//    memory by coalesced loads, and each thread takes 4 bins from it. Above 16 the
//    loop over the taps reads the halo as 16-byte words (16,384 x 1024 bins, R = 40:
//    106 us, R = 200: 381 us; with one word a tap 160 and 701, and one bin a
//    thread 157 and 698). Bound: FMA issue and the taps' indexed constant loads.
// Every bin adds its taps in the same order in all forms.
template <int R>
__global__ void __launch_bounds__(256) jitter_direct_kernel(const __grid_constant__ JitterShort a) {
  constexpr int kQ = (R + 3) / 4;  // 16-byte words of halo on each side
  const uint64_t t = blockIdx.x / a.tiles;
  const int b0 = (int)(blockIdx.x % a.tiles * a.len + 8 * threadIdx.x);
  const int B = (int)a.B;
  if (b0 >= B || 8 * threadIdx.x >= a.len) return;
  const float* row = a.in + t * a.B;
  float x[8 + 8 * kQ];
#pragma unroll
  for (int q = 0; q < 2 + 2 * kQ; ++q) {
    const int b = b0 + 4 * (q - kQ);  // a multiple of 4: the word lies inside or outside as a whole
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (b >= 0 && b < B) {
      v = __ldg(reinterpret_cast<const float4*>(row + b));
    } else if (a.replicate) {
      const float e = __ldg(row + (b < 0 ? 0 : B - 1));
      v = make_float4(e, e, e, e);
    }
    x[4 * q] = v.x;
    x[4 * q + 1] = v.y;
    x[4 * q + 2] = v.z;
    x[4 * q + 3] = v.w;
  }
  float acc[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    acc[e] = 0.0f;
#pragma unroll
    for (int j = -R; j <= R; ++j) acc[e] = fmaf(a.taps[j + R], x[4 * kQ + e - j], acc[e]);
  }
  float4* o = reinterpret_cast<float4*>(a.out + t * a.B + b0);
  o[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
  if (b0 + 4 < B) o[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
}

// RT >= 0: the radius at compile time; -1: a.R.
template <int RT, class Args>
__global__ void __launch_bounds__(256) jitter_kernel(const __grid_constant__ Args a) {
  extern __shared__ __align__(16) float sm[];  // [halo + len + halo], halo a multiple of 4
  const int R = RT >= 0 ? RT : a.R;
  const int halo = (R + 3) & ~3;
  const uint64_t t = blockIdx.x / a.tiles;
  const int b0 = (int)(blockIdx.x % a.tiles * a.len);
  const float* row = a.in + t * a.B;
  for (int i = threadIdx.x; i < (int)a.len + 2 * halo; i += blockDim.x) {
    const int b = b0 - halo + i;
    if (a.replicate) sm[i] = row[min(max(b, 0), (int)a.B - 1)];
    else sm[i] = (b >= 0 && b < (int)a.B) ? row[b] : 0.0f;
  }
  __syncthreads();
  const int o = 4 * (int)threadIdx.x;
  if (o >= (int)a.len) return;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  if (RT >= 0) {
    constexpr int kQ = ((RT >= 0 ? RT : 0) + 3) / 4;
    float x[4 + 8 * kQ];
#pragma unroll
    for (int q = 0; q < 1 + 2 * kQ; ++q) {
      const float4 v = *reinterpret_cast<const float4*>(sm + o + 4 * q);
      x[4 * q] = v.x;
      x[4 * q + 1] = v.y;
      x[4 * q + 2] = v.z;
      x[4 * q + 3] = v.w;
    }
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
      for (int j = -RT; j <= RT; ++j) acc[e] = fmaf(a.taps[j + RT], x[4 * kQ + e - j], acc[e]);
  } else {
    // out[b] = sum_j taps[j + R] * in[b - j]; in[b - j] sits at sm[o + e + halo - j].
    // Four taps take the seven inputs of two 16-byte words, one of them new (read
    // one by one, a warp's inputs 16 bytes apart met in the same banks).
    const float* c = sm + o + halo;
    int j = -R;
    auto one = [&]() {
      const float g = a.taps[j + R];
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[e] = fmaf(g, c[e - j], acc[e]);
      ++j;
    };
    while (j & 3) one();
    float4 hi = *reinterpret_cast<const float4*>(c - j);
#pragma unroll 4
    for (; j + 3 <= R; j += 4) {
      const float4 lo = *reinterpret_cast<const float4*>(c - j - 4);
      const float x[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float g = a.taps[j + k + R];
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[e] = fmaf(g, x[4 + e - k], acc[e]);
      }
      hi = lo;
    }
    while (j <= R) one();
  }
  float* orow = a.out + t * a.B + b0;
#pragma unroll
  for (int e = 0; e < 4; ++e)
    if (b0 + o + e < (int)a.B) orow[o + e] = acc[e];
}

template <int R>
void run_jitter(const JitterShort& a, bool direct, unsigned blocks, unsigned threads, size_t smem,
                cudaStream_t st) {
  if constexpr (R >= 0) {
    if (a.R != R) run_jitter<R - 1>(a, direct, blocks, threads, smem, st);
    else if (direct) jitter_direct_kernel<R><<<blocks, threads, 0, st>>>(a);
    else jitter_kernel<R><<<blocks, threads, smem, st>>>(a);
  }
}

cudaError_t launch_jitter(const float* in, float* out, uint64_t traces, uint32_t B, double sigma,
                          int replicate, cudaStream_t st) {
  if (traces == 0 || B == 0) return cudaSuccess;
  JitterLong a;
  a.in = in;
  a.out = out;
  a.traces = traces;
  a.B = B;
  a.replicate = replicate;
  const int k = jitter_taps(sigma, a.taps, kJitterMaxTaps);
  if (k < 0) return cudaErrorInvalidValue;
  a.R = (k - 1) / 2;
  const bool direct = a.R <= kJitterUnrolled && (B & 3u) == 0 &&
                      ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15u) == 0;
  // equal runs of a trace, so that no CTA is left with a short remainder
  const uint32_t per = direct ? 8u : 4u, most = direct ? 256u * 8u : (uint32_t)kJitterTile;
  a.tiles = (B + most - 1) / most;
  a.len = ((B + a.tiles - 1) / a.tiles + per - 1) / per * per;
  a.tiles = (B + a.len - 1) / a.len;
  const unsigned blocks = (unsigned)(traces * a.tiles);
  const unsigned threads = (a.len / per + 31u) & ~31u;
  const size_t smem = direct ? 0 : sizeof(float) * (a.len + 2 * ((a.R + 3) & ~3));
  if (a.R > kJitterUnrolled) {
    jitter_kernel<-1><<<blocks, threads, smem, st>>>(a);
  } else {
    JitterShort s{in, out, traces, B, a.R, replicate, a.tiles, a.len, {}};
    std::copy(a.taps, a.taps + k, s.taps);
    run_jitter<kJitterUnrolled>(s, direct, blocks, threads, smem, st);
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Reductions: one warp per transient. energy[t] = sum_b tau[t][b] to FP64
// accuracy (trace_sums, reduce_core.cuh: error-free FP32 pair sums per lane);
// the cube's maximum, FP64 sum and sum of squares are combined per CTA in
// shared memory, then one atomicMax on the float bits (tau >= 0 orders like
// its bits) and two double atomicAdds per CTA (per-warp atomics on the same
// three words serialised in L2).
// ---------------------------------------------------------------------------
constexpr int kReduceThreads = 256;

__global__ void __launch_bounds__(kReduceThreads) reduce_kernel(const float* __restrict__ tau,
                                                                uint64_t traces, uint32_t B,
                                                                double* energy,
                                                                SceneScratch* scratch) {
  __shared__ double s_sum[kReduceThreads / 32], s_sq[kReduceThreads / 32];
  __shared__ float s_max[kReduceThreads / 32];
  const int lane = threadIdx.x & 31;
  const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
  double csum = 0.0, csq = 0.0;
  float cmax = 0.0f;
  for (uint64_t t = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < traces;
       t += warps) {
    double s, q;
    float m;
    trace_sums(tau + t * B, B, lane, s, q, m);
    if (lane == 0 && energy) energy[t] = s;
    csum += s;
    csq += q;
    cmax = fmaxf(cmax, m);
  }
  if (!scratch) return;
  const int warp = threadIdx.x >> 5;
  if (lane == 0) {
    s_sum[warp] = csum;
    s_sq[warp] = csq;
    s_max[warp] = cmax;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
      csum += s_sum[w];
      csq += s_sq[w];
      cmax = fmaxf(cmax, s_max[w]);
    }
    atomicMax(&scratch->peak_bits, __float_as_uint(cmax));
    atomicAdd(&scratch->sum, csum);
    atomicAdd(&scratch->sumsq, csq);
  }
}

__global__ void stats_out_kernel(const SceneScratch* scratch, double* stats) {
  stats[0] = (double)__uint_as_float(scratch->peak_bits);
  stats[1] = scratch->sum;
  stats[2] = scratch->sumsq;
}

cudaError_t launch_stats_out(const SceneScratch* scratch, double* stats, cudaStream_t st) {
  stats_out_kernel<<<1, 1, 0, st>>>(scratch, stats);
  return cudaGetLastError();
}

cudaError_t launch_reduce(const float* tau, uint64_t traces, uint32_t B, double* energy,
                          SceneScratch* scratch, cudaStream_t st) {
  if (traces == 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const uint64_t want = (traces + 7) / 8;
  const unsigned blocks = (unsigned)(want < (uint64_t)sms * 8 ? want : (uint64_t)sms * 8);
  reduce_kernel<<<blocks, kReduceThreads, 0, st>>>(tau, traces, B, energy, scratch);
  return cudaGetLastError();
}

struct NoiseArgs {
  const float* tau;
  uint32_t* counts;
  uint64_t n;
  uint64_t index_base;
  uint64_t seed;
  uint32_t tag;
  float scale, dark;          // used when scratch == nullptr
  SceneScratch* scratch;      // else: scale from the reduced cube
  int mode;                   // nlos_noise_mode (scratch path)
  float peak_photons, dark_cfg, nr_db;
  const double* cube_stats;   // part of a larger cube: {max, sum, sumsq} of the whole
  uint64_t cube_bins;         // bins of the whole cube
  DeferList defer;            // deferred bright bins (defer.hdr null: one pass)
};

// CTAs of 7 warps, kNoiseBlocksPerSm resident per SM (32 registers), up to
// NLOS_NOISE_WAVES waves of them. A thread samples one group of four bins at a
// time (one Philox block for the four first draws, a 16-byte load and store);
// warp w takes the 32 consecutive groups of chunk c = w, w + W, w + 2W, ...
// (lane = group, coalesced). The warp count W is odd, so the stride W * 128
// bins moves a warp's bins through the time indices of the transients: a
// bin's cost grows with its lambda and the bright bins sit at a few time
// indices, and a stride that is a multiple of the bin count (a wave of
// 256-thread blocks of 1024-bin transients: 1216 * 256 = 304 * 1024) gave some
// warps every bright bin of the cube (ncu: SMs 40% active, ALU pipe from 19%
// to 99% over the SMs). A few waves of short CTAs balance the bright bins (16,384
// x 1,024 bins, mean 1 count: 2 / 4 / 16 waves 103.8 / 102.1 / 102.8 us of
// detector, and 69.7 / 67.0 / 72.3 us at a twentieth of the light). No atomics and
// no divisions in the loop. Bound: ALU issue; that detector took 140.6 us with a
// 13-instruction search step, an integer conversion a bin and tables of 1/k that
// each short CTA filled.
constexpr int kNoiseWarps = 7;
constexpr int kNoiseThreads = 32 * kNoiseWarps;
constexpr int kNoiseBlocksPerSm = 8;
#ifndef NLOS_NOISE_WAVES
#define NLOS_NOISE_WAVES 4   // resident waves of CTAs at most (the rest by the grid stride)
#endif

#ifndef NLOS_NOISE_DEFER
#define NLOS_NOISE_DEFER 1  // bins with lambda >= 30 sampled by a second kernel
#endif

// The noise scale and dark level of a launch (the same in every thread and
// in both kernels of a launch).
__device__ __forceinline__ void launch_scale(const NoiseArgs& a, float& scale, float& dark) {
  scale = a.scale;
  dark = a.dark;
  if (a.cube_stats) {
    scale = noise_scale_of((float)a.cube_stats[0], a.cube_stats[1], a.cube_stats[2], a.mode,
                           a.peak_photons, a.nr_db, a.cube_bins);
    dark = a.dark_cfg;
  } else if (a.scratch) {
    scale = noise_scale_from(a.scratch, a.mode, a.peak_photons, a.nr_db, a.n);
    dark = a.dark_cfg;
  }
}

template <bool DEFER>
__global__ void __launch_bounds__(kNoiseThreads, kNoiseBlocksPerSm) noise_kernel(const NoiseArgs a) {
  float scale, dark;
  launch_scale(a, scale, dark);
  if (a.scratch && blockIdx.x == 0 && threadIdx.x == 0) {
    a.scratch->scale = scale;
    a.scratch->dark = dark;
  }
  const uint64_t stride = (uint64_t)gridDim.x * kNoiseWarps * 32;
  const uint64_t j0 = ((uint64_t)blockIdx.x * kNoiseWarps + (threadIdx.x >> 5)) * 32 +
                      (threadIdx.x & 31);
  noise_groups<DEFER>(a.tau, a.counts, 0, a.n, a.index_base, scale, dark, a.seed, a.tag, j0,
                      stride, &a.defer);
}

// Second pass (after noise_kernel, in stream order): one thread per listed
// bin (the cube's bright bins, about 1% of them), then one warp per listed
// region of a warp whose bins did not fit the list.
constexpr int kDeferThreads = 256;

__global__ void __launch_bounds__(kDeferThreads) noise_deferred_kernel(const NoiseArgs a) {
  float scale, dark;
  launch_scale(a, scale, dark);
  const DeferList& d = a.defer;
  const unsigned long long claimed = *(volatile unsigned long long*)&d.hdr[0];
  const unsigned long long nd = claimed < d.cap ? claimed : d.cap;
  const uint64_t nt = (uint64_t)gridDim.x * kDeferThreads;
  for (uint64_t k = (uint64_t)blockIdx.x * kDeferThreads + threadIdx.x; k < nd; k += nt) {
    const uint32_t l = d.bins[k];
    if (l != kDeferredCount)
      noise_deferred_bin(a.tau, a.counts, l, a.index_base, scale, dark, a.seed, a.tag);
  }
  const unsigned long long nr = *(volatile unsigned long long*)&d.hdr[1];
  const uint64_t nw = nt / 32;
  for (uint64_t k = (uint64_t)blockIdx.x * (kDeferThreads / 32) + (threadIdx.x >> 5); k < nr;
       k += nw)
    noise_deferred_warp(a.tau, a.counts, a.n, d.regions[k], a.index_base, scale, dark, a.seed,
                        a.tag);
}

// Sizes of the deferred-bin lists: entries of the dense list, warp regions.
uint64_t noise_cap(uint64_t n) { return std::min<uint64_t>(n, n / 32 + 4096); }
uint64_t noise_groups_of(uint64_t n, uint64_t index_base) {
  return ((index_base + n + 3) >> 2) - (index_base >> 2);
}
uint64_t noise_regions(uint64_t n, uint64_t index_base) {
  return noise_groups_of(n, index_base) / 32 + 2;
}

size_t noise_list_bytes(uint64_t n, uint64_t index_base) {
  if (!NLOS_NOISE_DEFER || n == 0 || n >= 0xFFFFFFFFull) return 0;
  return noise_regions(n, index_base) * sizeof(unsigned long long) +
         ((noise_cap(n) * sizeof(uint32_t) + 15) & ~(size_t)15);
}

cudaError_t launch_noise_impl(const NoiseArgs& a, cudaStream_t st, void* lists = nullptr) {
  if (a.n == 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const uint64_t groups = noise_groups_of(a.n, a.index_base);
  const uint64_t want = (groups + kNoiseThreads - 1) / kNoiseThreads;
  const uint64_t wave = (uint64_t)sms * kNoiseBlocksPerSm * NLOS_NOISE_WAVES;
  uint64_t blocks = want < wave ? want : wave;
  if (blocks > 1 && (blocks & 1u) == 0) --blocks;  // an odd number of warps (7 per block)
  // the deferred-bin lists: a dense list of local indices for about 3% of the
  // bins, and one entry per warp region for the warps whose bins overflow it
  // (the regions of 32 groups cover the launch's groups, plus one for an
  // unaligned start). A scene keeps them (with their header in its scratch);
  // elsewhere they are a stream-ordered allocation with the header in front,
  // freed after the second pass. Without them (or for parts of 2^32 - 1 bins or
  // more) every bin is sampled in one pass.
  NoiseArgs b = a;
  b.defer = DeferList{};
  cudaError_t e = cudaSuccess;
  void* buf = nullptr;
  const size_t bytes = noise_list_bytes(a.n, a.index_base);
  if (lists && bytes) {
    b.defer.hdr = a.scratch->deferred;
    b.defer.regions = static_cast<unsigned long long*>(lists);
  } else if (bytes) {
    const size_t hdr = 2 * sizeof(unsigned long long);
    if (cudaMallocAsync(&buf, hdr + bytes, st) != cudaSuccess) {
      buf = nullptr;
      (void)cudaGetLastError();  // no lists: one pass
    } else if ((e = cudaMemsetAsync(buf, 0, hdr, st)) != cudaSuccess) {
      cudaFreeAsync(buf, st);
      return e;
    } else {
      b.defer.hdr = static_cast<unsigned long long*>(buf);
      b.defer.regions = b.defer.hdr + 2;
    }
  }
  if (b.defer.hdr) {
    b.defer.bins = reinterpret_cast<uint32_t*>(b.defer.regions + noise_regions(a.n, a.index_base));
    b.defer.cap = (uint32_t)noise_cap(a.n);
  }
  if (b.defer.hdr)
    noise_kernel<true><<<(unsigned)blocks, kNoiseThreads, 0, st>>>(b);
  else
    noise_kernel<false><<<(unsigned)blocks, kNoiseThreads, 0, st>>>(b);
  e = cudaGetLastError();
  if (b.defer.hdr) {
    if (e == cudaSuccess) {
      noise_deferred_kernel<<<(unsigned)(sms * 4), kDeferThreads, 0, st>>>(b);
      e = cudaGetLastError();
    }
  }
  if (buf) {
    const cudaError_t ef = cudaFreeAsync(buf, st);
    if (e == cudaSuccess) e = ef;
  }
  return e;
}

cudaError_t launch_noise(const float* tau, uint64_t n, float scale, float dark, uint64_t seed,
                         uint32_t tag, uint64_t index_base, uint32_t* counts, cudaStream_t st) {
  NoiseArgs a{};
  a.tau = tau;
  a.counts = counts;
  a.n = n;
  a.index_base = index_base;
  a.seed = seed;
  a.tag = tag;
  a.scale = scale;
  a.dark = dark;
  a.scratch = nullptr;
  return launch_noise_impl(a, st);
}

cudaError_t launch_noise_scene(const float* tau, uint64_t n, SceneScratch* scratch, int mode,
                               float peak_photons, float dark, float nr_db, uint64_t seed,
                               uint32_t tag, uint32_t* counts, cudaStream_t st,
                               uint64_t index_base, const double* cube_stats,
                               uint64_t cube_bins, void* lists) {
  NoiseArgs a{};
  a.tau = tau;
  a.counts = counts;
  a.n = n;
  a.index_base = index_base;
  a.cube_stats = cube_stats;
  a.cube_bins = cube_bins;
  a.seed = seed;
  a.tag = tag;
  a.scratch = scratch;
  a.mode = mode;
  a.peak_photons = peak_photons;
  a.dark_cfg = dark;
  a.nr_db = nr_db;
  return launch_noise_impl(a, st, lists);
}

// ---------------------------------------------------------------------------
// Raw Philox words (parity testing of the device generator).
// ---------------------------------------------------------------------------
__global__ void philox_kernel(const uint4* ctr, uint64_t n, uint32_t k0, uint32_t k1, uint4* out) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
    out[i] = philox4x32_10(ctr[i], k0, k1);
}

cudaError_t launch_philox(const uint32_t* ctr, uint64_t n, uint32_t k0, uint32_t k1,
                          uint32_t* out, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const uint64_t want = (n + 255) / 256;
  const unsigned blocks = (unsigned)(want < 4096 ? want : 4096);
  philox_kernel<<<blocks, 256, 0, st>>>(reinterpret_cast<const uint4*>(ctr), n, k0, k1,
                                        reinterpret_cast<uint4*>(out));
  return cudaGetLastError();
}

}  // namespace nlos

// The paper's FFT forward model (the light-cone-transform convolution of the
// Theory section, Algorithm 1 steps 1.1-2.2) for an N x N confocal depth map
// with M time bins (N, M powers of two):
//   tau = R_t^{-1} F^{-1}[ F(R_z V) . F(PSF) ]
// on a zero-padded (2N) x (2N) x (2M) grid.
//
// Readings (as in the oracle): V holds albedo at depth bin D[x, y]; R_z maps
// depth bin j (1-based) to squared-depth sample ceil(j^2 / M) with weight
// 1 / (j M^2) (the perfect-square rows of the printed fine matrix, averaged
// over log2 M levels of (1/2) S_k); R_t^{-1} reads time bin j from sample
// ceil(j^2 / M) with weight M / j^4 (the v^{-3/2} factor that Eq. 3 implies);
// the PSF has one node per (x, y) column, the z node nearest
// (4 slope)^2 (x^2 + y^2), slope = w / (M c dt), circularly shifted so that
// node (N, N, M) is the origin.
//
// Arithmetic: FP64 throughout. The time resampling weights the earliest bins
// by up to M / 1 against M / j^4 at the signal, so FP32 round-off of the
// transforms (1e-7 of the largest value) would exceed the signal there.
//
// Two forms of the convolution, chosen by the plan's sizes (direct_form):
//  * direct: both factors are sparse, R_z V with one sample a depth-map pixel
//    and the PSF with one node a column, so the convolution is N^4 additions
//    into [N][N][M] (one per pixel and scan point that meet in the window),
//    with no padding and no transform round-off;
//  * FFT: for short time axes under wide maps, where N^4 additions cost more
//    than transforms of the padded volume. Its work volume is [2N][2N][2M]
//    complex (time fastest); each 1-D transform runs in shared memory
//    (bit-reversed load, log2 L radix-2 stages); along x and y a CTA takes
//    several lines adjacent in time so that its loads and stores are coalesced.
#include "common.cuh"

#include <cmath>
#include <new>
#include <vector>

namespace nlos {
namespace {

constexpr int kFftThreads = 256;
constexpr size_t kFftSmem = 64 * 1024;  // bytes of lines per CTA

struct LctDims {
  uint32_t N, M;   // depth map side, bins
  uint32_t n2, m2; // 2N, 2M
};

// Lines of length L along one axis of the [2N][2N][2M] volume: line
// (o, i) starts at o * outer_stride + i (i < n_inner, consecutive in memory)
// and its samples are s_stride apart. A CTA takes T lines (o, i0..i0+T-1).
struct FftArgs {
  double2* data;
  const double2* tw;  // exp(-2 pi i k / Lmax), k < Lmax / 2
  uint32_t L, log2L, T, tw_step;
  uint64_t s_stride, outer_stride, n_inner;
  int inverse;         // conjugate twiddles and scale by 1 / L
};

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__global__ void __launch_bounds__(kFftThreads) fft_lines_kernel(const FftArgs a) {
  extern __shared__ double2 buf[];  // [T][L]
  const uint64_t groups_per_outer = (a.n_inner + a.T - 1) / a.T;
  const uint64_t o = blockIdx.x / groups_per_outer;
  const uint64_t i0 = (blockIdx.x % groups_per_outer) * a.T;
  const uint32_t nl = (uint32_t)min((uint64_t)a.T, a.n_inner - i0);
  const uint64_t base = o * a.outer_stride + i0;
  // load, bit-reversed within each line; consecutive threads take
  // consecutive lines of one sample (coalesced when s_stride > 1)
  for (uint32_t e = threadIdx.x; e < a.L * nl; e += blockDim.x) {
    const uint32_t s = a.s_stride == 1 ? e % a.L : e / nl;
    const uint32_t l = a.s_stride == 1 ? e / a.L : e % nl;
    const uint32_t r = __brev(s) >> (32 - a.log2L);
    buf[l * a.L + r] = a.data[base + l + (uint64_t)s * a.s_stride];
  }
  __syncthreads();
  const uint32_t half = a.L / 2;
  for (uint32_t m = 1; m < a.L; m <<= 1) {
    const uint32_t step = (a.L / (2 * m)) * a.tw_step;  // twiddle index stride
    for (uint32_t b = threadIdx.x; b < half * nl; b += blockDim.x) {
      const uint32_t l = b / half, k = b % half;
      const uint32_t j = k % m;
      const uint32_t i1 = (k / m) * 2 * m + j, i2 = i1 + m;
      double2 w = a.tw[j * step];
      if (a.inverse) w.y = -w.y;
      double2* line = buf + l * a.L;
      const double2 x = line[i1];
      const double2 y = cmul(w, line[i2]);
      line[i1] = make_double2(x.x + y.x, x.y + y.y);
      line[i2] = make_double2(x.x - y.x, x.y - y.y);
    }
    __syncthreads();
  }
  const double sc = a.inverse ? 1.0 / (double)a.L : 1.0;
  for (uint32_t e = threadIdx.x; e < a.L * nl; e += blockDim.x) {
    const uint32_t s = a.s_stride == 1 ? e % a.L : e / nl;
    const uint32_t l = a.s_stride == 1 ? e / a.L : e % nl;
    const double2 v = buf[l * a.L + s];
    a.data[base + l + (uint64_t)s * a.s_stride] = make_double2(v.x * sc, v.y * sc);
  }
}

// PSF (reading above): the z node k of column (i, j); false if it has none.
__device__ __forceinline__ bool psf_node(const LctDims& d, double slope4sq, uint32_t i, uint32_t j,
                                         int64_t& k) {
  const double x = -1.0 + 2.0 * i / (double)(d.n2 - 1);
  const double y = -1.0 + 2.0 * j / (double)(d.n2 - 1);
  const double dz = 2.0 / (double)(d.m2 - 1);
  const double target = slope4sq * (x * x + y * y);
  const double kf = rint((target + 1.0) / dz);
  if (!(kf >= 0.0 && kf < (double)d.m2)) return false;
  k = (int64_t)kf;
  return !(fabs(target - (-1.0 + (double)k * dz)) > 0.5 * dz + 1e-12);
}

// The PSF written circularly shifted into a zeroed volume.
__global__ void psf_kernel(double2* vol, LctDims d, double slope4sq) {
  const uint64_t col = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= (uint64_t)d.n2 * d.n2) return;
  const uint32_t i = (uint32_t)(col / d.n2), j = (uint32_t)(col % d.n2);
  int64_t k;
  if (!psf_node(d, slope4sq, i, j, k)) return;
  const uint32_t is = (i + d.N) % d.n2;  // origin at node (N, N, M)
  const uint32_t js = (j + d.N) % d.n2;
  const uint32_t ks = (uint32_t)((k + d.M) % d.m2);
  vol[((uint64_t)is * d.n2 + js) * d.m2 + ks] = make_double2(1.0, 0.0);
}

// R_z V into the zeroed volume: one voxel per depth-map pixel.
__global__ void volume_kernel(double2* vol, LctDims d, const int32_t* depth, const float* albedo) {
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= d.N * d.N) return;
  const uint32_t x = p / d.N, y = p % d.N;
  const int32_t z = depth[p];
  if (z < 0 || z >= (int32_t)d.M) return;
  const uint64_t j = (uint64_t)z + 1;
  const uint64_t r = (j * j + d.M - 1) / d.M - 1;
  const double a = albedo ? (double)albedo[p] : 0.5;
  vol[((uint64_t)x * d.n2 + y) * d.m2 + r] =
      make_double2(a / ((double)j * d.M * d.M), 0.0);
}

__global__ void multiply_kernel(double2* vol, const double2* psf_hat, uint64_t n) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x)
    vol[i] = cmul(vol[i], psf_hat[i]);
}

// Crop to N x N x M and resample time: tau[x][y][j - 1] = Re W[x][y][r(j)] M / j^4.
__global__ void time_kernel(const double2* vol, LctDims d, float* tau) {
  const uint64_t e = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (uint64_t)d.N * d.N * d.M) return;
  const uint64_t p = e / d.M;
  const uint64_t j = e % d.M + 1;
  const uint64_t x = p / d.N, y = p % d.N;
  const uint64_t r = (j * j + d.M - 1) / d.M - 1;
  const double jd = (double)j;
  tau[e] = (float)(vol[(x * d.n2 + y) * d.m2 + r].x * ((double)d.M / (jd * jd * jd * jd)));
}

// ---------------------------------------------------------------------------
// Direct form: tau[x][y][j - 1] = M / j^4 * sum of v(x', y') over the pixels
// with row(x', y') + k(x - x', y - y') = ceil(j^2 / M) - 1.
// One warp = a patch of 32 columns (x, y) (lane = column) times one window of
// time bins, whose FP64 samples it keeps in shared memory as [row][32]. Each
// lane adds to its own column only, so the additions are plain loads and
// stores without bank conflicts (red.shared.add.f64 is a compare-and-swap loop
// here, 45 cycles a warp and SM against 19 of the FP64 pipe). A warp is a CTA
// of its own, so the hardware balances windows of unequal load. Pixels come
// in 4 x 4 blocks with the range of their rows; a block that cannot reach the
// window from the patch is ruled out by one lane.
// Bound: the FP64 pipe's N^4 additions (1.68 lanes a cycle and SM: 0.53 ms at
// N = 128), taken about 1.3 times because a pixel's additions from one patch
// can straddle two windows, and the warps in flight (shared memory holds 12
// to 24). N = 128, M = 1024: 1.2 to 1.4 ms over several runs against 65.7 ms of the
// FFT form; N = 64: 0.29 against 15.4; N = 16: 0.04 against 0.92. Patches of 32 x 1
// columns and 1 x 32 segments of pixels took 1.7 ms. Sums as two FP32 words would
// take 0.73 ms at the same measured error, but carry 48 bits instead of 53.
// On a rough map (silhouettes, noise) a block spans many windows, and visiting
// all of its pixels in each costs 0.47 ms a window at N = 128, where one window's
// additions cost 1.3. Blocks of more than 2.5 windows' rows have their pixels
// tested one a lane first (0.05 ms a window, but 2.2 ms for additions that come
// four at a time): uniformly random depths, N = 128, M = 1024: 3.0 ms against 8.3
// with whole blocks; N = 512, M = 512: 477 against 1037 (FFTs 579); below 2.5 windows
// whole blocks are faster (N = 128, M = 128: 1.65 against 2.29).
// ---------------------------------------------------------------------------
constexpr int kDirSide = 4;      // side of a block of pixels
constexpr int kDirBins = 8;      // windows start at multiples of 8 bins (32-byte stores)
constexpr int kNoRow = 1 << 28;  // pixel without a surface
constexpr int kNoNode = 0x7fff;  // PSF column without a node

// Rows of a window. More rows make fewer straddled windows, fewer rows more
// and smaller warps: 64 against 32 rows take 1.16 / 1.42 ms at N = 128, 0.276 /
// 0.276 at N = 64, 0.105 / 0.094 at N = 32 and 0.070 / 0.045 at N = 16 (M = 1024).
int dir_rows(uint32_t N) { return N > 64 ? 64 : 32; }

struct __align__(16) Voxel {
  double v;
  int row, pad;
};

// Bins [j0, j1) (0-based) of a window and the first squared-time row they read.
struct DirWindow {
  int j0, j1, row0, rows;
};

struct DirArgs {
  const Voxel* vox;        // [N * N]
  const int2* seg;         // [n_seg] range of the rows of a block of pixels
  const int16_t* node;     // [2N][2N] time offset of the PSF node, kNoNode: none
  const double* weight;    // [M] M / j^4
  const DirWindow* win;
  float* tau;
  uint32_t N, M, n_seg, per_row;  // blocks of pixels; per_row along y
  int wide;                // rows beyond which a block's pixels are tested one by one
  uint32_t py, px, n_py;   // patch of py columns along y and px along x; patches along y
};

// Squared-depth sample of 0-based bin z: ceil((z + 1)^2 / M) - 1.
__host__ __device__ inline int sample_row(int64_t z, int64_t M) {
  return (int)(((z + 1) * (z + 1) + M - 1) / M - 1);
}

// R_z V as one (value, row) a pixel, in blocks of side * side pixels, and the
// row range of each block.
__global__ void __launch_bounds__(256) voxel_kernel(uint32_t N, uint32_t M, uint32_t side,
                                                    const int32_t* __restrict__ depth,
                                                    const float* __restrict__ albedo, Voxel* vox,
                                                    int2* seg) {
  const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
  int lo = kNoRow, hi = -1;
  if (k < N * N) {
    const uint32_t b = k / (side * side), i = k % (side * side), per_row = N / side;
    const uint32_t p = (b / per_row * side + i / side) * N + b % per_row * side + i % side;
    const int32_t z = depth[p];
    Voxel q{};
    q.row = kNoRow;
    if (z >= 0 && z < (int32_t)M) {
      const double a = albedo ? (double)albedo[p] : 0.5;
      q.v = a / ((double)(z + 1) * M * M);
      q.row = lo = hi = sample_row(z, M);
    }
    vox[k] = q;
  }
  for (uint32_t o = side * side >> 1; o > 0; o >>= 1) {
    lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (k < N * N && k % (side * side) == 0) seg[k / (side * side)] = make_int2(lo, hi);
}

// Time offset of the PSF node of each lateral offset (dx, dy) in [-N, N)^2.
__global__ void node_kernel(int16_t* node, LctDims d, double slope4sq) {
  const uint32_t col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= d.n2 * d.n2) return;
  int64_t k;
  node[col] = psf_node(d, slope4sq, col / d.n2, col % d.n2, k) ? (int16_t)(k - d.M)
                                                                 : (int16_t)kNoNode;
}

// The offsets of [a, b] nearest to and farthest from the PSF's centre (which
// lies between -1 and 0).
__device__ __forceinline__ int near_offset(int a, int b) { return a > 0 ? a : b < -1 ? b : 0; }
__device__ __forceinline__ int far_offset(int a, int b) { return -a - 1 > b ? a : b; }

template <int SIDE>
__global__ void __launch_bounds__(32) direct_kernel(const DirArgs a) {
  extern __shared__ double hist[];  // [rows of a window][32]
  const int lane = threadIdx.x;
  const DirWindow w = a.win[blockIdx.y];
  const int N = (int)a.N, n2 = 2 * N;
  const int x0 = (int)(blockIdx.x / a.n_py * a.px), y0 = (int)(blockIdx.x % a.n_py * a.py);
  const int x1 = min(x0 + (int)a.px, N) - 1, y1 = y0 + (int)a.py - 1;
  const int xl = x0 + lane / (int)a.py, y = y0 + lane % (int)a.py;
  const int x = min(xl, x1);  // lanes past the map repeat its last row and store nothing
  for (int i = 0; i < w.rows; ++i) hist[i * 32 + lane] = 0.0;
  const int16_t* at = a.node + (x + N) * n2 + y + N;
  double* h = hist + lane;
  // the pixels [xa, xa + side) x [ya, ya + side) with rows [lo, hi]: can they reach
  // the window from the patch? The node's offset grows with the distance from the
  // centre; one row of slack on each side against its rounding.
  auto reaches = [&](int xa, int ya, int side, int lo, int hi) {
    const int dx0 = x0 - (xa + side - 1), dx1 = x1 - xa, dy0 = y0 - (ya + side - 1), dy1 = y1 - ya;
    const int kn = a.node[(near_offset(dx0, dx1) + N) * n2 + near_offset(dy0, dy1) + N];
    const int kf = a.node[(far_offset(dx0, dx1) + N) * n2 + far_offset(dy0, dy1) + N];
    return kn != kNoNode && lo + kn - 1 < w.row0 + w.rows && hi + kf + 1 >= w.row0;
  };
  auto add = [&](const double2& q, int t) {
    // no node: at least 0x7fff - 4096 rows beyond any window
    const int r = __double2loint(q.y) + t - w.row0;
    if ((unsigned)r < (unsigned)w.rows) h[r * 32] += q.x;
  };
  for (uint32_t s0 = 0; s0 < a.n_seg; s0 += 32) {
    const uint32_t s = s0 + lane;
    bool live = false, wide = false;
    if (s < a.n_seg) {
      const int2 r = a.seg[s];
      live = r.x <= r.y && reaches((int)(s / a.per_row) * SIDE, (int)(s % a.per_row) * SIDE, SIDE,
                                   r.x, r.y);
      wide = SIDE == kDirSide && r.y - r.x > a.wide;
    }
    for (uint32_t m = __ballot_sync(0xffffffffu, live && !wide); m; m &= m - 1) {
      const uint32_t sl = s0 + __ffs(m) - 1;
      const int xs = (int)(sl / a.per_row) * SIDE, ys = (int)(sl % a.per_row) * SIDE;
      const double2* vp = reinterpret_cast<const double2*>(a.vox + sl * (SIDE * SIDE));
      const int16_t* kp = at - (xs * n2 + ys);
      double2 q[SIDE * SIDE];
      int t[SIDE * SIDE];
#pragma unroll
      for (int i = 0; i < SIDE * SIDE; ++i) {
        q[i] = __ldg(vp + i);
        t[i] = (int)__ldg(kp - (i / SIDE) * n2 - i % SIDE);
      }
#pragma unroll
      for (int i = 0; i < SIDE * SIDE; ++i) add(q[i], t[i]);
    }
    // two wide blocks at a time: each lane tests one pixel, and those that reach
    // the window are taken four at a time
    for (uint32_t m = __ballot_sync(0xffffffffu, live && wide); m;) {
      const uint32_t sa = s0 + __ffs(m) - 1;
      m &= m - 1;
      const uint32_t sb = m ? s0 + __ffs(m) - 1 : sa;
      const bool two = m != 0u;
      m &= m - 1;
      const uint32_t sl = lane < 16 ? sa : sb;
      const int xp = (int)(sl / a.per_row) * SIDE + lane % 16 / SIDE;
      const int yp = (int)(sl % a.per_row) * SIDE + lane % 16 % SIDE;
      const int row = a.vox[sl * 16 + lane % 16].row;
      const bool pix = (lane < 16 || two) && row != kNoRow && reaches(xp, yp, 1, row, row);
      for (uint32_t mp = __ballot_sync(0xffffffffu, pix); mp;) {
        double2 q[4];
        int t[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          // (past the last one: a pixel without a surface)
          q[i] = make_double2(0.0, __hiloint2double(0, kNoRow));
          t[i] = 0;
          if (mp) {
            const uint32_t j = __ffs(mp) - 1, sj = j < 16 ? sa : sb, p = j % 16;
            const int xj = (int)(sj / a.per_row) * SIDE + (int)p / SIDE;
            const int yj = (int)(sj % a.per_row) * SIDE + (int)p % SIDE;
            q[i] = __ldg(reinterpret_cast<const double2*>(a.vox + sj * 16 + p));
            t[i] = (int)__ldg(at - (xj * n2 + yj));
          }
          mp &= mp - 1;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) add(q[i], t[i]);
      }
    }
  }
  // each lane writes 8 bins (32 bytes) of its own column at a time
  if (xl > x1) return;
  float* out = a.tau + ((size_t)x * N + y) * a.M;
  const bool vec = ((reinterpret_cast<uintptr_t>(a.tau) & 15u) == 0) && (a.M % kDirBins) == 0;
  for (int j = w.j0; j < w.j1; j += kDirBins) {
    float v[kDirBins];
#pragma unroll
    for (int e = 0; e < kDirBins; ++e) {
      const int je = min(j + e, w.j1 - 1);
      const int t = (sample_row(je, a.M) - w.row0) * 32;
      v[e] = (float)(h[t] * a.weight[je]);
    }
    if (vec) {
      reinterpret_cast<float4*>(out + j)[0] = make_float4(v[0], v[1], v[2], v[3]);
      reinterpret_cast<float4*>(out + j)[1] = make_float4(v[4], v[5], v[6], v[7]);
    } else {
      for (int e = 0; e < kDirBins && j + e < w.j1; ++e) out[j + e] = v[e];
    }
  }
}

// Windows of at most max_rows squared-time rows, by bins.
std::vector<DirWindow> dir_windows(int M, int max_rows) {
  std::vector<DirWindow> out;
  for (int j = 0; j < M;) {
    DirWindow w{j, j, sample_row(j, M), 0};
    while (w.j1 < M) {
      const int e = std::min(w.j1 + kDirBins, M);
      if (sample_row(e - 1, M) - w.row0 + 1 > max_rows) break;
      w.j1 = e;
      w.rows = sample_row(e - 1, M) - w.row0 + 1;
    }
    out.push_back(w);
    j = w.j1;
  }
  return out;
}

// The direct form's N^4 additions (4.3 ps each on a smooth map) against the FFT
// form's passes over 8 N^2 M padded samples (about 490 ps each): direct below N^2 of
// about 900 M. Measured on both sides of the line, smooth maps: N = 128, M = 32: 1.34
// against 2.04 ms, M = 16: 1.2 against 1.39; N = 256, M = 128: 14.6 against 32, M = 64:
// 18 against 16. Random depths: N = 128, M = 32: 1.34 against 2.04 ms; N = 256, M = 128:
// 25 against 32; N = 512, M = 512: 477 against 579.
bool direct_form(uint32_t N, uint32_t M) { return (uint64_t)N * N <= 900ull * M; }

bool pow2(uint32_t v) { return v >= 2 && (v & (v - 1)) == 0; }
uint32_t ilog2(uint32_t v) {
  uint32_t r = 0;
  while ((1u << r) < v) ++r;
  return r;
}

}  // namespace
}  // namespace nlos

struct nlos_lct {
  nlos::LctDims d;
  double2* work = nullptr;
  double2* psf_hat = nullptr;
  double2* tw = nullptr;
  uint32_t lmax = 0;
  int device = 0;
  // direct form
  bool direct = false;
  nlos::DirArgs dir{};
  nlos::Voxel* vox = nullptr;
  int2* seg = nullptr;
  int16_t* node = nullptr;
  double* weight = nullptr;
  nlos::DirWindow* win = nullptr;
  uint32_t n_win = 0;
};

namespace nlos {
namespace {

cudaError_t fft3(const nlos_lct& p, double2* vol, int inverse, cudaStream_t st) {
  const LctDims& d = p.d;
  struct Axis {
    uint32_t L;
    uint64_t s_stride, outer_stride, n_inner, n_outer;
  };
  const uint64_t m2 = d.m2, n2 = d.n2;
  const Axis axes[3] = {
      {d.m2, 1, m2, 1, n2 * n2},             // time: contiguous lines
      {d.n2, m2, n2 * m2, m2, n2},           // y: lines (x, t)
      {d.n2, n2 * m2, m2, m2, n2},           // x: lines (y, t)
  };
  for (const Axis& ax : axes) {
    FftArgs a;
    a.data = vol;
    a.tw = p.tw;
    a.L = ax.L;
    a.log2L = ilog2(ax.L);
    a.tw_step = p.lmax / ax.L;
    a.s_stride = ax.s_stride;
    a.outer_stride = ax.outer_stride;
    a.n_inner = ax.n_inner;
    a.inverse = inverse;
    const size_t line_bytes = sizeof(double2) * ax.L;
    uint32_t T = ax.s_stride == 1 ? 1u : (uint32_t)std::max<size_t>(1, kFftSmem / line_bytes);
    if (T > 16) T = 16;
    if (ax.s_stride == 1) {
      // contiguous lines: each line is its own "outer" index of one line
      a.n_inner = 1;
      a.outer_stride = ax.L;
    }
    a.T = T;
    const uint64_t groups = (a.n_inner + T - 1) / T;
    const uint64_t blocks = (ax.s_stride == 1 ? ax.n_outer : ax.n_outer) * groups;
    const size_t smem = line_bytes * T;
    cudaError_t e = cudaFuncSetAttribute(fft_lines_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (blocks > 0x7fffffffull) return cudaErrorInvalidValue;
    fft_lines_kernel<<<(unsigned)blocks, kFftThreads, smem, st>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

void free_plan(nlos_lct* p) {
  for (void* q : {(void*)p->work, (void*)p->psf_hat, (void*)p->tw, (void*)p->vox, (void*)p->seg,
                  (void*)p->node, (void*)p->weight, (void*)p->win})
    if (q) cudaFree(q);
  delete p;
}

// The direct form's plan: the PSF's nodes, the time weights and the windows.
cudaError_t create_direct(nlos_lct* p, double slope4sq, cudaStream_t st) {
  const LctDims& d = p->d;
  const uint32_t n_pix = d.N * d.N;
  DirArgs& a = p->dir;
  a.N = d.N;
  a.M = d.M;
  const uint32_t side = std::min(d.N, (uint32_t)kDirSide);
  a.n_seg = n_pix / (side * side);
  a.per_row = d.N / side;
  a.py = std::min(d.N, 8u);
  a.px = 32u / a.py;
  a.n_py = d.N / a.py;
  a.wide = dir_rows(d.N) * 5 / 2;
  const std::vector<DirWindow> win = dir_windows((int)d.M, dir_rows(d.N));
  std::vector<double> weight(d.M);
  for (uint32_t z = 0; z < d.M; ++z) {
    const double j = (double)(z + 1);
    weight[z] = (double)d.M / (j * j * j * j);
  }
  p->n_win = (uint32_t)win.size();
  cudaError_t e;
  if ((e = cudaMalloc(&p->vox, sizeof(Voxel) * n_pix)) != cudaSuccess ||
      (e = cudaMalloc(&p->seg, sizeof(int2) * a.n_seg)) != cudaSuccess ||
      (e = cudaMalloc(&p->node, sizeof(int16_t) * d.n2 * d.n2)) != cudaSuccess ||
      (e = cudaMalloc(&p->weight, sizeof(double) * d.M)) != cudaSuccess ||
      (e = cudaMalloc(&p->win, sizeof(DirWindow) * win.size())) != cudaSuccess ||
      (e = cudaMemcpyAsync(p->weight, weight.data(), sizeof(double) * d.M, cudaMemcpyHostToDevice,
                           st)) != cudaSuccess ||
      (e = cudaMemcpyAsync(p->win, win.data(), sizeof(DirWindow) * win.size(),
                           cudaMemcpyHostToDevice, st)) != cudaSuccess)
    return e;
  a.vox = p->vox;
  a.seg = p->seg;
  a.node = p->node;
  a.weight = p->weight;
  a.win = p->win;
  node_kernel<<<(d.n2 * d.n2 + 255) / 256, 256, 0, st>>>(p->node, d, slope4sq);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return cudaStreamSynchronize(st);
}

}  // namespace
}  // namespace nlos

using namespace nlos;

extern "C" {

nlos_status nlos_lct_create(uint32_t n, uint32_t m, double wall_half_m, double bin_width_s,
                            void* cuda_stream, nlos_lct** out) {
  clear_error();
  if (!out) return set_error(NLOS_EINVAL, "out is NULL");
  *out = nullptr;
  if (!pow2(n) || !pow2(m) || n > 1024 || m > 4096)
    return set_error(NLOS_EINVAL, "n and m must be powers of two, 2 <= n <= 1024, 2 <= m <= 4096");
  if (!(std::isfinite(wall_half_m) && wall_half_m > 0 && std::isfinite(bin_width_s) && bin_width_s > 0))
    return set_error(NLOS_EINVAL, "wall_half_m and bin_width_s must be finite and > 0");
  nlos_lct* p = new (std::nothrow) nlos_lct();
  if (!p) return set_error(NLOS_ENOMEM, "host allocation failed");
  p->d = LctDims{n, m, 2 * n, 2 * m};
  p->lmax = std::max(2 * n, 2 * m);
  const uint64_t nvol = (uint64_t)p->d.n2 * p->d.n2 * p->d.m2;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  auto fail = [&](cudaError_t e, const char* what) {
    free_plan(p);
    return cuda_error(e, what);
  };
  cudaError_t e = cudaGetDevice(&p->device);
  if (e != cudaSuccess) return fail(e, "cudaGetDevice");
  const double slope = wall_half_m / ((double)m * kLightSpeed * bin_width_s);
  p->direct = direct_form(n, m);
  if (p->direct) {
    if ((e = create_direct(p, 16.0 * slope * slope, st)) != cudaSuccess)
      return fail(e, "depth-map model plan");
    *out = p;
    return NLOS_OK;
  }
  if ((e = cudaMalloc(&p->work, sizeof(double2) * nvol)) != cudaSuccess ||
      (e = cudaMalloc(&p->psf_hat, sizeof(double2) * nvol)) != cudaSuccess ||
      (e = cudaMalloc(&p->tw, sizeof(double2) * (p->lmax / 2))) != cudaSuccess)
    return fail(e, "cudaMalloc");
  std::vector<double2> tw(p->lmax / 2);
  const double pi = 3.14159265358979323846;
  for (uint32_t k = 0; k < p->lmax / 2; ++k) {
    const double ang = -2.0 * pi * (double)k / (double)p->lmax;
    tw[k] = make_double2(std::cos(ang), std::sin(ang));
  }
  if ((e = cudaMemcpyAsync(p->tw, tw.data(), sizeof(double2) * tw.size(), cudaMemcpyHostToDevice,
                           st)) != cudaSuccess ||
      (e = cudaMemsetAsync(p->psf_hat, 0, sizeof(double2) * nvol, st)) != cudaSuccess)
    return fail(e, "cudaMemcpyAsync");
  const uint64_t cols = (uint64_t)p->d.n2 * p->d.n2;
  psf_kernel<<<(unsigned)((cols + 255) / 256), 256, 0, st>>>(p->psf_hat, p->d, 16.0 * slope * slope);
  if ((e = cudaGetLastError()) != cudaSuccess) return fail(e, "psf_kernel");
  if ((e = fft3(*p, p->psf_hat, 0, st)) != cudaSuccess) return fail(e, "fft");
  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return fail(e, "cudaStreamSynchronize");
  *out = p;
  return NLOS_OK;
}

nlos_status nlos_lct_forward(nlos_lct* plan, const int32_t* depth_dev, const float* albedo_dev,
                             float* tau_dev, void* cuda_stream) {
  clear_error();
  if (!plan || !depth_dev || !tau_dev)
    return set_error(NLOS_EINVAL, "plan, depth_dev and tau_dev must not be NULL");
  const LctDims& d = plan->d;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  if (plan->direct) {
    DirArgs a = plan->dir;
    a.tau = tau_dev;
    const uint32_t n_pix = d.N * d.N;
    voxel_kernel<<<(n_pix + 255) / 256, 256, 0, st>>>(
        d.N, d.M, std::min(d.N, (uint32_t)kDirSide), depth_dev, albedo_dev, plan->vox, plan->seg);
    NLOS_CUDA_TRY(cudaGetLastError());
    const size_t smem = sizeof(double) * 32 * dir_rows(d.N);
    const dim3 grid(a.n_py * ((d.N + a.px - 1) / a.px), plan->n_win);
    if (d.N >= kDirSide) direct_kernel<kDirSide><<<grid, 32, smem, st>>>(a);
    else direct_kernel<2><<<grid, 32, smem, st>>>(a);  // a 2 x 2 map
    NLOS_CUDA_TRY(cudaGetLastError());
    return NLOS_OK;
  }
  const uint64_t nvol = (uint64_t)d.n2 * d.n2 * d.m2;
  NLOS_CUDA_TRY(cudaMemsetAsync(plan->work, 0, sizeof(double2) * nvol, st));
  volume_kernel<<<(d.N * d.N + 255) / 256, 256, 0, st>>>(plan->work, d, depth_dev, albedo_dev);
  NLOS_CUDA_TRY(cudaGetLastError());
  NLOS_CUDA_TRY(fft3(*plan, plan->work, 0, st));
  multiply_kernel<<<2048, 256, 0, st>>>(plan->work, plan->psf_hat, nvol);
  NLOS_CUDA_TRY(cudaGetLastError());
  NLOS_CUDA_TRY(fft3(*plan, plan->work, 1, st));
  const uint64_t n_out = (uint64_t)d.N * d.N * d.M;
  time_kernel<<<(unsigned)((n_out + 255) / 256), 256, 0, st>>>(plan->work, d, tau_dev);
  NLOS_CUDA_TRY(cudaGetLastError());
  return NLOS_OK;
}

nlos_status nlos_lct_destroy(nlos_lct* plan) {
  clear_error();
  if (!plan) return set_error(NLOS_EINVAL, "plan is NULL");
  cudaDeviceSynchronize();
  free_plan(plan);
  return NLOS_OK;
}

}  // extern "C"

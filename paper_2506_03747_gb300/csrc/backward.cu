// Adjoint of the Gaussian-splat forward (differentiable form of the binned
// transient of arXiv 2506.03747): gradients of a loss L(tau) with respect to
// per-point albedo rho_p and per-point displacement delta_p along the normal.
//
// For a pair (s, p) with x_b = b + 1/2 - u_sp and phi the splat kernel,
//   G0 = sum_b g[s][b] phi(x_b),   G1 = sum_b g[s][b] (x_b / sigma^2) phi(x_b),
//   dL/d rho_p   = sum_s (dw/d rho) G0,
//   dL/d delta_p = sum_s (dw/d delta) G0 + w (du/d delta) G1,
// with, for x -> x + delta n: dr/d delta = -cos, d cos/d delta = -(1 - cos^2)/r,
// d(z/r)/d delta = (n_z + (z/r) cos)/r and du/d delta = -(cos_l + cos_d)/(c dt).
//
// Two forms of the sums G0, G1 (adjoint_moments chooses):
//  * taps (any sigma): one CTA per (32-scan-point tile, point block); the
//    tile's g rows are staged into shared memory as [bin][32] (lane = scan
//    point, conflict-free gathers) and each lane runs the |x_b| < 6 sigma taps
//    of its own pair;
//  * moments (sigma up to 9.8 bins): with the rows, c and table D_n of the moment
//    forward (q rows a bin), phi(x_b) = sum_n c^n D_n[i] turns the sums into
//    polynomials in c,
//      G0 = sum_n c^n H_n[r],   H_n[r] = sum_b g[b] D_n[r - q b + q J],
//      G1 = -dG0/dx = -q sum_n n c^(n-1) H_n[r]   (x phi(x) / sigma^2 = -phi'(x)),
//    so a first kernel correlates every transient of g with the kMomTerms = 8
//    tables (32 bytes a row) and the pair kernel needs one 32-byte gather and
//    two Horner evaluations per pair instead of about 12 sigma taps.
// Taps form: points are broadcast from shared memory, and a warp sum over the
// 32 scan points of a tile gives the tile's contribution to each point, added
// to the outputs with one global atomic. Moments form: one thread per point,
// looping over a block of scan points broadcast from shared memory; the sums
// over s stay in the thread's registers (no warp sum), the laser leg of a
// non-confocal scan is computed once per point, and each block of scan points
// adds its contribution to each point with one global atomic.
#include "common.cuh"
#include "device_util.cuh"
#include "forward_core.cuh"

#include <algorithm>
#include <cmath>

namespace nlos {

namespace {

constexpr int kBwdTile = 32;
constexpr int kBwdPoints = 256;  // points per CTA
constexpr int kBwdMomThreads = 256;  // moments form: points per CTA (one per thread)
constexpr int kBwdMomScan = 128;     // moments form: scan points per CTA at most
constexpr int kAdjTabThreads = 128;
constexpr int kAdjTabBins = 4;       // bins of a thread
constexpr size_t kAdjTabBytes = 64u << 20;  // moment tables held at one time
static_assert(kMomTerms == 8, "a row of the adjoint table is four float2");

// The table of one transient: rows in groups of 16, of each group the terms
// (0, 1) of its rows, then (2, 3), (4, 5) and (6, 7), so that the 32 rows that a
// warp of neighbouring points gathers lie in two or three cache lines for each
// of the four loads (rows as two float4 took 13 L1 wavefronts a load).
constexpr uint32_t kTabGroup = 16;
constexpr uint32_t kTabPitch = kTabGroup * kMomTerms / 2;  // float2 a group
__host__ __device__ inline uint32_t tab_groups(uint32_t rows) {
  return (rows + kTabGroup - 1) / kTabGroup;
}
__device__ __forceinline__ uint32_t tab_at(uint32_t row) {
  return row + row / kTabGroup * (kTabPitch - kTabGroup);
}

struct BwdArgs {
  const float* raw;        // [P][8]
  const uint32_t* perm;    // [P] spatial order of the points
  const ScanPoint* scan;   // spots and offsets
  const float* g;          // [S][B]
  float* ga;               // [P] or null
  float* gd;               // [P] or null
  uint64_t P, S;
  uint32_t B;
  int scan_mode, cos_mode;
  float lx, ly;            // laser spot (non-confocal)
  float inv_cdt;           // 1 / (c dt)
  float inv2s2, inv_s2, norm, reach, qstep;
};

#ifndef NLOS_BWD_RSQRT
#define NLOS_BWD_RSQRT 1  // legs from a reciprocal square root estimate and one Newton step
#endif

// 1 / sqrt(x) for x > 0: the hardware estimate and one Newton step (about an
// ulp; the gradients are held to 1e-3 of their maximum).
__device__ __forceinline__ float rsqrt_newton(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y * fmaf(-0.5f * x, y * y, 1.5f);
}

// A leg's length and its reciprocal from its squared length.
__device__ __forceinline__ void leg_length(float r2, float& r, float& ri) {
#if NLOS_BWD_RSQRT
  ri = rsqrt_newton(r2);
  r = r2 * ri;
#else
  r = sqrtf(r2);
  ri = 1.0f / r;
#endif
}

// Squared length of a leg. A last-bit change of r moves u by up to 3e-5 bins,
// and with it the gradient of a rough g by 1e-5, so the widths that the taps
// form used to serve (below 2.5 bins) keep its roundings: this order of
// summation, and a rounded sum of the legs where the compiler would fuse it.
template <bool TAPS>
__device__ __forceinline__ float leg_r2(float vx, float vy, float vz) {
  return TAPS ? __fadd_rn(fmaf(vx, vx, __fmul_rn(vy, vy)), __fmul_rn(vz, vz))
              : fmaf(vx, vx, fmaf(vy, vy, vz * vz));
}

// Leg factor F = cosf * wallf / r^2 and its delta-derivative (FP32); ri = 1 / r.
__device__ __forceinline__ void leg(int cos_mode, float ndotv, float vz, float nz, float ri,
                                    float& F, float& dF, float& c) {
  c = -ndotv * ri;
  const float dc = -(1.0f - c * c) * ri;
  float fc = 1.0f, dfc = 0.0f;
  if (cos_mode >= NLOS_COS_OBJECT) {
    if (c > 0.0f) {
      fc = c;
      dfc = dc;
    } else {
      fc = 0.0f;
      dfc = 0.0f;
    }
  }
  float fw = 1.0f, dfw = 0.0f;
  if (cos_mode == NLOS_COS_OBJECT_WALL) {
    fw = vz * ri;
    dfw = (nz + fw * c) * ri;
  }
  const float ri2 = ri * ri;
  F = fc * fw * ri2;
  // d(r^-2)/d delta = -2 r^-3 dr/d delta = 2 c r^-3
  dF = (dfc * fw + fc * dfw) * ri2 + fc * fw * 2.0f * c * ri2 * ri;
}

// H_n of the rows of transients [s0, s0 + gridDim.y), row (k + J) q + ph for bins
// k in [-J, B + J) and phases ph of their rows.
struct AdjTabArgs {
  const float* g;  // [S][B]
  float2* T;
  uint64_t s0;
  uint32_t B, bins, per_cta;  // bins B + 2J, and those of a CTA
};

// A thread takes kAdjTabBins bins of one phase, so that the eight taps of a step
// (the same for the CTA) serve 32 FMAs. Bound: FMA; 4096 transients of 512
// bins, 43 taps: 54 us, against 80 us with one row a thread and twelve sums a row.
__global__ void __launch_bounds__(kAdjTabThreads)
    adj_table_kernel(const AdjTabArgs a, const __grid_constant__ MomTab mt) {
  __shared__ float gs[kAdjTabThreads * kAdjTabBins + 2 * kMomMaxJ];
  const int J = mt.J, q = mt.q, nt = (int)blockDim.x;
  const int k0 = (int)(blockIdx.x * a.per_cta) - J;  // first bin of the CTA
  const float* row = a.g + (a.s0 + blockIdx.y) * a.B;
  // gs[i] = g[k0 - J + i] (zero outside the transient)
  for (int i = threadIdx.x; i < nt * kAdjTabBins + 2 * J; i += nt) {
    const int b = k0 - J + i;
    gs[i] = (b >= 0 && b < (int)a.B) ? row[b] : 0.0f;
  }
  __syncthreads();
  float2* out = a.T + (size_t)blockIdx.y * tab_groups(a.bins * q) * kTabPitch;
  for (int ph = 0; ph < q; ++ph) {
    float h[kAdjTabBins][kMomTerms];
#pragma unroll
    for (int e = 0; e < kAdjTabBins; ++e)
#pragma unroll
      for (int n = 0; n < kMomTerms; ++n) h[e][n] = 0.0f;
    // row ph of bin k meets bin k + J - m with tap ph + q m
    const float* gp = gs + threadIdx.x + 2 * J;
    for (int m = 0; m <= 2 * J; ++m, --gp) {
      const float* d = mt.d[ph + q * m];
#pragma unroll
      for (int e = 0; e < kAdjTabBins; ++e) {
        const float gv = gp[e * nt];
#pragma unroll
        for (int n = 0; n < kMomTerms; ++n) h[e][n] = fmaf(gv, d[n], h[e][n]);
      }
    }
#pragma unroll
    for (int e = 0; e < kAdjTabBins; ++e) {
      const uint32_t local = threadIdx.x + e * nt, k = blockIdx.x * a.per_cta + local;
      if (local >= a.per_cta || k >= a.bins) continue;
      float2* o = out + tab_at(k * q + ph);
#pragma unroll
      for (int n = 0; n < kMomTerms; n += 2) o[n / 2 * kTabGroup] = make_float2(h[e][n], h[e][n + 1]);
    }
  }
}

// Taps form: one CTA per (32-scan-point tile, block of kBwdPoints points).
__global__ void __launch_bounds__(256) bwd_kernel(const BwdArgs a) {
  extern __shared__ float sm[];
  float* gt = sm;                              // [B][32]
  float* pts = sm + (size_t)a.B * kBwdTile;    // [kBwdPoints][8]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const uint64_t n_pblk = (a.P + kBwdPoints - 1) / kBwdPoints;
  const uint64_t tile = blockIdx.x / n_pblk;
  const uint64_t p0 = (blockIdx.x % n_pblk) * kBwdPoints;
  const int np = (int)min((uint64_t)kBwdPoints, a.P - p0);

  for (uint32_t i = tid; i < a.B * kBwdTile; i += blockDim.x) {
    const uint32_t s_loc = i & 31, b = i >> 5;
    const uint64_t s = tile * kBwdTile + s_loc;
    gt[i] = s < a.S ? a.g[s * a.B + b] : 0.0f;
  }
  for (int i = tid; i < np * 8; i += blockDim.x) pts[i] = a.raw[p0 * 8 + i];
  __syncthreads();

  const uint64_t s = tile * kBwdTile + lane;
  const bool valid = s < a.S;
  ScanPoint sp = valid ? a.scan[s] : ScanPoint{0.f, 0.f, -1e30f, 0u};
  const float dx_s = sp.sx, dy_s = sp.sy;
  const float lx = a.scan_mode == NLOS_CONFOCAL ? sp.sx : a.lx;
  const float ly = a.scan_mode == NLOS_CONFOCAL ? sp.sy : a.ly;

  for (int i = warp; i < np; i += nwarps) {
    const float* q = pts + 8 * i;
    const float x = q[0], y = q[1], z = q[2], nx = q[3], ny = q[4], nz = q[5], rho = q[6],
                area = q[7];
    // laser leg l -> x and detector leg d -> x
    const float vlx = x - lx, vly = y - ly, vlz = z;
    float rl, ril;
    leg_length(leg_r2<true>(vlx, vly, vlz), rl, ril);
    float Fl, dFl, cl, Fd, dFd, cd, rd;
    leg(a.cos_mode, nx * vlx + ny * vly + nz * vlz, vlz, nz, ril, Fl, dFl, cl);
    if (a.scan_mode == NLOS_CONFOCAL) {
      // the laser spot is the detector spot: the second leg is the first
      rd = rl;
      Fd = Fl;
      dFd = dFl;
      cd = cl;
    } else {
      const float vdx = x - dx_s, vdy = y - dy_s, vdz = z;
      float rid;
      leg_length(leg_r2<true>(vdx, vdy, vdz), rd, rid);
      leg(a.cos_mode, nx * vdx + ny * vdy + nz * vdz, vdz, nz, rid, Fd, dFd, cd);
    }
    const float qw = rho * area;
    const float w = qw * Fl * Fd;
    const float dw_drho = area * Fl * Fd;
    const float dw_dd = qw * (dFl * Fd + Fl * dFd);
    // u relative to bin 0: legs and window start are in sp.off (both legs
    // below are recomputed here rather than taken from the packed form)
    const float u = (rl + rd) * a.inv_cdt + sp.off;
    const float du_dd = -(cl + cd) * a.inv_cdt;
    float G0 = 0.f, G1 = 0.f;
    if (valid && (w != 0.f || dw_dd != 0.f || dw_drho != 0.f)) {
      const int lo = max(0, (int)(floorf(u - 0.5f - a.reach) + 1.0f));
      const int hi = min((int)a.B - 1, (int)(ceilf(u - 0.5f + a.reach) - 1.0f));
      if (lo <= hi) {
        // tap recurrence restarted every 8 taps (its rounding error grows
        // with the square of the number of steps)
        float K = 0.f, r = 0.f;
        for (int b = lo; b <= hi; ++b) {
          const float xb = (float)b + 0.5f - u;
          if (((b - lo) & 7) == 0) {
            K = a.norm * expf(-xb * xb * a.inv2s2);
            r = expf(-(2.0f * xb + 1.0f) * a.inv2s2);
          }
          const float gv = gt[b * kBwdTile + lane];
          G0 = fmaf(gv, K, G0);
          G1 = fmaf(gv * xb, K, G1);
          K *= r;
          r *= a.qstep;
        }
        G1 *= a.inv_s2;
      }
    }
    float ca = dw_drho * G0;
    float cdl = dw_dd * G0 + w * du_dd * G1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      ca += __shfl_xor_sync(0xffffffffu, ca, o);
      cdl += __shfl_xor_sync(0xffffffffu, cdl, o);
    }
    if (lane == 0) {
      if (a.ga) atomicAdd(a.ga + p0 + i, ca);
      if (a.gd) atomicAdd(a.gd + p0 + i, cdl);
    }
  }
}

// Moments form: thread = one point, CTA = (block of `per` scan points, block of
// points) with the scan block the slower index, so the CTAs resident at one
// time read the tables of few transients; scan points [s0, s0 + ns) of the
// tables in T. Points are taken in the forward's spatial order, so that a
// warp's points mostly leave the window together (then only the leg's length
// and v are computed) and gather neighbouring rows. Bound: FP32 issue (81% of
// the slots) and the L1 wavefronts of the gathers (68%). 64 x 64 scan, 65,536
// points: 400 us, against 526 us with points in the caller's order, every pair
// evaluated in full and 48-byte rows; 32 x 32 scan, 16,384 points, non-confocal
// at sigma = 1.6: 43 us, against 398 us pair by pair in taps.
// TAPS_R2: squared legs summed as the taps form sums them (leg_r2).
template <int SCAN, int COS, bool TAPS_R2>
__global__ void __launch_bounds__(kBwdMomThreads)
    bwd_mom_kernel(const BwdArgs a, const float2* __restrict__ T, uint64_t s0, uint32_t ns_all,
                   uint32_t per, int J, int q, uint32_t rows, uint32_t n_pblk) {
  __shared__ ScanPoint ss[kBwdMomScan];
  const uint32_t sb = blockIdx.x / n_pblk * per;  // first scan point of the CTA, from s0
  const uint64_t k = (uint64_t)(blockIdx.x % n_pblk) * kBwdMomThreads + threadIdx.x;
  const int ns = (int)min(per, ns_all - sb);
  const float fq = (float)q;
  for (int i = threadIdx.x; i < ns; i += blockDim.x) {
    ss[i] = a.scan[s0 + sb + i];
    ss[i].off *= fq;  // exact, as v = q u below
  }
  __syncthreads();
  if (k >= a.P) return;
  const uint32_t p = a.perm[k];
  const float4* rp = reinterpret_cast<const float4*>(a.raw + (size_t)p * 8);
  const float4 q0 = rp[0], q1 = rp[1];
  const float x = q0.x, y = q0.y, z = q0.z, nx = q0.w, ny = q1.x, nz = q1.y, rho = q1.z,
              area = q1.w;
  const float nzz = nz * z;
  // the laser leg of a non-confocal scan depends on the point only
  float rl = 0.f, Fl = 0.f, dFl = 0.f, cl = 0.f;
  if (SCAN != NLOS_CONFOCAL) {
    const float vlx = x - a.lx, vly = y - a.ly;
    float ril;
    leg_length(leg_r2<TAPS_R2>(vlx, vly, z), rl, ril);
    leg(COS, fmaf(nx, vlx, fmaf(ny, vly, nzz)), z, nz, ril, Fl, dFl, cl);
  }
  const float v_lo = (float)(-J * q), v_hi = (float)((int)rows - J * q);
  const float kv = (SCAN == NLOS_CONFOCAL ? 2.0f : 1.0f) * a.inv_cdt * fq;
  const uint32_t pitch = tab_groups(rows) * kTabPitch;
  const int row0 = kMagicBits - J * q;
  // sums without the factors of the point alone: area for the albedo's,
  // albedo * area for the offset's
  float ca = 0.f, sum0 = 0.f, sum1 = 0.f;
  uint32_t at = sb * pitch;  // the tables of one launch hold at most 2^32 float2
  for (int i = 0; i < ns; ++i, at += pitch) {
    const ScanPoint sp = ss[i];
    // the detector leg d -> x (for a confocal scan also the laser leg)
    const float vdx = x - sp.sx, vdy = y - sp.sy;
    float rd, rid;
    leg_length(leg_r2<TAPS_R2>(vdx, vdy, z), rd, rid);
    const float path = SCAN == NLOS_CONFOCAL ? rd : TAPS_R2 ? __fadd_rn(rl, rd) : rl + rd;
    const float v = fmaf(path, kv, sp.off);
    if (!(v >= v_lo && v < v_hi)) continue;
    const float ndotv = fmaf(nx, vdx, fmaf(ny, vdy, nzz));
    if (COS != NLOS_COS_NONE && !(ndotv < 0.f)) continue;  // faces away: no weight, no gradient
    float F2, dF2, dc;  // Fl Fd, its derivative along the normal, and -(c dt) du/d delta
    if (COS == NLOS_COS_OBJECT) {
      // Fd = c / r^2 and dFd/d delta = (3 c^2 - 1) / r^3 with c = -n.v / r
      const float cd = -ndotv * rid, i2 = rid * rid, e = fmaf(3.0f * cd, cd, -1.0f) * rid;
      if (SCAN == NLOS_CONFOCAL) {
        const float ci4 = cd * (i2 * i2);
        F2 = ci4 * cd;
        dF2 = 2.0f * ci4 * e;
        dc = 2.0f * cd;
      } else {
        F2 = Fl * i2 * cd;
        dF2 = i2 * fmaf(dFl, cd, Fl * e);
        dc = cl + cd;
      }
    } else {
      float Fd, dFd, cd;
      leg(COS, ndotv, z, nz, rid, Fd, dFd, cd);
      if (SCAN == NLOS_CONFOCAL) {
        F2 = Fd * Fd;
        dF2 = 2.0f * Fd * dFd;
        dc = 2.0f * cd;
      } else {
        F2 = Fl * Fd;
        dF2 = dFl * Fd + Fl * dFd;
        dc = cl + cd;
      }
    }
    const float tv = __fadd_rd(v, kMagic);  // kMagic + floor(v)
    const float c = 0.5f - (v - (tv - kMagic));
    const float2* t = T + (at + tab_at((uint32_t)(__float_as_int(tv) - row0)));
    const float2 b0 = __ldg(t), b1 = __ldg(t + kTabGroup), b2 = __ldg(t + 2 * kTabGroup),
                 b3 = __ldg(t + 3 * kTabGroup);
    // G0 and its derivative in c by one Horner scheme
    float G0 = b3.y, D = b3.y;
    G0 = fmaf(G0, c, b3.x);
    D = fmaf(D, c, G0);
    G0 = fmaf(G0, c, b2.y);
    D = fmaf(D, c, G0);
    G0 = fmaf(G0, c, b2.x);
    D = fmaf(D, c, G0);
    G0 = fmaf(G0, c, b1.y);
    D = fmaf(D, c, G0);
    G0 = fmaf(G0, c, b1.x);
    D = fmaf(D, c, G0);
    G0 = fmaf(G0, c, b0.y);
    D = fmaf(D, c, G0);
    G0 = fmaf(G0, c, b0.x);
    // du/d delta * G1 = (dc / (c dt)) * q D
    ca = fmaf(F2, G0, ca);
    sum0 = fmaf(dF2, G0, sum0);
    sum1 = fmaf(F2 * dc, D, sum1);
  }
  if (a.ga) atomicAdd(a.ga + p, ca * area);
  if (a.gd) atomicAdd(a.gd + p, fmaf(sum1, fq * a.inv_cdt, sum0) * (rho * area));
}

using BwdMomFn = void (*)(const BwdArgs, const float2*, uint64_t, uint32_t, uint32_t, int, int,
                          uint32_t, uint32_t);

template <bool T>
BwdMomFn pick_mom(int scan_mode, int cos_mode) {
  if (scan_mode == NLOS_CONFOCAL) {
    if (cos_mode == NLOS_COS_NONE) return bwd_mom_kernel<NLOS_CONFOCAL, NLOS_COS_NONE, T>;
    if (cos_mode == NLOS_COS_OBJECT) return bwd_mom_kernel<NLOS_CONFOCAL, NLOS_COS_OBJECT, T>;
    return bwd_mom_kernel<NLOS_CONFOCAL, NLOS_COS_OBJECT_WALL, T>;
  }
  if (cos_mode == NLOS_COS_NONE) return bwd_mom_kernel<NLOS_NONCONFOCAL, NLOS_COS_NONE, T>;
  if (cos_mode == NLOS_COS_OBJECT) return bwd_mom_kernel<NLOS_NONCONFOCAL, NLOS_COS_OBJECT, T>;
  return bwd_mom_kernel<NLOS_NONCONFOCAL, NLOS_COS_OBJECT_WALL, T>;
}

}  // namespace

cudaError_t launch_backward(const SceneImpl& sc, const float* grad_tau, float* grad_albedo,
                            float* grad_depth, cudaStream_t st) {
  const Geometry& g = sc.g;
  cudaError_t e;
  if (grad_albedo && (e = cudaMemsetAsync(grad_albedo, 0, sizeof(float) * g.P, st)) != cudaSuccess)
    return e;
  if (grad_depth && (e = cudaMemsetAsync(grad_depth, 0, sizeof(float) * g.P, st)) != cudaSuccess)
    return e;
  if (g.P == 0 || g.S == 0) return cudaSuccess;
  BwdArgs a{};
  a.raw = sc.raw_points;
  a.perm = sc.perm;
  a.scan = sc.scan;
  a.g = grad_tau;
  a.ga = grad_albedo;
  a.gd = grad_depth;
  a.P = g.P;
  a.S = g.S;
  a.B = g.B;
  a.scan_mode = g.scan_mode;
  a.cos_mode = g.cos_mode;
  a.lx = (float)sc.params.laser_x;
  a.ly = (float)sc.params.laser_y;
  a.inv_cdt = (float)(1.0 / g.cdt);
  const double s = g.sigma;
  a.inv2s2 = (float)(1.0 / (2.0 * s * s));
  a.inv_s2 = (float)(1.0 / (s * s));
  a.norm = (float)(1.0 / (s * std::sqrt(2.0 * 3.14159265358979323846)));
  a.reach = (float)(6.0 * s);
  a.qstep = (float)std::exp(-1.0 / (s * s));
  const size_t smem = sizeof(float) * ((size_t)g.B * kBwdTile + kBwdPoints * 8);
  int optin = 0;
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, sc.device);
  // the taps form holds a transient's bins in shared memory; splats below 2.5
  // bins, which it used to serve, keep its limit on their number
  const bool moments = adjoint_moments(s, g.P, g.B);
  if ((s < 2.5 || !moments) && smem > (size_t)optin) return cudaErrorInvalidValue;
  if (moments) {
    // moment tables of as many transients as kAdjTabBytes hold (in L2, where
    // the pair kernel gathers from them), stream-ordered, freed after use
    MomTab mt;
    moment_table(s, mt);
    AdjTabArgs t{};
    t.g = grad_tau;
    t.B = g.B;
    t.bins = g.B + 2u * (uint32_t)mt.J;
    const uint32_t rows = t.bins * (uint32_t)mt.q;
    const size_t trace_bytes = (size_t)tab_groups(rows) * kTabPitch * sizeof(float2);
    const uint64_t held = std::min<uint64_t>(
        std::min<uint64_t>(g.S, 65535), std::max<size_t>(1, kAdjTabBytes / trace_bytes));
    const uint64_t passes = (g.S + held - 1) / held;
    const uint32_t chunk = (uint32_t)((g.S + passes - 1) / passes);
    const uint32_t most = kAdjTabThreads * kAdjTabBins;
    const uint32_t ctas = (t.bins + most - 1) / most;
    t.per_cta = (t.bins + ctas - 1) / ctas;
    const unsigned threads = ((t.per_cta + kAdjTabBins - 1) / kAdjTabBins + 31u) & ~31u;
    const uint64_t n_pblk = (g.P + kBwdMomThreads - 1) / kBwdMomThreads;
    if (n_pblk * ((chunk + kBwdMomScan - 1) / kBwdMomScan) > 0x7fffffffull)
      return cudaErrorInvalidValue;
    e = cudaMallocAsync(reinterpret_cast<void**>(&t.T), trace_bytes * chunk, st);
    if (e != cudaSuccess) return e;
    for (t.s0 = 0; e == cudaSuccess && t.s0 < g.S; t.s0 += chunk) {
      const uint32_t ns = (uint32_t)std::min<uint64_t>(chunk, g.S - t.s0);
      adj_table_kernel<<<dim3(ctas, ns), threads, 0, st>>>(t, mt);
      if ((e = cudaGetLastError()) != cudaSuccess) break;
      // scan points a CTA: enough CTAs for two waves, at most kBwdMomScan
      const uint64_t want = (uint64_t)sc.num_sms * 16;
      const uint32_t per = (uint32_t)std::min<uint64_t>(
          kBwdMomScan, std::max<uint64_t>(8, (uint64_t)ns * n_pblk / want));
      const BwdMomFn fn = s < 2.5 ? pick_mom<true>(g.scan_mode, g.cos_mode)
                                  : pick_mom<false>(g.scan_mode, g.cos_mode);
      fn<<<(unsigned)(n_pblk * ((ns + per - 1) / per)), kBwdMomThreads, 0, st>>>(
          a, t.T, t.s0, ns, per, mt.J, mt.q, rows, (uint32_t)n_pblk);
      e = cudaGetLastError();
    }
    const cudaError_t ef = cudaFreeAsync(t.T, st);
    return e != cudaSuccess ? e : ef;
  }
  const uint64_t blocks = ((g.P + kBwdPoints - 1) / kBwdPoints) * ((g.S + kBwdTile - 1) / kBwdTile);
  if (blocks > 0x7fffffffull) return cudaErrorInvalidValue;
  e = cudaFuncSetAttribute(bwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  bwd_kernel<<<(unsigned)blocks, 256, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace nlos

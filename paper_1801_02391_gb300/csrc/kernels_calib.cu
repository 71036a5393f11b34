// Appendix A on the device: the calibrator's long segment, and per channel the delay that
// maximises the channel power after the common SBD is removed, then the residual phase.
//
//   X(n, j)  = sum_{k0 <= k < k0 + l} S(n, j, k)                         (FP64 sum)
//   z_j      = w(n, j) X(n, j) exp(-i 2 pi f_j SBD)
//   D(tau)   = sum_j z_j exp(-i omega_j tau),  omega_j = 2 pi (f_j - f_bw/2) 1e-3 (rad / ns)
//   tau_n    = argmax |D|^2: grid of 8 J delays (step J / (8 J f_bw) us), three-point parabola,
//              then Newton steps on |D(tau)|^2 while its curvature is negative
//   phi_n    = arg sum_j w X exp(-i 2 pi [f_j SBD + (f0_n - min f0) MBD + (f_j - f_bw/2) tau_n] 1e-3)
// The grid fit for SBD / MBD runs through the ordinary fit kernel on the summed spectrum.
//
// FP64 is the scarce pipe here (2 multiply-adds per cycle and SM against 128 in FP32), so both
// kernels are built around it.  A calibration of 15 baselines x 32 channels x 64 points from 1000
// APs: 0.21 ms, against 35.2 ms with one thread per channel (34.0 ms of FP64 sincos, one after the
// other), an FP64 chain of APs per thread (0.32 ms), the grid fit of all baselines in one CTA (0.69
// ms) and a stop on the host between the two.
#include <cfloat>

#include "frbx_internal.h"

namespace frbx {

namespace {
constexpr int kCalPad = 8;
constexpr int kCalNewton = 8;
constexpr int kSumPoints = 32;  // points per CTA of the sum (one per lane)
constexpr int kSumSplit = 32;   // interleaved shares of the APs (one per warp)
constexpr int kCalThreads = 256;

struct cd {
  double re, im;
};
__device__ __forceinline__ cd cmuld(cd a, cd b) {
  return {fma(a.re, b.re, -a.im * b.im), fma(a.re, b.im, a.im * b.re)};
}
__device__ __forceinline__ cd cis(double ph) {  // exp(i ph)
  double s, c;
  sincos(ph, &s, &c);
  return {c, s};
}

// Exact sum of two floats: a + b = s + e (Knuth's two-sum)
__device__ __forceinline__ float two_sum(float a, float b, float &e) {
  const float s = __fadd_rn(a, b), z = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
  return s;
}
// Running sum of floats kept as three floats: the rounding error of each addition is added to a
// second sum without error, and that sum's own errors to a third (about 2^-70 of the terms).
struct Sum3 {
  float s = 0.f, e = 0.f, f = 0.f;
  __device__ __forceinline__ void add(float x) {
    float d, g;
    s = two_sum(s, x, d);
    e = two_sum(e, d, g);
    f += g;
  }
  __device__ __forceinline__ double value() const { return (double)s + ((double)e + (double)f); }
};
}  // namespace

// Sum of the calibrator APs per (baseline, point), a complex64 copy of it (one "AP" per baseline)
// that feeds the grid fit, and that fit's unit weights (no calibration rotation: the extraction
// starts from zero delays and phases), zero shifts and segment rows.
//
// CTA: 32 points of one baseline x 32 warps, warp v taking APs v, v + 32, ...  The shares are
// summed in three floats each (Sum3), whose result is at least as near the exact sum as a chain of
// FP64 additions, and added up in FP64: an FP64 chain costs a conversion and an addition per value
// on a pipe 64 times slower.  A share that is not finite (overflow, or such an input) is summed
// again in FP64.
__global__ void __launch_bounds__(kSumPoints * kSumSplit)
    k_cal_sum(const float2 *vis, int T, int C, int k0, int l, const float2 *wrot, double2 *xsum, float2 *xcube,
              float2 *wunit, int *dk, int4 *rows) {
  __shared__ double2 part[kSumSplit][kSumPoints + 1];
  const int lane = threadIdx.x & 31, share = threadIdx.x >> 5;
  const int b = blockIdx.y, c = blockIdx.x * kSumPoints + lane;
  double2 t = make_double2(0.0, 0.0);
  if (c < C && share < l) {
    const float2 *p = vis + ((size_t)b * T + k0) * C + c;
    Sum3 sr, si;
#pragma unroll 8
    for (int k = share; k < l; k += kSumSplit) {
      const float2 v = __ldg(p + (size_t)k * C);
      sr.add(v.x);
      si.add(v.y);
    }
    t = make_double2(sr.value(), si.value());
    if (!(fabs(t.x) <= DBL_MAX && fabs(t.y) <= DBL_MAX)) {
      t = make_double2(0.0, 0.0);
      for (int k = share; k < l; k += kSumSplit) {
        const float2 v = __ldg(p + (size_t)k * C);
        t.x += (double)v.x;
        t.y += (double)v.y;
      }
    }
  }
  part[share][lane] = t;
  __syncthreads();
  if (share == 0 && c < C) {
    for (int v = 1; v < kSumSplit; ++v) {
      t.x += part[v][lane].x;
      t.y += part[v][lane].y;
    }
    const size_t i = (size_t)b * C + c;
    xsum[i] = t;
    xcube[i] = make_float2((float)t.x, (float)t.y);
    if (b == 0) {
      const float2 w = wrot[c];
      wunit[c] = (w.x != 0.f || w.y != 0.f) ? make_float2(1.f, 0.f) : make_float2(0.f, 0.f);
      dk[c] = 0;
    }
    if (c == 0) rows[b] = make_int4(b, 0, 1, 0);
  }
}

// One CTA per (channel, baseline).
//
// The grid search is a transform of J inputs onto L = 8 J delays: omega_j tau_p = 2 pi (j - J/2) p / L
// for the grid delay p (a common phase does not change |D|), so D(8 a + r) = sum_j [z_j w_L^(j r)]
// w_J^(j a): eight FFTs of J points in shared memory instead of 8 J sums of J sincos.  The Newton
// steps need exp(-i omega_j tau) at one tau for J equally spaced omega_j: products of two factors
// (j = 16 h + r), so 16 + J / 16 sincos instead of J.  Steps that no longer move tau end the loop.
// One warp takes the Newton steps and the residual phase.
__global__ void __launch_bounds__(kCalThreads)
    k_cal_channels(const double2 *xsum, const float2 *wrot, const frbx_seg *fit, int N, int J, int Ls, int Lm,
                   double f_bw, double df_grid, const double *f0, double f0_min, double *sbd_ns, double *mbd_ns,
                   double *delay_ns, double *phase_rad) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int n = blockIdx.x, b = blockIdx.y, L = kCalPad * J, lgJ = __ffs(J) - 1;
  cd *z = reinterpret_cast<cd *>(smem);  // [J]
  cd *g = z + J;                         // [8][J]
  cd *tw = g + L;                        // [J] w_J^a, then [8] w_L^r
  __shared__ double red_p[kCalThreads / 32];
  __shared__ int red_i[kCalThreads / 32];
  const double two_pi = 6.283185307179586476925286766559;
  // the grid cell of the common fit as delays (the order of operations of frbx_search's candidates)
  const int m = fit[b].sbd_idx, q = fit[b].mbd_idx;
  const int sm = m < Ls / 2 ? m : m - Ls, sq = q < Lm / 2 ? q : q - Lm;
  const double sbd = __ddiv_rn(__dmul_rn(__dmul_rn((double)sm, (double)J), 1000.0), __dmul_rn((double)Ls, f_bw));
  const double mbd = __ddiv_rn(__dmul_rn((double)sq, 1000.0), __dmul_rn((double)Lm, df_grid));
  if (n == 0 && threadIdx.x == 0) {
    sbd_ns[b] = sbd;
    mbd_ns[b] = mbd;
  }
  const double2 *x = xsum + (size_t)b * N * J + (size_t)n * J;
  const float2 *wr = wrot + (size_t)n * J;
  for (int j = threadIdx.x; j < J; j += blockDim.x) {
    const double fj = ((double)j * f_bw) / (double)J;
    const float2 w = wr[j];
    const bool used = (w.x != 0.f || w.y != 0.f);
    z[j] = used ? cmuld({x[j].x, x[j].y}, cis(-two_pi * fj * sbd * 1e-3)) : cd{0.0, 0.0};
    double s, c;
    sincospi(2.0 * (double)j / (double)J, &s, &c);
    tw[j] = {c, -s};
    if (j < kCalPad) {
      sincospi(2.0 * (double)j / (double)L, &s, &c);
      tw[J + j] = {c, -s};
    }
  }
  if (J < kCalPad)
    for (int j = J + threadIdx.x; j < kCalPad; j += blockDim.x) {
      double s, c;
      sincospi(2.0 * (double)j / (double)L, &s, &c);
      tw[J + j] = {c, -s};
    }
  __syncthreads();
  // g[r][j] = z_j w_L^(j r), j r = 8 a + e
  for (int i = threadIdx.x; i < L; i += blockDim.x) {
    const int r = i >> lgJ, j = i & (J - 1), ex = j * r;
    g[i] = cmuld(z[j], cmuld(tw[ex >> 3], tw[J + (ex & 7)]));
  }
  __syncthreads();
  // radix-2 decimation in frequency; position i of row r ends up holding a = bitrev(i)
  for (int lg = lgJ - 1; lg >= 0; --lg) {
    const int S = 1 << lg;
    for (int i = threadIdx.x; i < L / 2; i += blockDim.x) {
      const int r = i >> (lgJ - 1), k = i & (J / 2 - 1);
      const int lo = r * J + ((k >> lg) << (lg + 1)) + (k & (S - 1));
      const cd u = g[lo], v = g[lo + S];
      g[lo] = {u.re + v.re, u.im + v.im};
      g[lo + S] = cmuld({u.re - v.re, u.im - v.im}, tw[(k & (S - 1)) << (lgJ - 1 - lg)]);
    }
    __syncthreads();
  }
  auto power_at = [&](int p) {
    const int a = p >> 3, i = lgJ ? (int)(__brev((unsigned)a) >> (32 - lgJ)) : 0;
    const cd d = g[(p & 7) * J + i];
    return d.re * d.re + d.im * d.im;
  };
  // argmax in ascending p (the lowest of equal powers)
  double best = -1.0;
  int kb = 0;
  for (int p = threadIdx.x; p < L; p += blockDim.x) {
    const double pw = power_at(p);
    if (pw > best) {
      best = pw;
      kb = p;
    }
  }
  auto keep = [&](double p2, int k2) {
    if (p2 > best || (p2 == best && k2 < kb)) {
      best = p2;
      kb = k2;
    }
  };
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const double p2 = __shfl_xor_sync(0xffffffffu, best, o);
    keep(p2, __shfl_xor_sync(0xffffffffu, kb, o));
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    red_p[warp] = best;
    red_i[warp] = kb;
  }
  __syncthreads();
  if (warp != 0) return;
  for (int w = 1; w < kCalThreads / 32; ++w) keep(red_p[w], red_i[w]);
  if (!(best >= 0.0)) kb = 0;  // no finite power: the first delay, as a scan from there keeps it
  // three-point parabola
  const double pw_m = power_at((kb - 1 + L) % L), pw_p = power_at((kb + 1) % L);
  const double den = pw_m - 2.0 * best + pw_p;
  const double off = den == 0.0 ? 0.0 : 0.5 * (pw_m - pw_p) / den;
  const double step = ((double)J * 1000.0) / ((double)L * f_bw);
  double tau = ((kb < L / 2 ? kb : kb - L) + off) * step;
  // Newton steps on |D|^2
  const double dw = two_pi * 1e-3 * f_bw / (double)J, w_0 = -two_pi * 1e-3 * f_bw / 2.0;  // omega_j = w_0 + j dw
  auto rotor = [&](double t) {  // lane r < 16: exp(-i (w_0 + r dw) t); lane 16 + h: exp(-i 16 h dw t)
    return cis(-(lane < 16 ? w_0 + lane * dw : (lane - 16) * 16 * dw) * t);
  };
  auto warp_sum = [&](double v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  for (int it = 0; it < kCalNewton; ++it) {
    const cd ro = rotor(tau);
    double s[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int j0 = 0; j0 < J; j0 += 32) {
      const int j = j0 + lane, h = j >> 4, r = j & 15;
      const cd a = {__shfl_sync(0xffffffffu, ro.re, r), __shfl_sync(0xffffffffu, ro.im, r)};
      const cd c = {__shfl_sync(0xffffffffu, ro.re, 16 + (h & 15)), __shfl_sync(0xffffffffu, ro.im, 16 + (h & 15))};
      if (j < J) {
        const double om = w_0 + j * dw;
        const cd e = cmuld(z[j], cmuld(a, c));
        s[0] += e.re;
        s[1] += e.im;
        s[2] += om * e.im;  // (-i w) e: real part = w * imag
        s[3] -= om * e.re;
        s[4] -= om * om * e.re;
        s[5] -= om * om * e.im;
      }
    }
#pragma unroll
    for (double &v : s) v = warp_sum(v);
    const double f1 = 2.0 * (s[0] * s[2] + s[1] * s[3]);
    const double f2 = 2.0 * (s[2] * s[2] + s[3] * s[3] + s[0] * s[4] + s[1] * s[5]);
    if (!(f2 < 0.0)) break;
    const double d = f1 / f2;
    tau -= d;
    if (fabs(d) <= 1e-15 * step) break;
  }
  // residual phase with the common SBD / MBD and the channel delay removed
  double sr = 0.0, si = 0.0;
  for (int j = lane; j < J; j += 32) {
    const double fj = ((double)j * f_bw) / (double)J;
    const float2 w = wr[j];
    if (w.x == 0.f && w.y == 0.f) continue;
    const cd e = cmuld({x[j].x, x[j].y},
                       cis(-two_pi * (fj * sbd + (f0[n] - f0_min) * mbd + (fj - f_bw / 2.0) * tau) * 1e-3));
    sr += e.re;
    si += e.im;
  }
  sr = warp_sum(sr);
  si = warp_sum(si);
  if (lane == 0) {
    delay_ns[(size_t)b * N + n] = tau;
    phase_rad[(size_t)b * N + n] = atan2(si, sr);
  }
}

cudaError_t launch_cal_sum(const float2 *vis, int T, int C, int n_bl, int k0, int l, const float2 *wrot,
                           double2 *xsum, float2 *xcube, float2 *wunit, int *dk, int4 *rows, cudaStream_t st,
                           int64_t *launches) {
  const dim3 grid((unsigned)((C + kSumPoints - 1) / kSumPoints), (unsigned)n_bl);
  k_cal_sum<<<grid, kSumPoints * kSumSplit, 0, st>>>(vis, T, C, k0, l, wrot, xsum, xcube, wunit, dk, rows);
  ++*launches;
  return cudaGetLastError();
}

cudaError_t launch_cal_channels(const double2 *xsum, const float2 *wrot, const frbx_seg *fit, int n_bl, int N, int J,
                                int Ls, int Lm, double f_bw, double df_grid, const double *f0, double f0_min,
                                double *sbd_ns, double *mbd_ns, double *delay_ns, double *phase_rad, cudaStream_t st,
                                int64_t *launches) {
  // J <= 256 (kMaxPoint): 10 J + 8 values, 41 KB
  static_assert(sizeof(cd) * (10 * kMaxPoint + kCalPad) <= 48 * 1024, "default shared memory");
  static_assert(kMaxPoint <= 256, "16 x 16 rotors");
  const size_t smem = sizeof(cd) * (size_t)((2 + kCalPad) * J + kCalPad);
  k_cal_channels<<<dim3((unsigned)N, (unsigned)n_bl), kCalThreads, smem, st>>>(
      xsum, wrot, fit, N, J, Ls, Lm, f_bw, df_grid, f0, f0_min, sbd_ns, mbd_ns, delay_ns, phase_rad);
  ++*launches;
  return cudaGetLastError();
}

}  // namespace frbx

// Dispersion shift table (Eq. 1-2) and the normalisation / threshold stage (Eq. 6,
// Sec. 2.4.1 step a) for baselines and for baseline combinations (Sec. 2.4.2 step b).
#include <cfloat>
#include <cmath>

#include "frbx_internal.h"

namespace frbx {

// ---------------------------------------------------------------- Eq. 1-2
// dk = floor(0.5 + ((4.15e6 * DM) * (1/(f*f) - 1/(fref*fref))) / t_ap), every step a
// correctly rounded FP64 operation (explicit _rn intrinsics: no contraction), so the
// table is reproducible bit for bit on any IEEE host.
__global__ void k_shift_table(const double *__restrict__ f, int C, double inv_fref2,
                              const double *__restrict__ dm, int n_dm, double t_ap,
                              int *__restrict__ dk) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)n_dm * C) return;
  const int d = (int)(i / C), c = (int)(i - (long long)d * C);
  const double fc = f[c];
  const double b = __dsub_rn(__ddiv_rn(1.0, __dmul_rn(fc, fc)), inv_fref2);
  const double dt = __dmul_rn(__dmul_rn(4.15e6, dm[d]), b);
  double x = __dadd_rn(0.5, __ddiv_rn(dt, t_ap));
  x = fmin(x, 1.0e9);  // keeps the int conversion defined for absurd DM; no segment is then valid
  dk[i] = (int)floor(x);
}

__global__ void k_row_max(const int *__restrict__ dk, int C, int *__restrict__ out) {
  __shared__ int red[32];
  const int d = blockIdx.x;
  int m = 0;
  for (int c = threadIdx.x; c < C; c += blockDim.x) m = max(m, dk[(size_t)d * C + c]);
#pragma unroll
  for (int off = 16; off; off >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, off));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = max(m, red[w]);
    out[d] = m;
  }
}

int shift_of(double f, double inv_fref2, double dm, double t_ap) {
  const double b = 1.0 / (f * f) - inv_fref2, dt = (4.15e6 * dm) * b;
  return (int)std::floor(std::fmin(0.5 + dt / t_ap, 1.0e9));
}

cudaError_t launch_shift_table(const double *f, int C, double fref, const double *dm, int n_dm,
                               double t_ap, int *dk, int *dk_max, cudaStream_t st,
                               int64_t *launches) {
  const long long n = (long long)n_dm * C;
  if (n == 0) return cudaSuccess;
  const double inv_fref2 = 1.0 / (fref * fref);
  const int threads = 256;
  k_shift_table<<<(unsigned)((n + threads - 1) / threads), threads, 0, st>>>(f, C, inv_fref2, dm,
                                                                            n_dm, t_ap, dk);
  ++*launches;
  if (dk_max) {
    k_row_max<<<n_dm, 256, 0, st>>>(dk, C, dk_max);
    ++*launches;
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------- Eq. 6 + threshold
// Amplitude of slot i of series s at DM d: a baseline's |G|, or for a combination the
// sum of |G| over its baselines (Sec. 2.4.2: the "power" summed is the amplitude).
__device__ __forceinline__ double series_value(const StatsArgs &a, int s, int d, int slot) {
  if (!a.masks) return (double)a.series[((size_t)s * a.n_dm + d) * a.S_tot + slot].amp;
  const unsigned long long mask = a.masks[s];
  double v = 0.0;
  for (int b = 0; b < a.n_bl; ++b)
    if ((mask >> b) & 1ull) v += (double)a.series[((size_t)b * a.n_dm + d) * a.S_tot + slot].amp;
  return v;
}

__device__ __forceinline__ double block_sum(double v, double *red) {
#pragma unroll
  for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  const int warp = threadIdx.x >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[warp] = v;
  __syncthreads();
  double t = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
  return t;
}

// Exact sum of two floats: a + b = s + e (Knuth's two-sum)
__device__ __forceinline__ float two_sum(float a, float b, float &e) {
  const float s = __fadd_rn(a, b), z = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
  return s;
}
// a float pair hi + lo (|lo| at most half a unit in the last place of hi: about 48 bits)
struct Pair {
  float hi, lo;
};
__device__ __forceinline__ Pair to_pair(double v) {
  const float h = (float)v;
  return {h, (float)(v - (double)h)};
}
// running sum of floats in three floats: no rounding above about 2^-70 of the terms
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

// series_value as three floats (their sum to about 2^-70 of the amplitudes; a baseline's is one)
struct Tri {
  float hi = 0.f, mid = 0.f, lo = 0.f;
};
template <bool kCombo>
__device__ __forceinline__ Tri series_tri(const StatsArgs &a, int s, int d, int slot) {
  Tri v;
  if constexpr (!kCombo) {
    v.hi = a.series[((size_t)s * a.n_dm + d) * a.S_tot + slot].amp;
  } else {
    const unsigned long long mask = a.masks[s];
    for (int b = 0; b < a.n_bl; ++b)
      if ((mask >> b) & 1ull) {
        float e, g;
        v.hi = two_sum(v.hi, a.series[((size_t)b * a.n_dm + d) * a.S_tot + slot].amp, e);
        v.mid = two_sum(v.mid, e, g);
        v.lo += g;
      }
  }
  return v;
}

// v - c - (m.hi + m.lo) to about 2^-46 of itself, of m and of 2^-24 v (v.mid may be as large as the result)
template <bool kCombo>
__device__ __forceinline__ Pair minus(Tri v, float c, Pair m) {
  float e1, e2, rest;
  const float s1 = two_sum(v.hi, -c, e1);
  float s2 = two_sum(s1, -m.hi, e2);
  if constexpr (kCombo) {
    float f1, f2;
    const float t = two_sum(e1, v.mid, f1);
    s2 = two_sum(s2, t, f2);
    rest = (e2 + f2) + ((f1 + v.lo) - m.lo);
  } else {
    rest = e2 + (e1 - m.lo);
  }
  Pair r;
  r.hi = two_sum(s2, rest, r.lo);
  return r;
}

// words of the hit mask of window w of one (series, DM): its slots' bits start at word (off >> 5) + w
__host__ __device__ __forceinline__ size_t hit_words(int S_tot, int n_win) { return (size_t)(S_tot >> 5) + n_win + 1; }

// One CTA per (window, DM, series): population mean and std over the valid segments, then the
// crossings P = (A - mean) / std > threshold, their count and one bit each; optionally writes P.
//
// FP64 runs at a 64th of FP32's rate here, and a division of it per slot was most of this kernel and of
// the one that writes the events.  The results are those of FP64 all the same:
//  * mean and std come from the differences from c, an estimate of the mean, and their squares, without
//    rounding errors above 2^-48 of a term and summed in three floats each; c is taken anew where it is
//    farther than one std from the mean, so the shift of the squares loses one bit at most;
//  * P is formed in float pairs, and taken when every value within their error rounds to the same float;
//    otherwise the FP64 expression is evaluated (about one slot in 10^5);
//  * a crossing within 1e-9 of the threshold is decided by the FP64 expression.
// Series whose squares FP32 cannot hold, that vary by less than a float resolves, or with a
// value that is not finite, take FP64 throughout.  With k_events and k_scan below, for 3 baselines x 101
// DM trials x 4096 APs and four combinations: 0.76 -> 0.34 ms.
template <bool kCombo>
__global__ void __launch_bounds__(256) k_stats_count(StatsArgs a) {
  __shared__ double red[32];
  const int w = blockIdx.x, d = blockIdx.y, s = blockIdx.z;
  const int nv = a.n_valid[d * a.n_win + w];
  const int off = a.win_off[w];
  const size_t sid = ((size_t)s * a.n_dm + d) * a.n_win + w;
  unsigned *const bits = a.hits + ((size_t)s * a.n_dm + d) * hit_words(a.S_tot, a.n_win) + (off >> 5) + w;
  double mean = 0.0, sd = 0.0;
  float c = 0.f;
  bool fast = nv > 0;
  if (fast) {  // the mean of 32 slots spread over the series (every warp the same)
    c = series_tri<kCombo>(a, s, d, off + (int)((long long)(threadIdx.x & 31) * nv >> 5)).hi;
#pragma unroll
    for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    c *= 0.03125f;
  }
  for (int pass = 0; fast && pass < 2; ++pass) {
    Sum3 s1, s2;
    bool differ = false;
    for (int i = threadIdx.x; i < nv; i += blockDim.x) {
      const Pair x = minus<kCombo>(series_tri<kCombo>(a, s, d, off + i), c, {0.f, 0.f});
      differ = differ || x.hi != 0.f;
      const float q = __fmul_rn(x.hi, x.hi);
      s1.add(x.hi);
      s2.add(q);
      s2.add(fmaf(x.hi, x.hi, -q));
      if (x.lo != 0.f) {
        const float p = __fmul_rn(2.f * x.hi, x.lo);
        s1.add(x.lo);
        s2.add(p);
        s2.add(fmaf(x.lo, x.lo, fmaf(2.f * x.hi, x.lo, -p)));
      }
    }
    const double t1 = block_sum(s1.value(), red), t2 = block_sum(s2.value(), red);
    const double shift = t1 / nv, var = fmax(t2 / nv - shift * shift, 0.0);
    mean = (double)c + shift;
    sd = sqrt(var);
    // squares within FP32 with room for their rounding terms, or all equal (no difference at all: squares
    // that vanish are not it); false for NaN
    fast = __syncthreads_or(differ) == 0 || (t2 >= 1e-18 * nv && t2 <= 1e28);
    if (shift * shift <= var) break;
    if (pass == 1) fast = false;
    c = (float)mean;
  }
  if (!fast && nv > 0) {
    double sum = 0.0;
    for (int i = threadIdx.x; i < nv; i += blockDim.x) sum += series_value(a, s, d, off + i);
    mean = block_sum(sum, red) / nv;
    double sq = 0.0;
    for (int i = threadIdx.x; i < nv; i += blockDim.x) {
      const double dv = series_value(a, s, d, off + i) - mean;
      sq += dv * dv;
    }
    sd = sqrt(block_sum(sq, red) / nv);
  }
  const double inv = sd > 0.0 ? 1.0 / sd : 0.0;
  const Pair m = to_pair(mean - (double)c), r = to_pair(inv), th = to_pair(a.threshold);
  // P's error is below 2^-44 of itself and of m / sd; 1e-37: products that FP32 holds with fewer bits
  const float err0 = fmaf(fabsf(m.hi) * r.hi, 0x1p-43f, 1e-37f);
  int cnt = 0;
  for (int i0 = threadIdx.x & ~31; i0 < nv; i0 += blockDim.x) {  // 32 slots of a warp: one word
    const int i = i0 + (threadIdx.x & 31);
    bool hit = false;
    float pn = 0.f;
    if (i < nv) {
      bool sure = fast && sd > 0.0;
      if (sure) {
        const Tri v = series_tri<kCombo>(a, s, d, off + i);
        const Pair x = minus<kCombo>(v, c, m);
        const float ph = __fmul_rn(x.hi, r.hi), pl = fmaf(x.hi, r.lo, fmaf(x.lo, r.hi, fmaf(x.hi, r.hi, -ph)));
        const float g = (ph - th.hi) + (pl - th.lo);
        hit = g > 0.f;
        // (the FP64 sum of a combination is rounded itself: 2^-53 of each amplitude); false for NaN
        sure = fabsf(g) > 1e-9f * (1.f + fabsf(ph)) + (kCombo ? 1e-14f * fabsf(v.hi) * r.hi : 0.f);
        if (a.pnorm) {
          const float err = fmaf(fabsf(ph), 0x1p-43f, err0);
          pn = ph + (pl - err);
          sure = sure && pn == ph + (pl + err);
        }
      }
      if (!sure) {
        const double p = sd > 0.0 ? (series_value(a, s, d, off + i) - mean) / sd : 0.0;
        hit = p > a.threshold;
        pn = (float)p;
      }
      if (a.pnorm) a.pnorm[((size_t)s * a.n_dm + d) * a.S_tot + off + i] = pn;
    }
    const unsigned bal = __ballot_sync(0xffffffffu, hit);
    if ((threadIdx.x & 31) == 0) {
      if (a.hits) bits[i0 >> 5] = bal;
      cnt += __popc(bal);
    }
  }
  const double total = block_sum((double)cnt, red);
  if (threadIdx.x == 0) {
    a.mean_std[2 * sid] = mean;
    a.mean_std[2 * sid + 1] = sd;
    a.counts[sid] = (int)total;
  }
}

// Exclusive sum over a CTA of 1024 threads; total gets the sum.
__device__ __forceinline__ long long block_exclusive(long long v, long long *warp_sum, long long &total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  long long inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  __syncthreads();
  if (lane == 31) warp_sum[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const long long x = lane < nw ? warp_sum[lane] : 0;
    long long y = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long t = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += t;
    }
    warp_sum[lane] = y - x;
    if (lane == 31) warp_sum[32] = y;
  }
  __syncthreads();
  total = warp_sum[32];
  return warp_sum[warp] + inc - v;
}

// Exclusive scan of the per-(series, DM, window) counts into offsets (one CTA).
__global__ void __launch_bounds__(1024) k_scan(const int *__restrict__ counts, long long n,
                                               long long *__restrict__ offsets) {
  __shared__ long long part[33];
  const long long chunk = (n + blockDim.x - 1) / blockDim.x;
  const long long lo = threadIdx.x * chunk, hi = min(n, lo + chunk);
  long long s = 0, total;
  for (long long i = lo; i < hi; ++i) s += counts[i];
  long long run = block_exclusive(s, part, total);
  if (threadIdx.x == 0) offsets[n] = total;
  for (long long i = lo; i < hi; ++i) {
    offsets[i] = run;
    run += counts[i];
  }
}

// The crossings of one (window, DM, series) in ascending k0, from the bits k_stats_count left or, where there
// was no room for them, from the FP64 expression that they agree with.
__global__ void __launch_bounds__(256) k_events(StatsArgs a) {
  __shared__ long long part[33];
  const int w = blockIdx.x, d = blockIdx.y, s = blockIdx.z;
  const size_t sid = ((size_t)s * a.n_dm + d) * a.n_win + w;
  if (a.counts[sid] == 0) return;
  const int nv = a.n_valid[d * a.n_win + w], nw = (nv + 31) >> 5;
  const int off = a.win_off[w], step = a.win_step[w];
  const unsigned *const bits = a.hits + ((size_t)s * a.n_dm + d) * hit_words(a.S_tot, a.n_win) + (off >> 5) + w;
  const double mean = a.mean_std[2 * sid], sd = a.mean_std[2 * sid + 1];
  long long out = a.offsets[sid];
  const long long end = a.offsets[sid + 1];
  for (int c0 = 0; c0 < nw; c0 += blockDim.x) {
    const int q = c0 + threadIdx.x;
    unsigned word = 0u;
    if (a.hits) {
      if (q < nw) word = bits[q];
    } else {
      for (int i = q * 32; i < min(nv, q * 32 + 32); ++i)
        if ((sd > 0.0 ? (series_value(a, s, d, off + i) - mean) / sd : 0.0) > a.threshold) word |= 1u << (i & 31);
    }
    long long total;
    long long pos = out + block_exclusive(__popc(word), part, total);
    for (; word != 0u && pos < end; word &= word - 1u, ++pos) {
      const int i = q * 32 + __ffs((int)word) - 1;
      const double v = series_value(a, s, d, off + i);
      frbx_event e;
      e.series = a.series_base + s;
      e.dm_idx = d;
      e.win_idx = w;
      e.k0 = i * step;
      e.amp = (float)v;
      e.pnorm = (float)(sd > 0.0 ? (v - mean) / sd : 0.0);
      if (!a.masks) {
        const frbx_seg sg = a.series[((size_t)s * a.n_dm + d) * a.S_tot + off + i];
        e.sbd_idx = sg.sbd_idx;
        e.mbd_idx = sg.mbd_idx;
      } else {
        e.sbd_idx = 0;
        e.mbd_idx = 0;
      }
      a.events[pos] = e;
    }
    out += total;
  }
}

size_t stats_hit_bytes(int n_series, int n_dm, int S_tot, int n_win) {
  return sizeof(unsigned) * (size_t)n_series * n_dm * hit_words(S_tot, n_win);
}

cudaError_t launch_stats_count(const StatsArgs &a, cudaStream_t st, int64_t *launches) {
  if (a.n_series == 0 || a.n_dm == 0 || a.n_win == 0) return cudaSuccess;
  const dim3 grid(a.n_win, a.n_dm, a.n_series);
  if (a.masks) k_stats_count<true><<<grid, 256, 0, st>>>(a);
  else k_stats_count<false><<<grid, 256, 0, st>>>(a);
  ++*launches;
  return cudaGetLastError();
}

cudaError_t launch_scan(const StatsArgs &a, cudaStream_t st, int64_t *launches) {
  const long long n = (long long)a.n_series * a.n_dm * a.n_win;
  k_scan<<<1, 1024, 0, st>>>(a.counts, n, a.offsets);
  ++*launches;
  return cudaGetLastError();
}

cudaError_t launch_events(const StatsArgs &a, cudaStream_t st, int64_t *launches) {
  if (a.n_series == 0 || a.n_dm == 0 || a.n_win == 0) return cudaSuccess;
  k_events<<<dim3(a.n_win, a.n_dm, a.n_series), 256, 0, st>>>(a);
  ++*launches;
  return cudaGetLastError();
}

}  // namespace frbx

// Window tree of 16-column MBD grids (Lm = 16, the S-band layout) in one kernel.
//
// One AP of such a setup is small: 8 x 32 points make a delay-resolution matrix of 64 x 16 cells.  As
// two passes (k_tree_sbd and k_tree_mbd) every AP went through device memory and each step of the tree
// waited on it, with one AP in flight per CTA.  Here a CTA of 128 threads keeps everything on the SM:
// a thread owns one SBD row, all 16 cells of it, and 128 / Ls time tiles of one series run side by
// side.  A step takes four APs of every tile:
//   SBD   task (AP, channel, m1) per thread (16 N <= 128 of them): a 32-point register FFT of the
//         gathered points in shared memory, its rows written as pairs of channel slots;
//   tree  each thread reads its row of the four APs (8 slots, 16-byte reads of neighbouring rows),
//         16-point FFTs, and the window tree: the matrices of levels 0 to 2 of four APs are a fixed
//         pattern in registers, deeper anchors (every fourth AP and rarer) sit in local memory;
//   the points of the next step are gathered during the tree, four loads per thread beside each AP.
// The arithmetic, its order and the keys are those of k_tree_sbd and k_tree_mbd (Lm = 16), so the
// results are the same bits; segments' maxima are merged per warp by a 64-bit atomicMax.
// The S-band search of 3 baselines x 101 DM trials x 4096 APs: both passes 13.0 -> 3.1 ms (the two-pass
// form issued on few of its cycles: two serial device reads per AP, half of each CTA's threads idle).
// Three-input maxima, a first FFT stage without its zeros and reads of two points: call 4.64 -> 4.55 ms.
// Every sum (FFTs and windows) as packed pairs: kernel 2.98 -> 2.75 ms, call 4.40 -> 4.15 ms (the windows' sums
// alone 2.94 ms).  Three CTAs per SM allow 168 registers, at which ptxas spills 144 to 336 bytes a thread (80 to 548 of
// loads) beside the deep anchors that are meant to be there; four at 128 registers: 5.78 ms.
#include "fit_common.cuh"
#include "fft32.cuh"

namespace frbx {

namespace {

constexpr int kThreads16 = 128;
constexpr int kStep16 = 4;    // APs per step of a time tile
constexpr int kSlots16 = 8;   // channel slots: g_n < 8
constexpr int kDeep16 = 4;    // levels 3 to 6
constexpr int kMaxLev16 = 6;  // windows up to 64 APs

// SBD rows of a pair of slots: padded so that the pairs' rows fall on different banks
__host__ __device__ constexpr int pair_stride(int Ls) { return Ls + 2; }
__host__ __device__ inline size_t tree16_smem(int Ls, int N, int J1) {
  const int aps = kThreads16 / Ls * kStep16, xs = J1 * 32 + 2;
  return sizeof(float4) * (size_t)aps * (kSlots16 / 2) * pair_stride(Ls) +
         sizeof(float2) * ((size_t)aps * N * xs + (size_t)(Ls / 32) * xs);
}

}  // namespace

// kPS: Ls / 32.  kFull: the whole delay grid is searched.
template <int kPS, bool kFull>
__global__ void __launch_bounds__(kThreads16, 3)
    k_tree16(const __grid_constant__ FitArgs a, const __grid_constant__ TreeArgs t) {
  constexpr int Ls = 32 * kPS, kSub = kThreads16 / Ls, kAps = kSub * kStep16, kPairs = kSlots16 / 2;
  constexpr int kYAp = kPairs * pair_stride(Ls);  // float4 per AP
  extern __shared__ __align__(16) unsigned char smem[];
  const int N = a.N, J = a.J, C = a.C, xs = a.J1 * 32 + 2;  // even: two points a read, rows 16 bytes apart on the banks
  float4 *Y = reinterpret_cast<float4 *>(smem);           // [kAps][kPairs][Ls + 2] slots 2p, 2p + 1
  float2 *X = reinterpret_cast<float2 *>(Y + kAps * kYAp);  // [kAps][N][xs]
  float2 *stw = X + kAps * N * xs;                        // [kPS][xs]
  const int tid = threadIdx.x;
  for (int i = tid; i < kAps * kYAp; i += kThreads16) Y[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int i = tid; i < kAps * N * xs; i += kThreads16) X[i] = make_float2(0.f, 0.f);
  for (int i = tid; i < kPS * a.J1 * 32; i += kThreads16) {
    const int r = i / (a.J1 * 32), c = i - r * a.J1 * 32;
    stw[r * xs + c] = a.sbd_tw[i];
  }
  // DM trials vary fastest, so the CTAs resident together read the same stretch of the cube
  const int s = blockIdx.x % t.n_s, tg = blockIdx.x / t.n_s;
  const int2 sd = t.series[s];
  const int kd = t.T - t.dk_max[sd.y], lmax = 1 << t.nlev;
  const int kb0 = tg * kSub * t.TT;  // first AP of the CTA's first time tile
  auto tile_n = [&](int sub) { return min(kd - kb0 - sub * t.TT, t.TT + lmax - 1); };  // APs of a tile (may be < 0)
  const int n_step = (tile_n(0) + kStep16 - 1) / kStep16;  // tiles only get shorter
  if (n_step <= 0) return;
  __syncthreads();

  // gather: this thread's points c = tid + 128 h of every AP of the step
  const float2 *vis = a.vis + ((size_t)sd.x * t.T + kb0) * C;
  int coff[kPS], xi[kPS];
#pragma unroll
  for (int h = 0; h < kPS; ++h) {
    const int c = tid + kThreads16 * h;
    coff[h] = c < C ? __ldg(a.dk + (size_t)sd.y * C + c) * C + c : -1;
    xi[h] = c < C ? (c / J) * xs + c % J : 0;
  }
  constexpr int kPart = kAps * kPS / 4;  // 4 loads of each of the four batches
  auto load = [&](int step, int batch, float2(&v)[kPart]) {
#pragma unroll
    for (int i = 0; i < kPart; ++i) {
      const int e = batch * kPart + i, ap = e / kPS, h = e % kPS, sub = ap / kStep16;
      const int k = step * kStep16 + ap % kStep16;  // AP of its time tile
      v[i] = coff[h] >= 0 && k < tile_n(sub) ? __ldg(vis + (size_t)(sub * t.TT + k) * C + coff[h]) : make_float2(0.f, 0.f);
    }
  };
  auto keep = [&](int batch, const float2(&v)[kPart]) {
#pragma unroll
    for (int i = 0; i < kPart; ++i) {
      const int e = batch * kPart + i, ap = e / kPS, h = e % kPS;
      if (coff[h] >= 0) X[ap * N * xs + xi[h]] = cmul(v[i], __ldg(a.wrot + tid + kThreads16 * h));
    }
  };
  {
#pragma unroll
    for (int q = 0; q < kStep16; ++q) {
      float2 v[kPart];
      load(0, q, v);
      keep(q, v);
    }
  }
  __syncthreads();

  // SBD task of this thread: AP s_ap, channel s_n (slot of its residue), rows s_m1 + kPS b
  const bool task = tid < kAps * N * kPS;
  const int s_ap = task ? tid / (N * kPS) : 0, s_r = task ? tid % (N * kPS) : 0, s_n = s_r / kPS, s_m1 = s_r % kPS;
  const int slot = __ldg(t.slot_of + s_n);
  float2 *const yw = reinterpret_cast<float2 *>(Y + s_ap * kYAp + (slot >> 1) * pair_stride(Ls) + s_m1) + (slot & 1);
  const float2 *const xr = X + (s_ap * N + s_n) * xs, *const wr = stw + s_m1 * xs;

  // tree: this thread's row of its time tile
  const int sub = tid / Ls, m = tid % Ls;
  const float4 *const yr = Y + sub * kStep16 * kYAp + m;
  const int kb = kb0 + sub * t.TT, n_ap = tile_n(sub);
  unsigned cmask = 0xffffu;  // searched cells
  if (!kFull) {
    cmask = 0u;
    if (((m - t.m_lo) & (Ls - 1)) < t.m_len) {
#pragma unroll
      for (int c = 0; c < 16; ++c)
        if ((((bitrev5(c) >> 1) - t.q_lo) & 15) < t.q_len) cmask |= 1u << c;
    }
  }
  unsigned long long *const keys = t.keys + ((size_t)sd.x * t.n_dm + sd.y) * t.S_tot;
  const unsigned kmask = 0xfffffff0u;
  // maximum of the segment of level e ending at AP i of the tile, merged into the series
  auto emit = [&](const int e, const int i, const float2(&g)[16]) {
    const int w = t.emit_w[e], i0 = i - (1 << e) + 1;
    if (w < 0 || i >= n_ap || i0 < 0 || i0 >= t.TT) return;  // uniform across the warp
    unsigned k[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      k[c] = cell_key<kFull>(g[c], bitrev5(c) >> 1, 0, kmask);
      if (!kFull) k[c] = (cmask >> c) & 1u ? k[c] : 0u;
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) k[c] = __vimax3_u32(k[c], k[c + 5], k[c + 10]);
    const unsigned key = __vimax3_u32(__vimax3_u32(k[0], k[1], k[2]), __vimax3_u32(k[3], k[4], k[15]), 0u);
    const unsigned wmax = __reduce_max_sync(0xffffffffu, key);
    const unsigned pw = wmax & (kFull ? ~15u : ~63u);
    if (key == wmax && pw != 0u) {  // tied lanes share the column; the merge keeps the lowest row
      const unsigned q = kFull ? 15u - (wmax & 15u) : (32u - (wmax & 63u)) >> 1;
      const unsigned idx = (unsigned)m * 16u + q;
      // windows of 2^e APs start every 2^(e-1) APs (every AP for e = 0)
      atomicMax(keys + t.win_off[w] + ((kb + i0) >> (e > 0 ? e - 1 : 0)), ((unsigned long long)pw << 32) | (unsigned long long)(~idx));
    }
  };
  // G_1 of AP q of the step: the slots fold into the even half of a 32-point DIF (unit twiddles)
  auto one = [&](const int q, float2(&g)[16]) {
    const float2 unit = make_float2(1.f, -0.f);
#pragma unroll
    for (int p = 0; p < kPairs; ++p) {
      const float4 y = yr[q * kYAp + p * pair_stride(Ls)];
      g[2 * p] = cfma(make_float2(0.f, 0.f), make_float2(y.x, y.y), unit);
      g[2 * p + 1] = cfma(make_float2(0.f, 0.f), make_float2(y.z, y.w), unit);
    }
    fft16_dif_low(g);
  };

  float2 ga[16], gb[16], h2[16];  // G_1 of two consecutive APs, G_2 of the last odd AP
  float2 deep[kDeep16][16];       // first halves of levels 3 to 6 (local memory)
#pragma unroll
  for (int c = 0; c < 16; ++c) ga[c] = gb[c] = h2[c] = make_float2(0.f, 0.f);
  for (int e = 0; e < kDeep16; ++e)
    for (int c = 0; c < 16; ++c) deep[e][c] = make_float2(0.f, 0.f);

  for (int step = 0; step < n_step; ++step) {
    if (task) {
      float2 A[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) A[i] = make_float2(0.f, 0.f);
      for (int j1 = 0; j1 < a.J1; ++j1) {
#pragma unroll
        for (int j2 = 0; j2 < 32; j2 += 2) {
          const float4 x = *reinterpret_cast<const float4 *>(xr + j1 * 32 + j2);
          const float4 w = *reinterpret_cast<const float4 *>(wr + j1 * 32 + j2);
          A[j2] = cfma(A[j2], make_float2(x.x, x.y), make_float2(w.x, w.y));
          A[j2 + 1] = cfma(A[j2 + 1], make_float2(x.z, x.w), make_float2(w.z, w.w));
        }
      }
      fft32_dif(A);
#pragma unroll
      for (int i = 0; i < 32; ++i) yw[2 * kPS * bitrev5(i)] = A[i];
    }
    __syncthreads();
    const bool more = step + 1 < n_step;
    const int i = step * kStep16;
    float2 v[kPart], acc[16];
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int k = i + 2 * half;
      // even AP: levels 0 and 1
      if (more) load(step + 1, 2 * half, v);
      one(2 * half, ga);
      emit(0, k, ga);
      if (t.nlev >= 1) {
#pragma unroll
        for (int c = 0; c < 16; ++c) acc[c] = cadd(gb[c], ga[c]);
        emit(1, k, acc);
      }
      if (more) {
        keep(2 * half, v);
        load(step + 1, 2 * half + 1, v);
      }
      // odd AP: levels 0, 1 and 2
      one(2 * half + 1, gb);
      emit(0, k + 1, gb);
      if (t.nlev >= 1) {
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const float2 g = cadd(ga[c], gb[c]);
          acc[c] = cadd(h2[c], g);
          h2[c] = g;
        }
        emit(1, k + 1, h2);
        if (t.nlev >= 2) emit(2, k + 1, acc);
      }
      if (more) keep(2 * half + 1, v);
    }
    // levels 3 and up close at every fourth AP and rarer
    const int E = min(t.nlev, __ffs(i + kStep16));
    for (int e = 3; e <= E; ++e) {
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const float2 g = acc[c];
        acc[c] = cadd(deep[e - 3][c], g);
        deep[e - 3][c] = g;
      }
      emit(e, i + 3, acc);
    }
    __syncthreads();
  }
}

void set_tree16_constants() { upload_w32(); }

// One thread per row, eight slots (so channels at distinct g_n < 8), one SBD task per thread at most,
// 16 points of a step per thread; offsets within the tiles of a CTA in 32 bits.
bool tree16_supported(int Ls, int Lm, int N, int J, int s16, const int *g, int T) {
  if (Lm != 16 || (Ls != 32 && Ls != 64 && Ls != 128) || J > Ls || s16 != 1 || N > kSlots16 || N * J > 4 * Ls) return false;
  for (int n = 0; n < N; ++n)
    if (g[n] >= kSlots16) return false;
  return ((long long)T + 1) * N * J < (1LL << 31) && tree16_smem(Ls, N, (J + 31) / 32) <= max_smem_optin();
}

// Time tile: the largest that still gives kWaves16 rounds of CTAs (3 per SM); every tile repeats up to
// 2^nlev - 1 APs of the next one, so no less than 128.
constexpr int kWaves16 = 4;
int tree16_tile(int Ls, int T, long long n_series) {
  int TT = 1024;
  auto ctas = [&](int tt) { return n_series * (((T + tt - 1) / tt + kThreads16 / Ls - 1) / (kThreads16 / Ls)); };
  while (TT > 128 && ctas(TT) < (long long)kWaves16 * 3 * sm_count()) TT /= 2;
  return TT;
}

template <int kPS>
static cudaError_t launch_one16(const FitArgs &a, const TreeArgs &t, bool full, unsigned nb, size_t smem, cudaStream_t st) {
  auto kern = full ? k_tree16<kPS, true> : k_tree16<kPS, false>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<nb, kThreads16, smem, st>>>(a, t);
  return cudaGetLastError();
}

cudaError_t launch_tree16(const FitArgs &a, const TreeArgs &t, bool full, cudaStream_t st, int64_t *launches) {
  if (t.nlev > kMaxLev16 || t.TT % (1 << kMaxLev16) != 0) return cudaErrorInvalidValue;
  const int sub = kThreads16 / a.Ls;
  const long long nb = (long long)t.n_s * ((t.n_tt + sub - 1) / sub);
  if (nb <= 0) return cudaSuccess;
  if (nb > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  const size_t smem = tree16_smem(a.Ls, a.N, a.J1);
  cudaError_t e;
  switch (a.Ls) {
    case 32: e = launch_one16<1>(a, t, full, (unsigned)nb, smem, st); break;
    case 64: e = launch_one16<2>(a, t, full, (unsigned)nb, smem, st); break;
    case 128: e = launch_one16<4>(a, t, full, (unsigned)nb, smem, st); break;
    default: return cudaErrorInvalidValue;
  }
  ++*launches;
  return e;
}

}  // namespace frbx

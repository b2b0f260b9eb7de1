// Soft comb score and its adjoint (the differentiation pattern; the paper has
// no soft score, this builds on Eq. 6 and the comb idea of Eq. 8-10):
//
//   f_hq = h f0 + q delta,  h = 1..n_h, q = -Q..Q
//   G_hq = exp(-(q delta)^2 / (2 sigma_h^2)),  Z_h = sum_q G_hq
//   S    = sum_h w_h (sum_q G_hq P(f_hq) / Z_h) / B
//
// with P(f) = |F(f)|^2, F(f) = sum_k p_k exp(-2 pi i f (tau_k - tau_c)), B a
// constant background per pixel. The adjoint uses
// dP/df = 2 Re(conj(F) D), D = sum_k (-2 pi i (tau_k - tau_c)) p_k exp(...).
//
// One warp per pixel. For each harmonic h the phasor of event k at q = -Q is
// seeded exactly: the frequency, an integer number of micro-Hz (f0 and delta
// rounded to 1 uHz), is split into integer mHz (exact residue of a * tau mod 1e9,
// as in the grid NDFT) plus a sub-mHz remainder, and the constant window-centre
// phase is reduced exactly in integers (tau_c in half-microseconds); no FP64
// arithmetic runs per harmonic or per event. The next q values follow by
// rotation with e^{-2 pi i delta (tau - tau_c)}.
//
// The gradients with respect to w and sigma are sums of one signed term per
// pixel that cancel to a few thousandths of their absolute sum, so the order of
// every addition is fixed: events one per lane (strided by 32), then a butterfly
// over the lanes (16, 8, 4, 2, 1), frequencies and harmonics in sequence, pixels
// strided by 256 and a tree. What runs where follows that order:
//  * a pixel of at most 96 events (most have fewer than 16) with three or more
//    harmonics is taken by four groups of 8 lanes, a harmonic each; a lane takes
//    the events of lanes l, l + 16, l + 8, l + 24 one after the other and adds
//    them as the butterfly's first two steps would (beyond, the idle half of
//    the last harmonics' groups costs more than the shared reductions save);
//  * the last three steps halve the frequencies that a lane holds (7 exchanges
//    per component and eight frequencies instead of 24), so that lane i of eight
//    ends with frequencies i, i + 8, ... and squares them there. The backward pass
//    of more than nine frequencies reduces them one by one over the whole warp
//    instead: its 44 to 68 sums leave 16 warps per SM, and the halving's exchanges,
//    selections and broadcasts wait more than they save (60,000 pixels, 5 harmonics,
//    Q = 5: 1.42 ms halving, 1.23 so; 8 harmonics, Q = 8: 2.53 and 2.20);
//  * the weights G_hq and their sums depend on (h, q) alone: a table per block.
// Per-pixel gradient contributions to w and sigma are written to a workspace,
// one column each, and summed over pixels, so every output is deterministic.
#include <algorithm>

#include "ddhf_internal.cuh"

namespace ddhf {

namespace {

constexpr int kSoftMaxQ = 8;   // 2Q+1 <= 17 frequencies per harmonic
constexpr int kSoftMaxH = 8;
constexpr float kTwoPi = 6.28318530717958647692f;

struct SoftArgs {
  const uint32_t *ev;
  const uint32_t *offsets;
  const uint32_t *pixels;  // pixel keys
  int64_t n_px;
  const float *f0;
  const float *w;
  const float *sigma;
  const float *B;
  int n_h, Q;
  int64_t delta_uhz;       // evaluation step in micro-Hz
  float delta_hz;          // the same step in Hz
  int64_t tc2;             // 2 tau_c in half-microseconds (tau_c relative to the window start)
  float *S;                // forward output [n_px]
  const float *gS;         // backward input [n_px]
  float *g_f0;             // backward output [n_px]
  float *g_f;              // backward output [n_px][n_h][2Q+1], nullable
  float *part;             // backward workspace [2 n_h][n_px]
  uint64_t barrett;        // floor((2^64-1) / 1e9)
  int64_t npx;             // keys at or beyond it are skipped (DDHF_FLAG_INPUT)
  uint32_t *flags;
  uint32_t *cursor;        // next pixel to take (zeroed before each launch)
};

constexpr uint64_t kD9 = 1000000000ull;
// Events of a pixel up to which lane groups take a harmonic each. Forward and
// adjoint, 640x480 pixels of a textured scene / of Pareto noise, 6 harmonics,
// Q = 3: limit 32 1.11 / 2.48 ms, 96 0.97 / 2.39, 256 0.96 / 2.38, none 0.98 /
// up to a third more on the noise, whose longest pixels then run alone.
constexpr int kGroupMax = 96;

// Harmonic h's first frequency (q = -Q) of a pixel: integer mHz mod 1e9, the
// rest in Hz, and the phase f tau_c in cycles.
struct SoftFreq {
  uint64_t ai;
  float fr, cff;
};
__device__ __forceinline__ SoftFreq soft_freq(const SoftArgs &A, int h, int64_t f0u) {
  SoftFreq f;
  const int64_t fbu = (int64_t)h * f0u - (int64_t)A.Q * A.delta_uhz;
  int64_t fm = fbu / 1000, rem = fbu - fm * 1000;
  if (rem < 0) {
    rem += 1000;
    fm -= 1;
  }
  const uint64_t am = mod_barrett((uint64_t)(fm < 0 ? -fm : fm), kD9, A.barrett);
  f.ai = (fm < 0 && am != 0) ? kD9 - am : am;  // fm mod 1e9
  f.fr = __fmul_rn((float)(int)rem, 1e-6f);         // Hz, in [0, 1e-3)
  // constant phase f tau_c in cycles: (fbu * tc2 / 2e12) mod 1, exactly in
  // integers (fbu mod 2e12 < 2^41, tc2 < 2^21)
  const int64_t P2 = 2000000000000ll;
  int64_t fmod2 = fbu % P2;
  if (fmod2 < 0) fmod2 += P2;
  const int64_t cm = (int64_t)(((uint64_t)fmod2 * (uint64_t)A.tc2) % (uint64_t)P2);
  f.cff = __fmul_rn((float)cm, 5e-13f);
  return f;
}

// Phasor of event word wv at q = -Q (its polarity's sign on it), the step to the
// next q and 2 pi (tau - tau_c).
__device__ __forceinline__ void soft_event(const SoftArgs &A, const SoftFreq &f, uint32_t wv,
                                           float2 &z, float2 &u, float &wtt) {
  const uint64_t tau = wv & 0x7fffffffu;
  const uint64_t r = mod_barrett(f.ai * tau, kD9, A.barrett);
  float x = __fmul_rn((float)(uint32_t)r, 1e-9f);  // r < 1e9, tau < 2^31: 32-bit
  x = __fadd_rn(x, __fmul_rn(__fmul_rn(f.fr, (float)(uint32_t)tau), 1e-6f));
  x = __fsub_rn(x, f.cff);
  x = __fsub_rn(x, rintf(x));  // [-0.5, 0.5] cycles
  float sn, cs;
  sincospi_reduced(2.f * x, sn, cs);
  z.x = __uint_as_float(__float_as_uint(cs) ^ (wv & kSignBit));
  z.y = __uint_as_float(__float_as_uint(-sn) ^ (wv & kSignBit));
  // 2 tau - 2 tau_c fits 32 bits and a sign (a 64-bit conversion would run on
  // the FP64 pipe)
  const int64_t d2 = (int64_t)(2 * tau) - A.tc2;
  const float da = (float)(uint32_t)(d2 < 0 ? -d2 : d2);
  const float tt = __fmul_rn(d2 < 0 ? -da : da, 0.5e-6f);  // s
  float ss, sc;
  float xs = __fmul_rn(A.delta_hz, tt);  // cycles, folded to [-1/2, 1/2]
  xs = __fsub_rn(xs, rintf(xs));
  sincospi_reduced(2.f * xs, ss, sc);
  u = make_float2(sc, -ss);
  wtt = kTwoPi * tt;
}

// Events l, l + 32, ... of a pixel (one lane of the warp-wide order) into x.
template <int KQ, bool BWD>
__device__ __forceinline__ void soft_lane(const SoftArgs &A, const SoftFreq &f, const uint32_t *ev,
                                          int l, int cnt, int nq, float (&x)[BWD ? 4 : 2][KQ]) {
#pragma unroll 1
  for (int k = l; k < cnt; k += 32) {
    float2 z, u;
    float wtt;
    soft_event(A, f, ev[k], z, u, wtt);
#pragma unroll
    for (int q = 0; q < KQ; ++q) {
      if (q < nq) {
        x[0][q] += z.x;
        x[1][q] += z.y;
        if constexpr (BWD) {
          x[2][q] = __fmaf_rn(wtt, z.y, x[2][q]);  // D += -2 pi i (tau - tau_c) z
          x[3][q] = __fmaf_rn(-wtt, z.x, x[3][q]);
        }
        z = cmul(z, u);
      }
    }
  }
}

// NJ blocks of eight frequencies and EX = 1 more, 8 NJ + EX >= 2Q+1: 9 and 17
// frequencies with a whole block for the last one padded a third of the work
// away (Q = 8, 6 harmonics: 1.12 ms, 0.97 so; one butterfly per frequency 0.98).
// Bound by instruction issue (76 %). Measured on 153,600 pixels of a 640x480
// window (6 harmonics, Q = 3): forward 0.870 -> 0.378 ms, both ways with the
// gradient sums 2.29 -> 0.96 ms, the same bits.
template <int NJ, int EX, bool BWD>
__global__ void __launch_bounds__(256) k_softcomb(SoftArgs A) {
  constexpr int kC = BWD ? 4 : 2;  // components: F re, im, and D re, im for the backward pass
  constexpr int kQ = 8 * NJ + EX;
  // two sets of sums fit the registers
  constexpr bool kGroups = kC * kQ <= 32;
  constexpr bool kHalve = !BWD || NJ == 1;
  __shared__ float sG[kSoftMaxH][kQ];             // G_hq, 0 for q >= 2Q+1
  __shared__ float sZ[kSoftMaxH], sE[kSoftMaxH];  // Z_h, sum_q G qd^2
  const int lane = threadIdx.x & 31;
  const int nq = 2 * A.Q + 1;
  for (int i = threadIdx.x; i < A.n_h * kQ; i += blockDim.x) {
    const int h = i / kQ, q = i % kQ;
    const float sgm = A.sigma[h], qd = __fmul_rn((float)(q - A.Q), A.delta_hz);
    sG[h][q] = q < nq ? expf(-(qd * qd) / (2.f * sgm * sgm)) : 0.f;
  }
  __syncthreads();
  if (threadIdx.x < A.n_h) {
    float Z = 0.f, Ec = 0.f;
    for (int q = 0; q < nq; ++q) {
      const float G = sG[threadIdx.x][q];
      const float qd = __fmul_rn((float)(q - A.Q), A.delta_hz);
      Z += G;
      Ec = __fmaf_rn(__fmul_rn(G, qd), qd, Ec);
    }
    sZ[threadIdx.x] = Z;
    sE[threadIdx.x] = Ec;
  }
  __syncthreads();
  // pixels are taken one at a time from a counter (a pixel's cost grows with
  // its events, which are heavy-tailed); the next index is fetched while the
  // current pixel is processed
  uint32_t next = 0;
  if (lane == 0) next = atomicAdd(A.cursor, 1u);
  for (int64_t a = __shfl_sync(0xffffffffu, next, 0); a < A.n_px;
       a = __shfl_sync(0xffffffffu, next, 0)) {
    if (lane == 0) next = atomicAdd(A.cursor, 1u);
    const uint32_t key = A.pixels[a];
    // a key off the sensor has no events: S = 0, zero gradients, flagged
    const bool key_ok = (int64_t)key < A.npx;
    if (!key_ok && lane == 0) atomicOr(A.flags, DDHF_FLAG_INPUT);
    const uint32_t o0 = key_ok ? A.offsets[key] : 0u;
    const int cnt = key_ok ? (int)(A.offsets[key + 1] - o0) : 0;
    // f0 in integer micro-Hz: every frequency h f0 + q delta is then an exact
    // integer number of micro-Hz
    const int64_t f0u = __double2ll_rn((double)A.f0[a] * 1e6);
    const float Bv = A.B[a];
    const float gs = BWD ? A.gS[a] : 0.f;
    const bool grouped = kGroups && A.n_h >= 3 && cnt <= kGroupMax;  // a harmonic per 8 lanes
    const int hg = grouped ? lane >> 3 : 0, groups = grouped ? 4 : 1;
    float S = 0.f, g0 = 0.f;
    for (int h0 = 0; h0 < A.n_h; h0 += groups) {
      const int h = min(h0 + hg, A.n_h - 1);  // harmonic h + 1
      const SoftFreq f = soft_freq(A, h + 1, f0u);
      float x[kC][kQ];
#pragma unroll
      for (int c = 0; c < kC; ++c)
#pragma unroll
        for (int q = 0; q < kQ; ++q) x[c][q] = 0.f;
      if (grouped) {
        if constexpr (kGroups) {
#pragma unroll 1
          for (int half = 0; half < 2 && 8 * half < cnt; ++half) {
            float t[kC][kQ];  // lanes l + 8 half and l + 8 half + 16 of the butterfly
#pragma unroll
            for (int p = 0; p < 2; ++p) {
              float y[kC][kQ];
#pragma unroll
              for (int c = 0; c < kC; ++c)
#pragma unroll
                for (int q = 0; q < kQ; ++q) y[c][q] = 0.f;
              soft_lane<kQ, BWD>(A, f, A.ev + o0, (lane & 7) + 8 * half + 16 * p, cnt, nq, y);
#pragma unroll
              for (int c = 0; c < kC; ++c)
#pragma unroll
                for (int q = 0; q < kQ; ++q) t[c][q] = p == 0 ? y[c][q] : t[c][q] + y[c][q];
            }
#pragma unroll
            for (int c = 0; c < kC; ++c)
#pragma unroll
              for (int q = 0; q < kQ; ++q) x[c][q] += t[c][q];
          }
        }
      } else {
        soft_lane<kQ, BWD>(A, f, A.ev + o0, lane, cnt, nq, x);
        if constexpr (kHalve) {
#pragma unroll 1
          for (int o = 16; o >= 8; o >>= 1)
#pragma unroll
            for (int c = 0; c < kC; ++c)
#pragma unroll
              for (int q = 0; q < kQ; ++q)
                if (q < nq) x[c][q] += __shfl_xor_sync(0xffffffffu, x[c][q], o);
        } else {
#pragma unroll
          for (int q = 0; q < kQ; ++q)
            if (q < nq)
#pragma unroll
              for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int c = 0; c < kC; ++c)
                  x[c][q] += __shfl_xor_sync(0xffffffffu, x[c][q], o);
        }
      }
      // the last three steps, halving: lane i of eight gets frequencies i, i + 8, ...
      float y[kC][NJ];
      if constexpr (kHalve)
#pragma unroll
      for (int c = 0; c < kC; ++c)
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
          float v[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) v[i] = x[c][8 * j + i];
#pragma unroll
          for (int o = 4; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < o; ++i) {
              const bool up = (lane & o) != 0;
              const float send = up ? v[i] : v[i + o], keep = up ? v[i + o] : v[i];
              v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
          y[c][j] = v[0];
        }
      // the frequency beyond the blocks: whole, in every lane
      if constexpr (kHalve && EX != 0)
#pragma unroll
        for (int o = 4; o > 0; o >>= 1)
#pragma unroll
          for (int c = 0; c < kC; ++c)
            x[c][8 * NJ] += __shfl_xor_sync(0xffffffffu, x[c][8 * NJ], o);
      // of the lane's own frequencies, or (not kHalve) of all
      constexpr int kP = kHalve ? NJ + EX : kQ;
      float P[kP], Pd[kP];
#pragma unroll
      for (int j = 0; j < kP; ++j) {
        float v[kC];
#pragma unroll
        for (int c = 0; c < kC; ++c)
          v[c] = !kHalve ? x[c][j] : j < NJ ? y[c][j < NJ ? j : 0] : x[c][kQ - 1];
        P[j] = v[0] * v[0] + v[1] * v[1];
        if constexpr (BWD) Pd[j] = 2.f * (v[0] * v[2] + v[1] * v[3]);
      }
      // sums over q, in order, by every lane of the group
      const float wh = A.w[h], Z = sZ[h];
      float Ac = 0.f, Ad = 0.f, Cc = 0.f;
#pragma unroll
      for (int q = 0; q < kQ; ++q) {
        const int src = (lane & 24) + (q & 7);
        float Pq = P[kHalve ? q / 8 : q], Pdq = BWD ? Pd[kHalve ? q / 8 : q] : 0.f;
        if (kHalve && q < 8 * NJ) {
          Pq = __shfl_sync(0xffffffffu, Pq, src);
          if constexpr (BWD) Pdq = __shfl_sync(0xffffffffu, Pdq, src);
        }
        if (q < nq) {
          const float G = sG[h][q];
          Ac += G * Pq;
          if constexpr (BWD) {
            const float qd = __fmul_rn((float)(q - A.Q), A.delta_hz);
            Ad += G * Pdq;
            Cc += G * Pq * qd * qd;
          }
        }
      }
      const bool h_ok = h0 + hg < A.n_h;
      const float sgm = BWD ? A.sigma[h] : 0.f;
      if constexpr (BWD) {
        if (A.g_f && h_ok && (grouped || !kHalve || lane < 8)) {
          // per evaluation frequency: g dS/df_hq = g w_h G_hq P'(f_hq) / (Z_h B)
#pragma unroll
          for (int j = 0; j < kP; ++j) {
            const int q = kHalve ? 8 * j + (lane & 7) : j;
            // of the frequency beyond the blocks, lane 0 alone
            if (q < nq && (kHalve || lane == q))
              A.g_f[(a * A.n_h + h) * (int64_t)nq + q] = gs * (wh * sG[h][q] * Pd[j] / (Z * Bv));
          }
        }
        if (h_ok && (grouped ? (lane & 7) == 0 : lane == 0)) {
          A.part[(int64_t)h * A.n_px + a] = gs * ((Ac / Z) / Bv);
          A.part[(int64_t)(A.n_h + h) * A.n_px + a] =
              gs * (wh / (Bv * sgm * sgm * sgm) * (Cc / Z - (Ac / Z) * (sE[h] / Z)));
        }
      }
      // harmonics in order
      const float Sh = wh * (Ac / Z) / Bv;
      const float gh = BWD ? wh * (float)(h + 1) * (Ad / Z) / Bv : 0.f;
      for (int i = 0; i < groups && h0 + i < A.n_h; ++i) {
        S += __shfl_sync(0xffffffffu, Sh, 8 * i);
        if constexpr (BWD) g0 += __shfl_sync(0xffffffffu, gh, 8 * i);
      }
    }
    if (lane == 0) {
      if (BWD) A.g_f0[a] = gs * g0;
      else A.S[a] = S;
    }
  }
}

// out[c] = sum_a part[c][a] for c < ncol, fixed order: rows strided by 256 per
// thread, then a tree (out: columns below half, out2: the others). 16 loads are
// in flight per thread: the additions are a serial chain.
__global__ void __launch_bounds__(256) k_col_sum(const float *part, int64_t n_rows, float *out,
                                                 float *out2, int half) {
  __shared__ float sh[256];
  const int c = blockIdx.x;
  const float *col = part + (int64_t)c * n_rows;
  float s = 0.f;
  int64_t a = threadIdx.x;
  for (; a + 15 * 256 < n_rows; a += 16 * 256) {
    float v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = col[a + 256 * i];
#pragma unroll
    for (int i = 0; i < 16; ++i) s += v[i];
  }
  for (; a < n_rows; a += 256) s += col[a];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int st = 128; st > 0; st >>= 1) {
    if ((int)threadIdx.x < st) sh[threadIdx.x] += sh[threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    if (c < half) out[c] = sh[0];
    else out2[c - half] = sh[0];
  }
}

template <int NJ, int EX>
cudaError_t launch_soft(const SoftArgs &A, bool bwd, int blocks, cudaStream_t s) {
  if (bwd) k_softcomb<NJ, EX, true><<<blocks, 256, 0, s>>>(A);
  else k_softcomb<NJ, EX, false><<<blocks, 256, 0, s>>>(A);
  return cudaGetLastError();
}

// Median of each spectrum row (the mean of the two middle values for an even
// count), exact, one warp per row: the two middle ranks are selected by an
// 8-bit radix select over the (value, index) keys.
__device__ uint64_t select_key(const float *Pr, int N, int R, uint32_t *hist) {
  const int lane = threadIdx.x & 31;
  uint64_t prefix = 0, pmask = 0;
  int r = R;
  for (int shift = 40; shift >= 0; shift -= 8) {
    for (int i = lane; i < 256; i += 32) hist[i] = 0;
    __syncwarp();
    for (int j = lane; j < N; j += 32) {
      const uint64_t key = ((uint64_t)__float_as_uint(Pr[j]) << 16) | (uint32_t)j;
      if ((key & pmask) == prefix) atomicAdd(&hist[(key >> shift) & 255], 1u);
    }
    __syncwarp();
    uint32_t hv[8], s = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      hv[q] = hist[lane * 8 + q];
      s += hv[q];
    }
    uint32_t inc = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t u = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += u;
    }
    const uint32_t ex = inc - s;
    const bool own = (uint32_t)r >= ex && (uint32_t)r < ex + s;
    int src = __ffs(__ballot_sync(0xffffffffu, own)) - 1;
    src = src < 0 ? 0 : src;
    int g = 0;
    uint32_t below = 0;
    if (lane == src) {
      uint32_t c = ex;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if ((uint32_t)r >= c && (uint32_t)r < c + hv[q]) {
          g = lane * 8 + q;
          below = c;
        }
        c += hv[q];
      }
    }
    g = __shfl_sync(0xffffffffu, g, src);
    below = __shfl_sync(0xffffffffu, below, src);
    prefix |= (uint64_t)g << shift;
    pmask |= (uint64_t)0xFF << shift;
    r -= (int)below;
    __syncwarp();
  }
  return prefix;
}

__global__ void k_row_median(const float *P, int64_t rows, int N, float *med) {
  __shared__ uint32_t hist[8][256];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t a = wid; a < rows; a += nwarps) {
    const float *Pr = P + a * N;
    const uint64_t k1 = select_key(Pr, N, (N - 1) / 2, hist[warp]);
    float v = __uint_as_float((uint32_t)(k1 >> 16));
    if ((N & 1) == 0) {
      const uint64_t k2 = select_key(Pr, N, N / 2, hist[warp]);
      v = __fmul_rn(__fadd_rn(v, __uint_as_float((uint32_t)(k2 >> 16))), 0.5f);
    }
    if (lane == 0) med[a] = v;
  }
}

}  // namespace
}  // namespace ddhf

using namespace ddhf;

extern "C" ddhf_status ddhf_softcomb(ddhf_ctx *h, int64_t n_px, const uint32_t *pixels,
                                     const float *f0, int32_t n_h, int32_t Q, double delta_hz,
                                     double tau_c_us, const float *w, const float *sigma,
                                     const float *B, float *S, const float *grad_S,
                                     float *grad_f0, float *grad_w, float *grad_sigma,
                                     float *grad_f, ddhf_stream stream) {
  if (!h) return DDHF_ERR_INVALID_ARG;
  Ctx *c = &h->c;
  if (!c->binned) {
    c->last_error = "no binned window";
    return DDHF_ERR_STATE;
  }
  if (n_px < 0 || n_px > c->npx || n_h < 1 || n_h > kSoftMaxH || Q < 0 || Q > kSoftMaxQ ||
      !(delta_hz >= 1e-6) || !(delta_hz < 1e6) || !(tau_c_us >= 0.0) ||
      !(tau_c_us < (double)(1 << 20)) ||
      (n_px > 0 && (!pixels || !f0 || !w || !sigma || !B))) {
    c->last_error = "softcomb: bad arguments";
    return DDHF_ERR_INVALID_ARG;
  }
  const bool bwd = grad_S != nullptr;
  if (!bwd && !S) {
    c->last_error = "softcomb: need S (forward) or grad_S (backward)";
    return DDHF_ERR_INVALID_ARG;
  }
  if (bwd && (!grad_f0 || !grad_w || !grad_sigma)) {
    c->last_error = "softcomb: backward needs grad_f0, grad_w, grad_sigma";
    return DDHF_ERR_INVALID_ARG;
  }
  if (n_px == 0) return DDHF_OK;
  cudaStream_t s = (cudaStream_t)stream;
  c->last_stream = s;
  SoftArgs A;
  A.ev = c->slots[0].ev;
  A.offsets = c->slots[0].offsets;
  A.pixels = pixels;
  A.n_px = n_px;
  A.f0 = f0;
  A.w = w;
  A.sigma = sigma;
  A.B = B;
  A.n_h = n_h;
  A.Q = Q;
  A.delta_uhz = llround(delta_hz * 1e6);
  A.delta_hz = (float)delta_hz;
  A.tc2 = llround(2.0 * tau_c_us);
  A.S = S;
  A.gS = grad_S;
  A.g_f0 = grad_f0;
  A.g_f = bwd ? grad_f : nullptr;
  A.part = c->soft_part;  // [2 n_h][n_px]
  A.barrett = ~0ull / 1000000000ull;
  A.npx = c->npx;
  A.flags = c->flags;
  A.cursor = c->qctl + 4;
  DDHF_CUDA_TRY(c, cudaMemsetAsync(A.cursor, 0, sizeof(uint32_t), s));
  const int blocks = (int)std::min<int64_t>(ceil_div(n_px, 8), (int64_t)c->num_sms * 16);
  const int nq = 2 * Q + 1;
  if (nq <= 8) DDHF_CUDA_TRY(c, (launch_soft<1, 0>(A, bwd, blocks, s)));
  else if (nq == 9) DDHF_CUDA_TRY(c, (launch_soft<1, 1>(A, bwd, blocks, s)));
  else if (nq <= 16) DDHF_CUDA_TRY(c, (launch_soft<2, 0>(A, bwd, blocks, s)));
  else DDHF_CUDA_TRY(c, (launch_soft<2, 1>(A, bwd, blocks, s)));
  if (bwd) k_col_sum<<<2 * n_h, 256, 0, s>>>(A.part, n_px, grad_w, grad_sigma, n_h);
  DDHF_CUDA_TRY(c, cudaGetLastError());
  return DDHF_OK;
}

extern "C" ddhf_status ddhf_spectrum_median(ddhf_ctx *h, const float *P, int64_t rows,
                                            float *median, ddhf_stream stream) {
  if (!h) return DDHF_ERR_INVALID_ARG;
  Ctx *c = &h->c;
  if (rows < 0 || (rows > 0 && (!P || !median))) {
    c->last_error = "spectrum_median: bad arguments";
    return DDHF_ERR_INVALID_ARG;
  }
  if (rows == 0) return DDHF_OK;
  cudaStream_t s = (cudaStream_t)stream;
  c->last_stream = s;
  const int blocks = (int)std::min<int64_t>(ceil_div(rows, 8), (int64_t)c->num_sms * 8);
  k_row_median<<<blocks, 256, 0, s>>>(P, rows, c->grid.n_bins, median);
  DDHF_CUDA_TRY(c, cudaGetLastError());
  return DDHF_OK;
}

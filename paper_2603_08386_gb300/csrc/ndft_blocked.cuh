// Per-pixel non-uniform DFT power (Sec. 3.3 Eq. 6, P_k = |F_k|^2) on the tensor
// cores: the persistent kernel of DDHF_FORM_BLOCKED, writing spectra or (fused)
// scoring them where they are (Eq. 7-11, comb.cuh).
//
// Bins j = 32 b + r. With the centre frequency of row b, a_c(b) = a0 + (32 b +
// 15.5) da, and s = r - 15.5 = +-(k + 1/2), k = 0..15,
//   F[32 b + r] = sum_e A_b(e) u_s(e),  A_b = p e^{-2 pi i a_c(b) tau / D},
//                                       u_s = e^{-2 pi i s da tau / D} = c_k -+ i d_k,
// and the sums over the events e of the four real products of (Re A, Im A) with
// (c_k, d_k) give both bins +-s:
//   F[+s] = (X1 - X2) + i (X3 + X4),  F[-s] = (X1 + X2) + i (X3 - X4),
//   X1 = sum Ar c, X2 = sum Ai d, X3 = sum Ai c, X4 = sum Ar d:
// two real multiply-adds per event and bin (a complex product needs three or
// four), as one real matrix product per pixel, [Ar; Ai] (2 rows per b) x events
// x [c d] (32 columns).
//
// The product runs on the tensor cores in FP32 accuracy: each factor x is split
// into two FP16 words, x = hi + lo + O(2^-22) (|x| <= 1, so the error is absolute
// and below the factor's own FP32 generation error), and one m16n8k16
// instruction takes 8 events as 16 K entries (hi and lo of A side by side), once
// against hi of B and once against lo: all four partial products, accumulated
// in FP32. A pixel's product is too small and its operands too private for
// tcgen05 (48 x 32 x a few tens of events, every pixel with operands of its own,
// so each 64-row tcgen05 step would read as many shared-memory bytes as it has
// multiply-adds to do): mma.sync takes its operands from registers and leaves
// every accumulator of a bin pair in the lane that squares it.
//
// Factors are generated for 32 events at a time, one lane per event, into shared
// memory: a column and a row phasor straight from their phases, the others by
// rotation away from them on both sides (at most 8 steps for the columns, 4 MT for
// the rows, each step a phasor straight from its phase too). Phases are fixed-point
// fractions of a turn: the frequency's fraction a / D mod 1, rounded to 2^-64, times
// tau < 2^31 (error below 2^-34 of a turn), cut to its top 32 bits (below 2^-32);
// the sine and cosine then take it as an FP32 number of at most 1/8 turn (below
// 2^-28). Measured error of the spectra
// against FP64 (2-norm over all pixels): 2.4e-7 at 2000 bins on 640x480 pixels,
// 4.0e-7 at 10,000 bins on 320x180 (the FP32 three-multiplication product
// before it, with its longer rotation chains: 8.1e-7 and 1.3e-6).
//
// Measured (one 1280x720 window of 19.9M events, 750 bins, default tuning):
// 2.58 -> 1.33 ms (issue 55 % at 16 warps per SM, tensor pipe 38 %, 920 warp
// instructions per pixel; bound by the latency of its dependent chains at the
// occupancy that 128 registers allow); 640x480 at 2000 bins 1.79 -> 0.82 ms,
// 320x180 at 10,000 bins 7.4 -> 2.7 ms, a sparse 1280x720 window (1.06M events)
// 190 -> 80 us.
//
// Bins whose frequency is a multiple of D (in practice bin 0 of a grid that
// starts at 0 Hz) have the phase 0 for every event: their power is the squared
// integer sum of the polarities, counted exactly (Eq. 7 takes the logarithm of
// it, and a sum of zero must be exactly zero).
//
// Who takes a pixel, by its event count n alone; up to 2047 events the order in
// which they are summed, too (from there on it also depends on the warps per block):
//   n < 256 (kTeamPixel)   one warp, group after group (unless the tuning's
//                          heavy_min lists it);
//   n >= 256, or listed    four sums over every fourth chunk of 32 events, added
//                          in order, by a team of four warps (or of two): one
//                          warp needs 1.6 us per chunk, so that a 1000-event
//                          pixel alone took 62 us, longer than the rest of a
//                          sparse window; by a team 19 us (threshold 256 / 512 /
//                          1024: dense 1280x720 spectra 1.38 / 1.38 / 1.41 ms, sparse
//                          84 / 92 / 119 us, 320x180 at 10,000 bins 2.68 / 2.79 / 2.98 ms);
//   n >= 2048 (kBigPixel)  (and heavy_min) a cluster of four blocks (fused, of two or
//                          one in more rounds too), one sum per warp, added in
//                          order through shared memory: 20,000 events are 156
//                          chunks per warp of a block.
// Big pixels first, then the listed ones, then the light. When several passes
// cover the bins, each (pixel, pass) of the first two is an item of its own.
#pragma once

#include <cooperative_groups.h>

#include <algorithm>

#include "comb.cuh"
#include "ddhf_internal.cuh"
#include "ndft_const.cuh"

namespace ddhf {
namespace blocked {

constexpr int kGenChunk = 32;  // events staged per warp, one lane each
constexpr int kGroup = 8;      // events per tensor-core step
constexpr int kShares = 4;     // shares of a big pixel: the blocks of its cluster

__device__ __forceinline__ void raise_flag(uint32_t *flags, uint32_t f) { atomicOr(flags, f); }

// e^{-2 pi i phi}, phi = f tau as a fraction of a turn (f in units of 2^-64).
__device__ __forceinline__ float2 phasor_of_turn(uint64_t f, uint32_t tau) {
  return phasor_of_turn32(__umulhi((uint32_t)f, tau) + (uint32_t)(f >> 32) * tau);
}

// Each element of v (|v| <= 1) as two FP16 values, hi in the low half of its
// word: hi is v rounded to a multiple of 2^-11 (exact in FP16), lo the rest
// (|lo| <= 2^-12) rounded to FP16.
__device__ __forceinline__ void split_half2(float2 v, uint32_t &wx, uint32_t &wy) {
  const float2 m = make_float2(6144.f, 6144.f), nm = make_float2(-6144.f, -6144.f);
  const float2 hi = __fadd2_rn(__fadd2_rn(v, m), nm);
  const float2 lo = __ffma2_rn(hi, make_float2(-1.f, -1.f), v);
  asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(wx) : "f"(lo.x), "f"(hi.x));
  asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(wy) : "f"(lo.y), "f"(hi.y));
}

// Two rotation chains in paired FP32 instructions (each element rounded as
// cmul rounds it): `up` steps by r, `dn` by its conjugate.
struct ChainPair {
  float2 x, y;          // (up, dn) real and imaginary parts
  float2 rx, ry, nry;   // (rx, rx), (ry, -ry), (-ry, ry)
  __device__ __forceinline__ ChainPair(float2 up, float2 dn, float2 r)
      : x(make_float2(up.x, dn.x)), y(make_float2(up.y, dn.y)), rx(make_float2(r.x, r.x)),
        ry(make_float2(r.y, -r.y)), nry(make_float2(-r.y, r.y)) {}
  __device__ __forceinline__ void step() {
    const float2 a = __fmul2_rn(y, nry), b = __fmul2_rn(y, rx);
    y = __ffma2_rn(x, ry, b);
    x = __ffma2_rn(x, rx, a);
  }
};

// Shared-memory record of one event's factors: the 32 words of B, word 8 c + g
// for lane group g (columns k = 4 (g / 2) + c, real part c_k for an even g,
// imaginary d_k for an odd one), then A's rows in order, Re and Im, and 32 bytes
// of padding: lane (g, t) of a step reads word 8 c + g and row 8 i + g of events
// t and t + 4, and with this stride no two lanes of a load share a bank. The
// words are loaded one and two at a time, straight into the register pairs that
// the tensor instruction takes: 16-byte loads cost 18-27 % more instructions in
// moves.
template <int MT>
struct Stage {
  static constexpr int kRows = 128;                   // byte offset of the rows
  static constexpr int kRec = 128 + 64 * MT + 32;     // bytes per event
  static constexpr int kBytes = kRec * kGenChunk;
};

__device__ __forceinline__ uint32_t lds32(uint32_t sa) {
  uint32_t x;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(x) : "r"(sa) : "memory");
  return x;
}
__device__ __forceinline__ void lds64(uint32_t sa, uint32_t &x, uint32_t &y) {
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(x), "=r"(y) : "r"(sa) : "memory");
}

// The factors of event word w (lane = event of the chunk) into the warp's
// staging area. Every lane writes, so that no slot holds anything but finite
// factors (a lane past the last event generates those of word 0).
template <int MT>
__device__ __forceinline__ void gen_chunk(uint32_t w, const NdftConst &nd, uint64_t f_row,
                                          unsigned char *stage) {
  const uint32_t tau = w & 0x7fffffffu, sg = w & kSignBit;
  unsigned char *rec = stage + (threadIdx.x & 31) * Stage<MT>::kRec;
  // columns: k = 8 exact, 9..15 and 7..0 by rotation
  {
    const float2 u = phasor_of_turn(nd.f_u, tau), k8 = phasor_of_turn(nd.f_k8, tau);
    ChainPair z(k8, cmul(k8, make_float2(u.x, -u.y)), u);
    uint4 *b = reinterpret_cast<uint4 *>(rec);
    uint32_t up[4][2], dn[4][2];  // columns 8 + c and 4 + c
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (i > 0) z.step();  // k = 8 + i and 7 - i
      uint32_t cu, cd, du, dd;
      split_half2(z.x, cu, cd);
      split_half2(z.y, du, dd);
      if (i < 4) {
        up[i][0] = cu, up[i][1] = du;
        dn[3 - i][0] = cd, dn[3 - i][1] = dd;
      } else {
        b[2 * (i - 4) + 1] = make_uint4(up[i - 4][0], up[i - 4][1], cu, du);
        b[2 * (7 - i)] = make_uint4(cd, dd, dn[7 - i][0], dn[7 - i][1]);
      }
    }
  }
  // rows: 4 MT exact (the polarity's sign on it), the others by rotation
  {
    const float2 v = phasor_of_turn(nd.f_v, tau);
    float2 s = phasor_of_turn(f_row, tau);
    s.x = __uint_as_float(__float_as_uint(s.x) ^ sg);
    s.y = __uint_as_float(__float_as_uint(s.y) ^ sg);
    ChainPair z(s, cmul(s, make_float2(v.x, -v.y)), v);
    uint4 *a = reinterpret_cast<uint4 *>(rec + Stage<MT>::kRows);  // two rows each
#pragma unroll
    for (int i = 0; i < 2 * MT; ++i) {
      uint32_t u[4], d[4];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        if (i + j > 0) z.step();  // rows 4 MT + 2 i + j and 4 MT - 1 - 2 i - j
        split_half2(z.x, u[2 * j], d[2 - 2 * j]);
        split_half2(z.y, u[2 * j + 1], d[3 - 2 * j]);
      }
      a[2 * MT + i] = make_uint4(u[0], u[1], u[2], u[3]);
      a[2 * MT - 1 - i] = make_uint4(d[0], d[1], d[2], d[3]);
    }
  }
}

// A lane's accumulators: x[i][q] = (X1, X4, X3, X2) of row 8 i + g and column
// pair k = 4 t + q (lane (g, t) = (lane / 4, lane % 4)): the C fragment of an
// m16n8k16 step whose rows g and g + 8 are Re and Im of A and whose columns 2 t
// and 2 t + 1 are c and d.
template <int MT>
struct Acc {
  float x[MT][4][4];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int c = 0; c < 4; ++c) x[i][q][c] = 0.f;
  }
  // Powers of the bins at +s (k = 4 t + q) and -s of row i.
  __device__ __forceinline__ void powers(int i, int q, float &pp, float &pm) const {
    const float *a = x[i][q];
    const float rp = __fsub_rn(a[0], a[3]), ip = __fadd_rn(a[2], a[1]);
    const float rm = __fadd_rn(a[0], a[3]), im = __fsub_rn(a[2], a[1]);
    pp = __fmaf_rn(rp, rp, __fmul_rn(ip, ip));
    pm = __fmaf_rn(rm, rm, __fmul_rn(im, im));
  }
};

// d = A B + c, an m16n8k16 step.
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1, const float (&c)[4]) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%10,%11,%12,%13};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c[0]), "f"(c[1]),
        "f"(c[2]), "f"(c[3]));
}

// Staged events q .. q + m - 1 (m <= 8, q + m <= 32) into the accumulators
// (FIRST: which take their values instead of adding them). A pixel's events
// enter in groups of 8 counted from its first one, whatever the chunk they were
// staged in, so its sums do not depend on how the work is split.
//
// A word of A against the same event's word of B gives hi hi + lo lo, against
// the word with its halves swapped hi lo + lo hi. The tensor core cuts its sums
// off instead of rounding them, so a long chain of steps through one accumulator
// drifts towards zero (1.5e-5 of the spectra at 2000 bins, 25 times the FP32
// product's error): each group is summed on its own (the small products first)
// and added to the accumulators in FP32.
template <int MT, bool FIRST>
__device__ __forceinline__ void mma_group(int q, int m, const unsigned char *stage, Acc<MT> &acc) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  int e0 = q + t, e1 = q + t + 4;
  if (m < kGroup) {  // a slot past the chunk
    e0 = min(e0, kGenChunk - 1);
    e1 = min(e1, kGenChunk - 1);
  }
  const uint32_t sa = (uint32_t)__cvta_generic_to_shared(stage);
  const uint32_t s0 = sa + e0 * Stage<MT>::kRec, s1 = sa + e1 * Stage<MT>::kRec;
  uint32_t w0[4], w1[4], a[MT][4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    w0[c] = lds32(s0 + 4 * g + 32 * c);
    w1[c] = lds32(s1 + 4 * g + 32 * c);
  }
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    lds64(s0 + 8 * g + Stage<MT>::kRows + 64 * i, a[i][0], a[i][1]);
    lds64(s1 + 8 * g + Stage<MT>::kRows + 64 * i, a[i][2], a[i][3]);
  }
  if (m < kGroup) {  // past the pixel's last event
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (t >= m) w0[c] = 0u;
      if (t + 4 >= m) w1[c] = 0u;
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const uint32_t x0 = __byte_perm(w0[c], 0u, 0x1032u), x1 = __byte_perm(w1[c], 0u, 0x1032u);
    float d[MT][4];
    const float zero[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < MT; ++i) mma16816(d[i], a[i], x0, x1, zero);
#pragma unroll
    for (int i = 0; i < MT; ++i) mma16816(FIRST ? acc.x[i][c] : d[i], a[i], w0[c], w1[c], d[i]);
    if (!FIRST) {
#pragma unroll
      for (int i = 0; i < MT; ++i) {
        float *x = acc.x[i][c];
#pragma unroll
        for (int k = 0; k < 4; k += 2) {
          const float2 r =
              __fadd2_rn(make_float2(x[k], x[k + 1]), make_float2(d[i][k], d[i][k + 1]));
          x[k] = r.x;
          x[k + 1] = r.y;
        }
      }
    }
  }
}

struct BlockedArgs {
  const SlotView *views;
  int slot0;                 // first slot of the light-pixel range
  int n_slots;
  int64_t npx;
  const uint64_t *heavy;     // heavy work items (slot << 32 | active index)
  const uint32_t *n_heavy;   // [0] heavy items, from the list's front, [1] big ones, from its back
  uint32_t heavy_cap;        // capacity of the heavy list
  uint32_t *cursors;         // [0] heavy cursor, [1] light cursor, [2] big cursor
  int N, nbr;                // bins, rows of 32 bins
  CombConst cc;
  float *P;                  // spectra (write mode), rows in active order of slot 0
  int64_t ld;                // row stride of P in floats (>= N)
  int vec_store;             // P and ld 16-byte aligned
  int64_t cap_px;
  int heavy_min;             // events from which the list holds a pixel
  int light_max;             // the light path takes pixels of fewer events (<= heavy_min)
  int skip_min;              // > 0: pixels with at least this many events are left to the
                             // hybrid grid path (their rows are written there)
  int warp_bytes;            // per-warp shared memory (bytes)
  int pw_offset;             // byte offset of the spectrum buffer inside a warp's area
  uint32_t *flags;
  int64_t ev_cap;            // events each slot's event array holds (CSR bound)
  NdftConst nd;
};

// Bins of [j_begin, j_end) whose phase is 0 for every event: the squared sum
// of the pixel's polarities, after the tile that holds them was written.
__device__ __forceinline__ void exact_bins(const BlockedArgs &A, int sum_p, int j_begin, int j_end,
                                           float *row) {
  if (A.nd.dc_first < 0 || A.nd.dc_first >= j_end) return;
  __syncwarp();
  const float p2 = __fmul_rn((float)sum_p, (float)sum_p);
  for (int j = A.nd.dc_first; j < j_end; j += A.nd.dc_step)
    if (j >= j_begin && (threadIdx.x & 31) == 0) row[j] = p2;
}

// Rows of 32 bins that a fused warp's spectrum takes: whole tiles, but single
// tiles only up to four rows (the scratch of 640 bins in 4-row steps fits eight
// warps of a block, 24 rows of it do not).
template <int MT>
__host__ __device__ inline int spectrum_rows(int nbr) {
  const int unit = MT == 1 ? 4 : 8 * MT;
  return (nbr + unit - 1) / unit * unit;
}

// Power of the lane's tile into Pw (row-major bins from row_base on, nbr rows).
template <int MT>
__device__ __forceinline__ void finalize_tile(const Acc<MT> &acc, float *Pw, int row_base,
                                              int nbr) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    float pp[4], pm[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) acc.powers(i, q, pp[q], pm[q]);
    if (MT == 1 && row_base + g >= nbr) return;  // beyond spectrum_rows
    float *row = Pw + (row_base + 8 * i + g) * 32;
    *reinterpret_cast<float4 *>(row + 16 + 4 * t) = make_float4(pp[0], pp[1], pp[2], pp[3]);
    *reinterpret_cast<float4 *>(row + 12 - 4 * t) = make_float4(pm[3], pm[2], pm[1], pm[0]);
  }
}

// Power of the lane's tile straight to spectrum row `prow` (bin rows from b0),
// by 16-byte stores when rows are 16-byte aligned; bins at or beyond N are not
// written.
template <int MT>
__device__ __forceinline__ void store_tile(const BlockedArgs &A, const Acc<MT> &acc, int64_t prow,
                                           int b0, int sum_p) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  float *dst = A.P + prow * A.ld;
  const int row = b0 + g, whole = A.vec_store ? A.N >> 5 : 0;  // rows below it: 16-byte stores
  float *up = dst + 32 * row + 16 + 4 * t, *dn = dst + 32 * row + 12 - 4 * t;
#pragma unroll
  for (int i = 0; i < MT; ++i) {
    float pv[2][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) acc.powers(i, q, pv[1][q], pv[0][3 - q]);
    if (row + 8 * i < whole) {
      *reinterpret_cast<float4 *>(up + 256 * i) = make_float4(pv[1][0], pv[1][1], pv[1][2], pv[1][3]);
      *reinterpret_cast<float4 *>(dn + 256 * i) = make_float4(pv[0][0], pv[0][1], pv[0][2], pv[0][3]);
    } else {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = 32 * (row + 8 * i) + (h ? 16 + 4 * t : 12 - 4 * t);
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (j + q < A.N) dst[j + q] = pv[h][q];
      }
    }
  }
  exact_bins(A, sum_p, 32 * b0, min(A.N, 32 * (b0 + 8 * MT)), dst);
}

// Events of a pixel in chunks chunk0, chunk0 + step, ... of 32 (warp w of a
// block takes chunks w, w + nw, ...); returns how many of them are negative.
template <int MT>
__device__ __forceinline__ int accumulate(const uint32_t *__restrict__ evp, int cnt, int chunk0,
                                          int step, const NdftConst &nd, uint64_t f_row,
                                          unsigned char *stage, Acc<MT> &acc) {
  const int lane = threadIdx.x & 31;
  int c0 = chunk0 * kGenChunk, neg = 0;
  uint32_t w = c0 + lane < cnt ? evp[c0 + lane] : 0u;
  for (; c0 < cnt; c0 += step * kGenChunk) {
    const int ne = min(kGenChunk, cnt - c0);
    gen_chunk<MT>(w, nd, f_row, stage);
    neg += __popc(__ballot_sync(0xffffffffu, (w & kSignBit) != 0));
    __syncwarp();
    const int c1 = c0 + step * kGenChunk;  // the next chunk's event word, loaded ahead
    w = c1 + lane < cnt ? evp[c1 + lane] : 0u;
    for (int q = 0; q < ne; q += kGroup) mma_group<MT, false>(q, min(kGroup, ne - q), stage, acc);
    __syncwarp();
  }
  return neg;
}

// One pixel's spectrum into Pw (all passes).
template <int MT>
__device__ __forceinline__ void pixel_spectrum_warp(const BlockedArgs &A, const uint32_t *evp,
                                                    int cnt, unsigned char *stage, float *Pw) {
  for (int b0 = 0, pass = 0; b0 < A.nbr; b0 += 8 * MT, ++pass) {
    Acc<MT> acc;
    acc.zero();
    const int neg = accumulate<MT>(evp, cnt, 0, 1, A.nd, A.nd.f_row[pass], stage, acc);
    finalize_tile<MT>(acc, Pw, b0, A.nbr);
    exact_bins(A, cnt - 2 * neg, 32 * b0, min(A.N, 32 * (b0 + 8 * MT)), Pw);
    __syncwarp();
  }
}

// Light pixels of one slot, spectra to global memory. A warp takes runs of
// `run` consecutive active pixels and, when their event lists follow one
// another in memory (the CSR order of the binning), streams the run's events
// through the 32-event factor chunks in that order: the factors of an event do
// not depend on its pixel, so one chunk serves the end of one pixel and the
// start of the next, and a pixel's tile is stored and cleared as soon as its
// last event is in. A pixel's groups of 8 events count from its first one; a
// group that does not lie in the staged chunk as a whole starts the next chunk
// (at most 7 events are generated again). Events of pixels outside the run's
// light set (heavy ones, pixels left to the hybrid path, inactive pixels) are
// skipped. Runs whose lists are not in order (caller-built lists) are streamed
// one pixel at a time. The run length is 16 pixels when there are at least
// eight such runs per warp of the grid, and halves (down to one pixel) until
// there are: on a sparse window the warps then share the pixels evenly instead
// of a few runs of heavy-tailed pixels setting the kernel's time. A pixel's
// events are accumulated in the same groups and order whatever the run length,
// so the spectra do not depend on it.
template <int MT>
__device__ __forceinline__ void light_stream(const BlockedArgs &A, unsigned char *stage) {
  const int lane = threadIdx.x & 31;
  const SlotView &v = A.views[A.slot0];
  const int64_t n_act = (int64_t)v.counters[2];
  const int64_t n_warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  int run = 16;
  while (run > 1 && (int64_t)run * n_warps * 8 > n_act) run >>= 1;
  for (;;) {
    uint32_t a0 = 0;
    if (lane == 0) a0 = atomicAdd(&A.cursors[1], (uint32_t)run);
    a0 = __shfl_sync(0xffffffffu, a0, 0);
    if ((int64_t)a0 >= n_act) break;
    // lane q < run: pixel a0 + q of the run, its event range and whether it is light
    const int64_t aq = (int64_t)a0 + lane;
    uint32_t q_lo = 0, q_hi = 0;
    bool q_ok = false;
    if (lane < run && aq < n_act) {
      const uint32_t key = v.active[aq];
      q_lo = v.offsets[key];
      q_hi = v.offsets[key + 1];
      const int cnt = (int)(q_hi - q_lo);
      q_ok = cnt < A.light_max && !(A.skip_min > 0 && cnt >= A.skip_min) &&
             ddhf_check((int64_t)q_hi <= A.ev_cap, A.flags);
      if (q_ok && aq >= A.cap_px) {
        raise_flag(A.flags, DDHF_FLAG_CAPACITY);
        q_ok = false;
      }
    }
    const uint32_t okm = __ballot_sync(0xffffffffu, q_ok);
    if (!okm) continue;
    // in order: every light pixel's list starts at or after the previous one's end
    const uint32_t lower = okm & lanemask_lt();
    const int prev = lower ? 31 - __clz(lower) : -1;
    const uint32_t prev_end = __shfl_sync(0xffffffffu, q_hi, prev < 0 ? 0 : prev);
    const bool bad = q_ok && (q_hi < q_lo || (prev >= 0 && q_lo < prev_end));
    const bool in_order = !__any_sync(0xffffffffu, bad);
    // the whole run at once, or (lists out of order) one pixel at a time
    for (uint32_t todo = okm; todo;) {
      const uint32_t sub = in_order ? todo : (todo & (0u - todo));
      todo &= ~sub;
      const uint32_t e_end = __shfl_sync(0xffffffffu, q_hi, 31 - __clz(sub));
      for (int b0 = 0, pass = 0; b0 < A.nbr; b0 += 8 * MT, ++pass) {
        // the staged chunk holds events [c0, c0 + 32) of the run (c0 = ~0: none
        // yet), words wc; wn: the 32 words after them; sgn: their signs
        uint32_t c0 = 0xffffffffu, wc = 0, wn = 0, sgn = 0;
        const bool has_dc = A.nd.dc_first >= 0 && A.nd.dc_first < 32 * (b0 + 8 * MT);
        for (uint32_t rem = sub; rem; rem &= rem - 1) {
          const int p = __ffs(rem) - 1;
          const uint32_t pe0 = __shfl_sync(0xffffffffu, q_lo, p);
          const uint32_t pe1 = __shfl_sync(0xffffffffu, q_hi, p);
          Acc<MT> acc;
          int neg = 0;
          // a step of its own for the first group saves the clearing and adding,
          // but costs registers: 834 against 867 us at 2000 bins (MT 4), 1.38
          // against 1.33 ms at 750 (MT 3)
          constexpr bool kFirst = MT == 4;
          if (!kFirst || pe0 >= pe1) acc.zero();
          for (uint32_t pos = pe0; pos < pe1; pos += kGroup) {
            const int m = (int)min((uint32_t)kGroup, pe1 - pos);
            uint32_t d = pos - c0;
            if (c0 == 0xffffffffu || d + m > (uint32_t)kGenChunk) {  // stage from pos on
              if (c0 != 0xffffffffu && d <= 32u) {  // among the words already loaded
                const uint32_t x = __shfl_sync(0xffffffffu, wc, (lane + d) & 31u);
                const uint32_t y = __shfl_sync(0xffffffffu, wn, (lane + d) & 31u);
                wc = lane + d < 32u ? x : y;
              } else {
                wc = pos + lane < e_end ? v.ev[pos + lane] : 0u;
              }
              c0 = pos;
              d = 0;
              __syncwarp();  // the previous chunk's products are done
              gen_chunk<MT>(wc, A.nd, A.nd.f_row[pass], stage);
              sgn = __ballot_sync(0xffffffffu, (wc & kSignBit) != 0);
              __syncwarp();
              wn = pos + 32u + lane < e_end ? v.ev[pos + 32u + lane] : 0u;
            }
            if (has_dc) neg += __popc((sgn >> d) & (0xffu >> (kGroup - m)));
            if (kFirst && pos == pe0) mma_group<MT, true>((int)d, m, stage, acc);
            else mma_group<MT, false>((int)d, m, stage, acc);
          }
          store_tile<MT>(A, acc, (int64_t)a0 + p, b0, (int)(pe1 - pe0) - 2 * neg);
        }
        __syncwarp();
      }
    }
  }
}

template <int NW>
__device__ __forceinline__ void store_scores(const BlockedArgs &A, const SlotView &v, int64_t a,
                                             uint32_t key, const CombOut &o) {
  if ((threadIdx.x & 31) == 0) {
    if (o.bad) atomicOr(A.flags, DDHF_FLAG_INTERNAL);
    v.log_sf[a] = o.log_sf;
    v.snr[a] = o.snr;
    v.f0[a] = o.w;
    v.mask[key] = o.rotor;
  }
}

// Barrier of a team of TW warps (team `id` of the block).
template <int TW>
__device__ __forceinline__ void team_sync(int id) {
  asm volatile("bar.sync %0, %1;" ::"r"(id + 1), "n"(32 * TW) : "memory");
}

// The four sums of a pixel's events (chunks r, r + 4, ... of 32), added in order
// by a team of TW warps (this one: warp tw), into the accumulators of warp 0;
// returns the number of negative events there. s_neg: four words per team.
template <int MT, int TW>
__device__ __forceinline__ int team_sum(const uint32_t *evp, int cnt, const NdftConst &nd,
                                        uint64_t f_row, unsigned char *stage, int warp_bytes,
                                        int tw, int id, int *s_neg, Acc<MT> &acc) {
  const int lane = threadIdx.x & 31;
  float *part = reinterpret_cast<float *>(stage);
  float tot[16 * MT];  // the sum so far, when the team takes several rounds
  int neg_tot = 0;
#pragma unroll 1
  for (int r0 = 0; r0 < 4; r0 += TW) {
    acc.zero();
    const int neg = accumulate<MT>(evp, cnt, r0 + tw, 4, nd, f_row, stage, acc);
    // partial sums of this warp -> its staging area, [row, column, component][lane]
#pragma unroll
    for (int i = 0; i < 16 * MT; ++i) part[i * 32 + lane] = acc.x[i / 16][(i / 4) % 4][i % 4];
    if (lane == 0) s_neg[tw] = neg;
    team_sync<TW>(id);
    if (tw == 0) {
      neg_tot += neg;
      if (r0 > 0)
#pragma unroll
        for (int i = 0; i < 16 * MT; ++i) {
          float &x = acc.x[i / 16][(i / 4) % 4][i % 4];
          x = __fadd_rn(tot[i], x);
        }
      for (int w2 = 1; w2 < TW; ++w2) {
        const float *op = reinterpret_cast<const float *>(stage + w2 * warp_bytes);
#pragma unroll
        for (int i = 0; i < 16 * MT; ++i) {
          float &x = acc.x[i / 16][(i / 4) % 4][i % 4];
          x = __fadd_rn(x, op[i * 32 + lane]);
        }
        neg_tot += s_neg[w2];
      }
      if (TW < 4)
#pragma unroll
        for (int i = 0; i < 16 * MT; ++i) tot[i] = acc.x[i / 16][(i / 4) % 4][i % 4];
    }
    team_sync<TW>(id);  // the partial sums have been read
  }
  return neg_tot;
}

// Warp 0 of a team or cluster: the finished sums of pass ps to the spectrum row,
// or to Pw (FUSED).
template <int MT, bool FUSED>
__device__ __forceinline__ void heavy_store(const BlockedArgs &A, const Acc<MT> &acc, int64_t a,
                                            int ps, int sum_p, float *Pw) {
  const int b0 = ps * 8 * MT;
  if (FUSED) {
    finalize_tile<MT>(acc, Pw, b0, A.nbr);
    exact_bins(A, sum_p, 32 * b0, min(A.N, 32 * (b0 + 8 * MT)), Pw);
  } else {
    store_tile<MT>(A, acc, a, b0, sum_p);
  }
  __syncwarp();
}

// An item of the heavy list: its active index, slot, events; false when the
// item is not this kernel's.
struct HeavyPixel {
  int64_t a;
  const SlotView *v;
  uint32_t key, o0;
  int cnt;
};
template <bool FUSED>
__device__ __forceinline__ bool heavy_pixel(const BlockedArgs &A, uint64_t it, HeavyPixel &h) {
  h.a = (int64_t)(uint32_t)it;
  h.v = &A.views[it >> 32];
  h.key = h.v->active[h.a];
  h.o0 = h.v->offsets[h.key];
  h.cnt = (int)(h.v->offsets[h.key + 1] - h.o0);
  if (A.skip_min > 0 && h.cnt >= A.skip_min) return false;
  if (!ddhf_check((int64_t)h.o0 + h.cnt <= A.ev_cap, A.flags)) return false;
  if (!FUSED && h.a >= A.cap_px) {
    raise_flag(A.flags, DDHF_FLAG_CAPACITY);
    return false;
  }
  return true;
}

// A listed pixel (pass >= 0: that pass of the bins alone, else all of them, and
// the pixel is scored, FUSED) by a team of TW warps. Out of line, so that its
// registers do not count against the light pixels' loop.
template <int MT, int NW, bool FUSED, int TW>
__device__ __noinline__ void team_item(const BlockedArgs &A, uint64_t it, int pass,
                                       unsigned char *stage, int tw, int id, int *s_neg) {
  HeavyPixel h;
  if (!heavy_pixel<FUSED>(A, it, h)) return;
  float *Pw = reinterpret_cast<float *>(stage + A.pw_offset);
  const int p0 = pass >= 0 ? pass : 0;
  const int p1 = pass >= 0 ? pass + 1 : (A.nbr + 8 * MT - 1) / (8 * MT);
  for (int ps = p0; ps < p1; ++ps) {
    Acc<MT> acc;
    const int neg = team_sum<MT, TW>(h.v->ev + h.o0, h.cnt, A.nd, A.nd.f_row[ps], stage,
                                     A.warp_bytes, tw, id, s_neg, acc);
    if (tw == 0) heavy_store<MT, FUSED>(A, acc, h.a, ps, h.cnt - 2 * neg, Pw);
  }
  if (FUSED && tw == 0) {
    CombOut o = comb_warp<NW>(Pw, A.cc, stage);
    store_scores<NW>(A, *h.v, h.a, h.key, o);
  }
}

// A pass of a big pixel by the four blocks of a cluster: warp w of block r takes
// chunks r nw + w, + 4 nw, ...; warp 0 of each block adds its warps' sums, that of the
// first block the other blocks'.
template <int MT>
__device__ __noinline__ void cluster_item(const BlockedArgs &A, uint64_t it, int pass,
                                          unsigned char *stage, int *s_neg) {
  namespace cg = cooperative_groups;
  const cg::cluster_group cluster = cg::this_cluster();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int blocks = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  HeavyPixel h;
  if (!heavy_pixel<false>(A, it, h)) return;  // the same answer in every block
  float *part = reinterpret_cast<float *>(stage);
  const int p0 = pass >= 0 ? pass : 0;
  const int p1 = pass >= 0 ? pass + 1 : (A.nbr + 8 * MT - 1) / (8 * MT);
  for (int ps = p0; ps < p1; ++ps) {
    Acc<MT> acc;
    acc.zero();
    int neg = accumulate<MT>(h.v->ev + h.o0, h.cnt, rank * nw + warp, blocks * nw, A.nd,
                             A.nd.f_row[ps], stage, acc);
#pragma unroll
    for (int i = 0; i < 16 * MT; ++i) part[i * 32 + lane] = acc.x[i / 16][(i / 4) % 4][i % 4];
    if (lane == 0) s_neg[warp] = neg;
    __syncthreads();
    if (warp == 0) {
      for (int w2 = 1; w2 < nw; ++w2) {
        const float *op = reinterpret_cast<const float *>(stage + w2 * A.warp_bytes);
#pragma unroll
        for (int i = 0; i < 16 * MT; ++i) {
          float &x = acc.x[i / 16][(i / 4) % 4][i % 4];
          x = __fadd_rn(x, op[i * 32 + lane]);
        }
        neg += s_neg[w2];
      }
      if (rank != 0) {
#pragma unroll
        for (int i = 0; i < 16 * MT; ++i) part[i * 32 + lane] = acc.x[i / 16][(i / 4) % 4][i % 4];
        if (lane == 0) s_neg[0] = neg;
      }
    }
    cluster.sync();
    if (warp == 0 && rank == 0) {
      for (int r = 1; r < blocks; ++r) {
        const float *op = cluster.map_shared_rank(part, r);
#pragma unroll
        for (int i = 0; i < 16 * MT; ++i) {
          float &x = acc.x[i / 16][(i / 4) % 4][i % 4];
          x = __fadd_rn(x, op[i * 32 + lane]);
        }
        neg += *cluster.map_shared_rank(s_neg, r);
      }
      heavy_store<MT, false>(A, acc, h.a, ps, h.cnt - 2 * neg, nullptr);
    }
    cluster.sync();  // the other blocks' sums have been read
  }
}

// All passes of a big pixel and its scores (FUSED), by a cluster of four blocks, or of
// two or one in rounds: four shares, added in the order of cluster_item. A form of
// its own: the sum kept between rounds spills (in cluster_item 320x180 pixels of
// 10,000 bins 2.84 -> 2.93 ms).
template <int MT, int NW>
__device__ __noinline__ void cluster_rounds(const BlockedArgs &A, uint64_t it,
                                            unsigned char *stage, int *s_neg) {
  namespace cg = cooperative_groups;
  const cg::cluster_group cluster = cg::this_cluster();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int blocks = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  HeavyPixel h;
  if (!heavy_pixel<true>(A, it, h)) return;  // the same answer in every block
  float *Pw = reinterpret_cast<float *>(stage + A.pw_offset);
  float *part = reinterpret_cast<float *>(stage);
  for (int ps = 0; ps < (A.nbr + 8 * MT - 1) / (8 * MT); ++ps) {
    float tot[16 * MT];  // the sum so far
    int neg_tot = 0;
#pragma unroll 1
    for (int r0 = 0; r0 < kShares; r0 += blocks) {
      Acc<MT> acc;
      acc.zero();
      int neg = accumulate<MT>(h.v->ev + h.o0, h.cnt, (r0 + rank) * nw + warp, kShares * nw, A.nd,
                               A.nd.f_row[ps], stage, acc);
#pragma unroll
      for (int i = 0; i < 16 * MT; ++i) part[i * 32 + lane] = acc.x[i / 16][(i / 4) % 4][i % 4];
      if (lane == 0) s_neg[warp] = neg;
      __syncthreads();
      if (warp == 0) {
        for (int w2 = 1; w2 < nw; ++w2) {
          const float *op = reinterpret_cast<const float *>(stage + w2 * A.warp_bytes);
#pragma unroll
          for (int i = 0; i < 16 * MT; ++i) {
            float &x = acc.x[i / 16][(i / 4) % 4][i % 4];
            x = __fadd_rn(x, op[i * 32 + lane]);
          }
          neg += s_neg[w2];
        }
        if (rank != 0) {
#pragma unroll
          for (int i = 0; i < 16 * MT; ++i)
            part[i * 32 + lane] = acc.x[i / 16][(i / 4) % 4][i % 4];
          if (lane == 0) s_neg[0] = neg;
        }
      }
      cluster.sync();
      if (warp == 0 && rank == 0) {
        neg_tot += neg;
        if (r0 > 0)
#pragma unroll
          for (int i = 0; i < 16 * MT; ++i) {
            float &x = acc.x[i / 16][(i / 4) % 4][i % 4];
            x = __fadd_rn(tot[i], x);
          }
        for (int r = 1; r < blocks; ++r) {
          const float *op = cluster.map_shared_rank(part, r);
#pragma unroll
          for (int i = 0; i < 16 * MT; ++i) {
            float &x = acc.x[i / 16][(i / 4) % 4][i % 4];
            x = __fadd_rn(x, op[i * 32 + lane]);
          }
          neg_tot += *cluster.map_shared_rank(s_neg, r);
        }
        if (r0 + blocks < kShares) {
#pragma unroll
          for (int i = 0; i < 16 * MT; ++i) tot[i] = acc.x[i / 16][(i / 4) % 4][i % 4];
        } else {
          heavy_store<MT, true>(A, acc, h.a, ps, h.cnt - 2 * neg_tot, Pw);
        }
      }
      cluster.sync();  // the other blocks' sums have been read
    }
  }
  if (warp == 0 && rank == 0) {
    CombOut o = comb_warp<NW>(Pw, A.cc, stage);
    store_scores<NW>(A, *h.v, h.a, h.key, o);
  }
}

// The listed pixels, item by item, by teams of TW warps.
template <int MT, int NW, bool FUSED, int TW>
__device__ __forceinline__ void team_loop(const BlockedArgs &A, uint32_t per_px,
                                          unsigned char *stage, uint32_t *s_item, int *s_neg) {
  const int warp = threadIdx.x >> 5, tw = warp % TW, id = warp / TW;
  const uint32_t n_heavy = min(A.n_heavy[0], A.heavy_cap);
  if (n_heavy == 0) return;
  for (;;) {
    if (tw == 0 && (threadIdx.x & 31) == 0) s_item[id] = atomicAdd(&A.cursors[0], 1u);
    team_sync<TW>(id);
    const uint32_t item = s_item[id];
    team_sync<TW>(id);
    if (item / per_px >= n_heavy) break;
    team_item<MT, NW, FUSED, TW>(A, A.heavy[item / per_px], FUSED ? -1 : (int)(item % per_px),
                                 stage, tw, id, s_neg + 4 * id);
  }
}

// Big pixels, one cluster each, then the other listed ones, a team of warps each.
template <int MT, int NW, bool FUSED>
__device__ __noinline__ void listed_pixels(const BlockedArgs &A, unsigned char *stage,
                                           uint32_t *s_item, int *s_neg) {
  namespace cg = cooperative_groups;
  // items of a pixel: its passes (a fused pixel is scored once all are in)
  const uint32_t per_px = FUSED ? 1u : (uint32_t)((A.nbr + 8 * MT - 1) / (8 * MT));
  const uint32_t n_big = min(A.n_heavy[1], A.heavy_cap);
  if (n_big > 0) {
    const cg::cluster_group cluster = cg::this_cluster();
    for (;;) {
      if (cluster.block_rank() == 0 && threadIdx.x == 0) s_item[0] = atomicAdd(&A.cursors[2], 1u);
      cluster.sync();
      const uint32_t item = *cluster.map_shared_rank(&s_item[0], 0);
      cluster.sync();
      if (item / per_px >= n_big) break;
      const uint64_t it = A.heavy[A.heavy_cap - 1 - item / per_px];
      if constexpr (FUSED) cluster_rounds<MT, NW>(A, it, stage, s_neg);
      else cluster_item<MT>(A, it, (int)(item % per_px), stage, s_neg);
    }
  }
  if (blockDim.x >= 128) team_loop<MT, NW, FUSED, 4>(A, per_px, stage, s_item, s_neg);
  else team_loop<MT, NW, FUSED, 2>(A, per_px, stage, s_item, s_neg);
  __syncwarp();
}

template <int MT, int NW, bool FUSED>
__global__ void __launch_bounds__(256, 2) k_blocked(const __grid_constant__ BlockedArgs A) {
  extern __shared__ float4 smem4[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char *stage = reinterpret_cast<unsigned char *>(smem4) + warp * A.warp_bytes;
  float *Pw = reinterpret_cast<float *>(stage + A.pw_offset);
  __shared__ uint32_t s_item[2];
  __shared__ int s_neg[8];
  listed_pixels<MT, NW, FUSED>(A, stage, s_item, s_neg);

  if constexpr (!FUSED) {
    light_stream<MT>(A, stage);
    return;
  }

  // ---------------- light pixels: one warp each, virtual index over slots x pixels.
  // A warp grabs kGrab consecutive virtual pixels; lanes 0..kGrab-1 fetch
  // their metadata in parallel, then the warp takes the pixels in order.
  const int64_t total = (int64_t)A.n_slots * A.npx;
  constexpr int kGrab = 4;
  for (;;) {
    uint32_t v0 = 0;
    if (lane == 0) v0 = atomicAdd(&A.cursors[1], (uint32_t)kGrab);
    v0 = __shfl_sync(0xffffffffu, v0, 0);
    if ((int64_t)v0 >= total) break;
    int m_slot = A.slot0, m_cnt = -1;
    int64_t m_a = 0;
    uint32_t m_key = 0, m_o0 = 0;
    const uint32_t *m_ev = nullptr;
    if (lane < kGrab) {
      const int64_t vi = (int64_t)v0 + lane;
      if (vi < total) {
        const int64_t q = A.n_slots == 1 ? 0 : vi / A.npx;
        m_slot = A.slot0 + (int)q;
        m_a = vi - q * A.npx;
        const SlotView &v = A.views[m_slot];
        if (m_a < (int64_t)v.counters[2]) {
          m_key = v.active[m_a];
          m_o0 = v.offsets[m_key];
          m_cnt = (int)(v.offsets[m_key + 1] - m_o0);
          m_ev = v.ev + m_o0;
        }
      }
    }
    for (int q = 0; q < kGrab; ++q) {
      const int cnt = __shfl_sync(0xffffffffu, m_cnt, q);
      const int slot = __shfl_sync(0xffffffffu, m_slot, q);
      const int64_t a = __shfl_sync(0xffffffffu, m_a, q);
      const uint32_t key = __shfl_sync(0xffffffffu, m_key, q);
      const uint32_t *evp = reinterpret_cast<const uint32_t *>(
          __shfl_sync(0xffffffffu, reinterpret_cast<uintptr_t>(m_ev), q));
      if (cnt < 0 || cnt >= A.light_max) continue;  // inactive, past the end, or listed
      pixel_spectrum_warp<MT>(A, evp, cnt, stage, Pw);
      CombOut o = comb_warp<NW>(Pw, A.cc, stage);
      store_scores<NW>(A, A.views[slot], a, key, o);
    }
  }
}

// Pixels of kTeamPixel events and fewer than A.heavy_min, which no list holds
// (the no-allocation entry point with many active pixels, whose fixed scratch lists
// the larger ones), by teams of four warps, one team per block. A block takes runs of
// up to 32 active pixels, short enough that every block gets sixteen of them, and
// looks at four runs at once. n_heavy[6] says whether there is any such pixel.
template <int MT>
__global__ void __launch_bounds__(128, 4) k_team_scan(const __grid_constant__ BlockedArgs A) {
  extern __shared__ float4 smem4[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char *stage = reinterpret_cast<unsigned char *>(smem4) + warp * A.warp_bytes;
  __shared__ int s_neg[4];
  if (A.n_heavy[6] == 0) return;
  const SlotView &v = A.views[0];
  const int64_t n_act = (int64_t)v.counters[2], blocks = gridDim.x;
  const int64_t run = max((int64_t)1, min((int64_t)32, n_act / (16 * blocks)));
  for (int64_t r0 = blockIdx.x; r0 * run < n_act; r0 += 4 * blocks) {
    uint32_t m[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t a = (r0 + u * blocks) * run + lane;
      int cnt = 0;
      if (lane < run && a < n_act) {
        const uint32_t key = v.active[a];
        cnt = (int)(v.offsets[key + 1] - v.offsets[key]);
      }
      m[u] = __ballot_sync(0xffffffffu, cnt >= kTeamPixel && cnt < A.heavy_min);
    }
#pragma unroll 1
    for (int u = 0; u < 4; ++u)
      for (uint32_t k = u == 0 ? m[0] : u == 1 ? m[1] : u == 2 ? m[2] : m[3]; k; k &= k - 1) {
        // the same pixels in every warp of the block
        const int64_t px = (r0 + u * blocks) * run + __ffs(k) - 1;
        for (int ps = 0; ps < (A.nbr + 8 * MT - 1) / (8 * MT); ++ps)
          team_item<MT, 1, false, 4>(A, (uint64_t)px, ps, stage, warp, 0, s_neg);
      }
  }
}

// m-tiles (of 8 rows) per pass for a grid of nbr rows: rows_per_lane (4 rows of
// a pass each) when the tuning sets it, else as few passes as MT <= 4 allows
// (every pass generates the columns again), evenly filled.
inline int tiles_per_pass(int nbr, int rows_per_lane) {
  if (rows_per_lane > 0) return std::max(1, rows_per_lane / 2);
  const int tiles = (nbr + 7) / 8, passes = (tiles + 3) / 4;
  return (tiles + passes - 1) / passes;
}

template <int MT>
int blocked_warp_bytes(const Ctx *c, bool fused, int NW, int *pw_offset) {
  int scratch = Stage<MT>::kBytes;
  *pw_offset = 0;
  if (!fused) return scratch;
  scratch = std::max(scratch, comb_scratch_bytes(c->comb, NW));
  scratch = (scratch + 15) & ~15;
  *pw_offset = scratch;
  return scratch + spectrum_rows<MT>((int)c->gconst.nbr) * 32 * 4;
}

// Blocks per cluster of a fused grid with `bps` blocks per SM (an unfused one has
// clusters of four). A GPC that its clusters do not fill leaves slots idle for the
// whole launch: with four blocks per SM clusters of four divide every GPC's blocks
// evenly, with the two that the fused kernel's scratch often leaves those of two, where
// four cost 3 to 5 % (640 bins, comb of 35 bins, 76,800 pixels: whole detection 4.80 ms,
// by two 4.55). Clusters of 2 / 4 / 8 of the unfused kernel (whole calls, us): sparse
// 1280x720 window 319 / 305 / 303, dense 3746 / 3783 / 3798, 320x180 at 10,000 bins
// 2772 / 2853 / 2913.
inline int fused_cluster(int bps) { return bps % 4 == 0 ? 4 : bps > 1 ? 2 : 1; }

// A grid of `blocks` blocks (rounded down to whole clusters).
template <typename K>
cudaError_t launch_clusters(K kern, int blocks, int cluster, int threads, size_t smem,
                            cudaStream_t s, const BlockedArgs &A) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)std::max(cluster, blocks / cluster * cluster));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)cluster;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, A);
}

// The caller zeroes the cursors (words 5 to 7 of qctl) and, when the list is not
// the one of a binning under this tuning, fills it (list_slot0).
template <int MT, int NW, bool FUSED>
ddhf_status launch_blocked_t(Ctx *c, int n_slots, float *P, int64_t cap_px, cudaStream_t s,
                             int slot0 = 0, int64_t ld = 0, int skip_min = 0) {
  BlockedArgs A{};
  A.views = c->d_views;
  A.slot0 = slot0;
  A.n_slots = n_slots;
  A.npx = c->npx;
  A.heavy = c->work;
  A.n_heavy = c->qctl + 0;
  A.heavy_cap = (uint32_t)std::min<int64_t>(c->heavy_cap, 0xffffffffll);
  A.cursors = c->qctl + 5;
  A.N = c->gconst.N;
  A.nbr = c->gconst.nbr;
  A.nd = make_ndft_const(c->gconst.a0, c->gconst.da, c->gconst.denom, A.N, A.nbr, MT);
  A.cc = c->comb;
  A.P = P;
  A.ld = ld > 0 ? ld : c->gconst.N;
  A.vec_store = (A.ld % 4 == 0) && (reinterpret_cast<uintptr_t>(P) % 16 == 0);
  A.cap_px = cap_px;
  A.heavy_min = A.light_max = list_min(c->tuning);  // as the list was filled
  A.skip_min = skip_min;
  A.warp_bytes = blocked_warp_bytes<MT>(c, FUSED, NW, &A.pw_offset);
  A.flags = c->flags;
  A.ev_cap = std::max<int64_t>(c->max_events, 1);
  const int wpb = c->tuning.warps_per_block;
  const size_t smem = (size_t)A.warp_bytes * wpb;
  auto kern = k_blocked<MT, NW, FUSED>;
  DDHF_CUDA_TRY(c, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)smem));
  int occ = 0;
  DDHF_CUDA_TRY(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, wpb * 32, smem));
  if (occ < 1) {
    c->last_error = "blocked kernel does not fit on an SM (shared memory)";
    return DDHF_ERR_UNSUPPORTED;
  }
  int bps = c->tuning.blocks_per_sm > 0 ? std::min(occ, c->tuning.blocks_per_sm) : occ;
  DDHF_CUDA_TRY(c, launch_clusters(kern, c->num_sms * bps, FUSED ? fused_cluster(bps) : kShares,
                                   wpb * 32, smem, s, A));
  return DDHF_OK;
}

// One kernel instantiation per m-tile count, for comb variant NW.
template <int NW, bool FUSED>
ddhf_status launch_blocked_mt(Ctx *c, int n_slots, float *P, int64_t cap_px, cudaStream_t s,
                              int slot0, int64_t ld, int skip_min) {
  switch (tiles_per_pass(c->gconst.nbr, c->tuning.rows_per_lane)) {
    case 1: return launch_blocked_t<1, NW, FUSED>(c, n_slots, P, cap_px, s, slot0, ld, skip_min);
    case 2: return launch_blocked_t<2, NW, FUSED>(c, n_slots, P, cap_px, s, slot0, ld, skip_min);
    case 3: return launch_blocked_t<3, NW, FUSED>(c, n_slots, P, cap_px, s, slot0, ld, skip_min);
    case 4: return launch_blocked_t<4, NW, FUSED>(c, n_slots, P, cap_px, s, slot0, ld, skip_min);
  }
  return DDHF_ERR_UNSUPPORTED;
}

// The fused kernels with the generic comb (1 or 8 mask words) are
// instantiated in their own translation unit.
extern template ddhf_status launch_blocked_mt<1, true>(Ctx *, int, float *, int64_t, cudaStream_t,
                                                       int, int64_t, int);
extern template ddhf_status launch_blocked_mt<8, true>(Ctx *, int, float *, int64_t, cudaStream_t,
                                                       int, int64_t, int);

template <bool FUSED>
ddhf_status launch_blocked_any(Ctx *c, int n_slots, float *P, int64_t cap_px, cudaStream_t s,
                               int slot0 = 0, int64_t ld = 0, int skip_min = 0) {
  if constexpr (!FUSED) {
    return launch_blocked_mt<1, false>(c, n_slots, P, cap_px, s, slot0, ld, skip_min);
  } else {
    // the comb variant of the spectrum size: fast, or generic with 1 or 8 mask words
    switch (comb_variant(c->comb)) {
      case 0: return launch_blocked_mt<0, true>(c, n_slots, P, cap_px, s, slot0, ld, 0);
      case 1: return launch_blocked_mt<1, true>(c, n_slots, P, cap_px, s, slot0, ld, 0);
      default: return launch_blocked_mt<8, true>(c, n_slots, P, cap_px, s, slot0, ld, 0);
    }
  }
}

}  // namespace blocked
}  // namespace ddhf

// Constants of the blocked NDFT's phases for one grid: host arithmetic in plain
// integers (no CUDA), done at every launch.
#pragma once

#include <stdint.h>

namespace ddhf {
namespace blocked {

constexpr int kMaxPasses = 64;  // 512 rows of 32 bins, at least 8 per pass

// Phases as fractions of a turn in units of 2^-64.
struct NdftConst {
  uint64_t f_u;                // da / D (one bin)
  uint64_t f_k8;               // 8.5 da / D (column k = 8)
  uint64_t f_v;                // 32 da / D (one row)
  uint64_t f_row[kMaxPasses];  // a_c(b0 + 4 MT) / D: the middle row of each pass in use
  int32_t dc_first, dc_step;   // bins with a_j = 0 mod D: dc_first + i dc_step (-1: none)
};

inline uint64_t turn_fraction(unsigned __int128 num, uint64_t den) {
  const uint64_t r = (uint64_t)(num % den);
  return (uint64_t)((((unsigned __int128)r << 64) + den / 2) / den);
}

// Grid a_j = a0 + j da < 2^32 in units of 1 / D (0 < D < 2^31), N bins in nbr
// rows of 32, mt m-tiles (of 8 rows) per pass. The rows of the passes in use alone,
// and the bins of phase 0 from the congruence j da = -a0 (mod D) solved by the
// extended Euclidean algorithm: 0.2 us at 750 bins and 0.6 us at 10,000 from 0.5 Hz
// (every pass and a search over the bins: 2.7 and 19 us, on an x86 host).
inline NdftConst make_ndft_const(uint64_t a0, uint64_t da, uint64_t D, int N, int nbr, int mt) {
  NdftConst n{};
  const unsigned __int128 a = a0, d = da;
  n.f_u = turn_fraction(d, D);
  n.f_k8 = turn_fraction(17 * d, 2 * D);
  n.f_v = turn_fraction(32 * d, D);
  for (int i = 0; i < kMaxPasses && 8 * mt * i < nbr; ++i)
    n.f_row[i] = turn_fraction(2 * a + (64 * (unsigned)(8 * mt * i + 4 * mt) + 31) * d, 2 * D);
  // x = gcd(da, D) = u da (mod D)
  int64_t x = (int64_t)da, y = (int64_t)D, u = 1, v = 0;
  while (y) {
    const int64_t q = x / y, r = x - q * y, w = u - q * v;
    x = y;
    y = r;
    u = v;
    v = w;
  }
  const uint64_t step = D / (uint64_t)x;
  n.dc_step = (int32_t)(step < ((uint64_t)1 << 30) ? step : (uint64_t)1 << 30);
  n.dc_first = -1;
  if (a0 % (uint64_t)x == 0) {
    const int64_t m = u % (int64_t)step;
    const uint64_t inv = (uint64_t)(m < 0 ? m + (int64_t)step : m);  // (da / x)^-1 mod step
    const uint64_t j = (step - a0 / (uint64_t)x % step) % step * inv % step;
    if (j < (uint64_t)N) n.dc_first = (int32_t)j;
  }
  return n;
}

}  // namespace blocked
}  // namespace ddhf

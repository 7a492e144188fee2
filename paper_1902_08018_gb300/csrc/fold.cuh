// fold.cuh -- folding a band's compensated lane sums over the lanes of a warp.
//
// A warp ends every piece of a band with 4 R values per lane, each a
// compensated FP32 pair, to be added over its lanes.  GB300 retires about two
// FP64 lane operations per SM and clock (16 clocks an instruction of a warp), so
// widening each lane's pairs and adding them in FP64 butterflies took about 500
// clocks of an SM per piece and column, with every warp of the grid arriving at
// the end of its range together.  Here the values are exchanged while they are
// added -- a level hands half of them to the partner lane, so N values take about
// N + log2(lanes) additions, not N log2(lanes) -- in FP32 without loss, and only
// the totals are widened (by integer instructions).  Two arithmetics:
//   pairs (hi, lo): good to about 2^-48;
//   triples (hi, lo, rest), for the FP64 fold: good to about 2^-70, beyond FP64.
// Each addition is symmetric in its operands, so a value's total has the same
// bits whatever the number of values folded with it.  Per pass, before and
// after: 4096^2 at rate 16 28.3 -> 22.6 us, a slit of 378 x 32768 34.8 -> 23.8,
// 16384^2 at rate 16 101.7 -> 97.2, 256000 x 378 in BF16 47.2 -> 43.7 us.
#pragma once
#include <cstdint>

namespace whff {
namespace dev {

// f as FP64 by integer instructions (the conversion runs on the FP64 pipe).
__device__ __forceinline__ double widen(float f) {
  const uint32_t u = __float_as_uint(f), m = u & 0x7FFFFFFFu;
  if (m - 0x00800000u >= 0x7F000000u && m) return (double)f;  // subnormal, infinite, NaN
  const uint32_t hi = (u & 0x80000000u) | ((m >> 3) + (896u << 20));
  return m ? __hiloint2double((int)hi, (int)(u << 29)) : __hiloint2double((int)u, 0);
}

// z * 2^k on the exponent field where that stays in the normal range.
__device__ __forceinline__ double times_pow2(double z, int k) {
  const int hi = __double2hiint(z), e = (hi >> 20) & 2047;
  if (e > 8 && e < 2039) return __hiloint2double(hi + (k << 20), __double2loint(z));
  return z * (k < 0 ? 1.0 / (double)(1 << -k) : (double)(1 << k));
}

__device__ __forceinline__ double negate_if(double z, bool n) {
  return __hiloint2double(__double2hiint(z) ^ (n ? (int)0x80000000 : 0), __double2loint(z));
}

__device__ __forceinline__ float two_sum_err(float a, float b, float s) {  // s = a + b: its rounding error
  const float bp = s - a;
  return (a - (s - bp)) + (b - bp);
}

// Sums over aligned groups of GL lanes of N values per lane (N, GL powers of
// two), value k being hi[k] + lo[k].  Lane l of a group ends with the totals of
// values fold_index<N, GL>(l) .. + C - 1, C = max(1, N / GL), in z; the GL / N
// lanes that share a value (N < GL) all hold it.  All 32 lanes call it.
template <int N, int GL>
__device__ __forceinline__ constexpr int fold_index(int l) {
  return N >= GL ? l * (N / GL) : l / (GL / N);
}

// The level at lane distance O, with the first C of the N values still apart.
template <int N, int C, int O, bool TRIPLE>
__device__ __forceinline__ void fold_level(float (&h)[N], float (&l)[N], float (&m)[TRIPLE ? N : 1], int lane) {
  constexpr unsigned kAll = 0xFFFFFFFFu;
  constexpr int kHalf = C > 1 ? C / 2 : 1;
  const bool up = C > 1 && (lane & O);
#pragma unroll
  for (int k = 0; k < kHalf; ++k) {
    constexpr int kGap = C > 1 ? kHalf : 0;
    const float h2 = __shfl_xor_sync(kAll, up ? h[k] : h[k + kGap], O);
    const float l2 = __shfl_xor_sync(kAll, up ? l[k] : l[k + kGap], O);
    const float h1 = up ? h[k + kGap] : h[k], l1 = up ? l[k + kGap] : l[k];
    const float s = h1 + h2, e = two_sum_err(h1, h2, s);
    h[k] = s;
    if constexpr (TRIPLE) {
      const float m2 = __shfl_xor_sync(kAll, up ? m[k] : m[k + kGap], O), m1 = up ? m[k + kGap] : m[k];
      const float t = l1 + l2, f = two_sum_err(l1, l2, t);
      const float u = t + e, g = two_sum_err(t, e, u);
      l[k] = u;
      m[k] = (m1 + m2) + (f + g);
    } else {
      l[k] = (l1 + l2) + e;
    }
  }
  if constexpr (O > 1) fold_level<N, kHalf, O / 2, TRIPLE>(h, l, m, lane);
}

// Triples: sums that might leave FP32's range go down by 2^5 first (FP64 held them).
template <int N, int GL, bool TRIPLE>
__device__ __forceinline__ void fold_lanes(float (&h)[N], float (&l)[N], int lane, double (&z)[N >= GL ? N / GL : 1]) {
  float m[TRIPLE ? N : 1];
#pragma unroll
  for (int k = 0; k < (TRIPLE ? N : 1); ++k) m[k] = 0.f;
  bool big = false;
  if constexpr (TRIPLE) {
    float top = 0.f;
#pragma unroll
    for (int k = 0; k < N; ++k) top = fmaxf(top, fabsf(h[k]));
    big = __any_sync(0xFFFFFFFFu, top >= 5.3e36f);  // 2^122
    if (big) {
#pragma unroll
      for (int k = 0; k < N; ++k) h[k] *= 0.03125f, l[k] *= 0.03125f;
    }
  }
  fold_level<N, N, GL / 2, TRIPLE>(h, l, m, lane);
#pragma unroll
  for (int k = 0; k < (N >= GL ? N / GL : 1); ++k) {
    if constexpr (TRIPLE) {
      z[k] = widen(h[k]) + (widen(l[k]) + widen(m[k]));
    } else {
      z[k] = widen(h[k]) + widen(l[k]);
    }
    if (TRIPLE && big) z[k] *= 32.0;
  }
}

}  // namespace dev
}  // namespace whff

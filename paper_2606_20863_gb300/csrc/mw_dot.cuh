// What the inner-product kernel (mw_dot.cu) and the power-series kernel
// (mw_series.cu) share: the arguments, the compiled piece counts and the 24-bit
// balanced digits of a fixed-point value.
#pragma once
#include <cstdint>

#include "mw_column.cuh"
#include "mw_device.cuh"
#include "mw_internal.h"
#include "mw_limbs.cuh"

namespace mw {

constexpr int kDotW = 24;           // digit width
constexpr int kDotThreads = 256;
constexpr int kDotExtraD = 4;       // diagonals kept beyond S (D <= S + kDotExtraD)

struct DotArgs {
  const double *A, *B;
  double *C;
  int64_t lda, psa, ldb, psb, psc;
  int64_t count, K;
  int D, range_A, range_B;
  unsigned int *status;
  // power series: count series of n = K coefficients, product u = (s, i) for
  // u < count * n, output at C[s * ldc + i]
  int conv;
  int64_t ldc;
};

// instances: S for w = 24 and exponent spreads of up to about 80 bits
template <int MW> struct DotS;
template <> struct DotS<2> { static constexpr int lo = 4, hi = 8; };
template <> struct DotS<4> { static constexpr int lo = 8, hi = 12; };
template <> struct DotS<8> { static constexpr int lo = 17, hi = 21; };
template <> struct DotS<16> { static constexpr int lo = 35, hi = 36; };

// Whether mw_series.cu takes count power series of n coefficients: their digits fit in shared
// memory and they are not so few that the inner-product kernel is the faster one.
bool series_fits(int m, int S, int64_t count, int64_t n);
int launch_series(int m, int S, const DotArgs &a, cudaStream_t st);

namespace {

// 32-bit limbs of a fixed-point value of S digits (|T| < 2^(24 S + 1), a sign bit).
__host__ __device__ constexpr int dot_limbs(int S) { return (kDotW * S + 3 + 31) / 32 < 4 ? 4 : (kDotW * S + 3 + 31) / 32; }

// limb i of H = sum of 2^(24k + 23) for k = 0 .. S-2: adding it makes the low digits
// plain 24-bit fields
template <int S>
__host__ __device__ constexpr uint32_t dot_bias(int limb) {
  uint32_t v = 0;
  for (int k = 0; k + 1 < S; ++k) {
    const int bit = kDotW * k + kDotW - 1;
    if (bit / 32 == limb) v |= 1u << (bit % 32);
  }
  return v;
}

// Balanced digits d[p] (p = 0 most significant) of T = sum_j trunc(x_j 2^F), w = 24:
// 24-bit fields of T + H minus 2^23; the top digit is the signed value above
// them.  Returns false when T lies outside [-2^(wS-1), 2^(wS-1)), which is checked on the
// digits where the exponents do not show it (surely_in_range).
template <int MW, int S>
__device__ __forceinline__ bool dot_cut(const double (&x)[MW], int F, int32_t (&d)[S]) {
  constexpr int NL = dot_limbs(S);
  uint32_t T[NL];
#pragma unroll
  for (int i = 0; i < NL; ++i) T[i] = dot_bias<S>(i);
  const uint32_t h0 = (uint32_t)__double2hiint(x[0]) << 1;
  uint32_t h1 = 0;
#pragma unroll
  for (int j = 0; j < MW; ++j) {
    if (j) h1 = max(h1, (uint32_t)__double2hiint(x[j]) << 1);
    add_word32<NL>(x[j], F, T);
  }
  int lsign = 0;
  static_assert(MW <= 4, "m >= 8 goes through cut_column");
  const bool plain = surely_in_range<MW>(h0, h1, kDotW * S - 2 - F);
#pragma unroll
  for (int k = 0; k < S; ++k) {          // k: position from the least significant digit
    const int bit = kDotW * k, li = bit >> 5, off = bit & 31;
    uint32_t win = T[li] >> off;
    if (k + 1 < S) {
      if (off > 8) win |= T[li + 1] << (32 - off);
      d[S - 1 - k] = (int32_t)(win & 0xFFFFFFu) - (1 << 23);
    } else {                             // everything from bit 24 (S-1) up, sign included
      d[0] = li + 1 < NL ? (int32_t)__funnelshift_r(T[li], T[li + 1], off)
                         : (int32_t)T[li] >> off;
    }
  }
  if (plain) return true;
  // T = top 2^(w(S-1)) + L with L of the sign of its highest nonzero digit: in range for
  // |top| < 2^(w-1), for top = -2^(w-1) with L >= 0 and top = 2^(w-1) with L < 0
#pragma unroll
  for (int k = 0; k + 1 < S; ++k)
    if (d[S - 1 - k] != 0) lsign = d[S - 1 - k] > 0 ? 1 : -1;
  constexpr int top_bits = 32 * NL - kDotW * (S - 1);            // bits of the top field
  bool above = true;                                             // they extend d[0]'s sign
  if constexpr (top_bits > 32) {
    constexpr int li = kDotW * (S - 1) / 32, off = kDotW * (S - 1) % 32;
    static_assert(li + 1 == NL - 1, "the top field ends in the last limb");
    above = ((int32_t)T[NL - 1] >> off) == (d[0] >> 31);
  }
  constexpr int half = 1 << 23;
  return above && ((d[0] > -half && d[0] < half) || (d[0] == -half && lsign >= 0) ||
                   (d[0] == half && lsign < 0));
}

// ilogb + 1 of the largest word of an entry (kExpZero, kExpNonFinite as exp_plus1):
// the largest high word without its sign holds it unless it is zero, subnormal or not finite.
template <int MW>
__device__ __forceinline__ int entry_exp(const double (&x)[MW]) {
  uint32_t h = 0;
#pragma unroll
  for (int j = 0; j < MW; ++j) h = max(h, (uint32_t)__double2hiint(x[j]) << 1);
  const int be = (int)(h >> 21);
  if (be != 0 && be != 0x7ff) return be - 1022;
  // zeros first: a warp with one of them would go through every word's exponent (1,000
  // hexa-double products of 40 with half of the entries zero 331 us, 312 before)
#pragma unroll
  for (int j = 0; j < MW; ++j) h |= (uint32_t)__double2loint(x[j]);
  if (h == 0) return kExpZero;
  int e = kExpZero;
#pragma unroll
  for (int j = 0; j < MW; ++j) e = max(e, exp_plus1(x[j]));      // non-finite: the largest
  return e;
}

}  // namespace
}  // namespace mw

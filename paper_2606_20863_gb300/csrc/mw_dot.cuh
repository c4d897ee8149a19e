// What the inner-product kernel (mw_dot.cu) and the power-series kernel
// (mw_series.cu) share: the arguments, the compiled piece counts and the 24-bit
// balanced digits of a fixed-point value.
#pragma once
#include <cstdint>

#include "mw_device.cuh"
#include "mw_internal.h"
#include "mw_pieces.cuh"

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

// Power series of n coefficients whose digits fit in shared memory (mw_series.cu);
// false (nothing launched) when they do not: the inner-product kernel takes them.
bool series_fits(int m, int S, int64_t n);
int launch_series(int m, int S, const DotArgs &a, cudaStream_t st);

namespace {

// bits 24k + 23 for k = 0 .. S-2 (the bias that makes the low digits bytes-like)
template <int S>
__host__ __device__ constexpr uint64_t dot_bias(int limb) {
  uint64_t v = 0;
  for (int k = 0; k + 1 < S; ++k) {
    const int bit = kDotW * k + kDotW - 1;
    if (bit / 64 == limb) v |= 1ull << (bit % 64);
  }
  return v;
}

// Balanced digits d[p] (p = 0 most significant) of the NL-limb fixed-point
// value T, w = 24: with 2^23 added to every low digit the digits are 24-bit
// fields minus 2^23; the top digit is the signed value above them.  Returns
// false when T lies outside [-2^(wS-1), 2^(wS-1)).
template <int S, int NL>
__device__ __forceinline__ bool dot_digits(uint64_t (&T)[NL], int32_t (&d)[S]) {
  constexpr int b = kDotW * S - 1, lb = b >> 6, ob = b & 63;
  static_assert(lb < NL, "limbs cover the digits");
  const int64_t v = (int64_t)T[lb] >> ob;
  bool ok = v == 0 || v == -1;
#pragma unroll
  for (int i = lb + 1; i < NL; ++i) ok &= T[i] == (uint64_t)v;
  uint64_t H[NL];
#pragma unroll
  for (int i = 0; i < NL; ++i) H[i] = dot_bias<S>(i);
  add_limbs<NL>(T, H);
#pragma unroll
  for (int k = 0; k < S; ++k) {          // k: position from the least significant digit
    const int bit = kDotW * k, li = bit >> 6, off = bit & 63;
    uint64_t win = T[li] >> off;
    if (off != 0 && li + 1 < NL) win |= T[li + 1] << (64 - off);
    if (k + 1 < S) {
      d[S - 1 - k] = (int32_t)(win & 0xFFFFFF) - (1 << 23);
    } else {
      // the top digit: everything from bit 24 (S-1) up, sign included
      const int64_t top = (li + 1 < NL || off == 0) ? (int64_t)win : ((int64_t)T[li] >> off);
      d[0] = (int32_t)top;
    }
  }
  return ok;
}

}  // namespace
}  // namespace mw

// Cutting entries into pieces and rounding exact integers into m words with a
// per-thread column of 32-bit words in shared memory, indexed at run time, so
// that each word of an m-double touches only the few slots or limbs at its own
// position (device side; also compiles as plain C++).
//   cut_column:   the balanced w-bit digits (w = 8 or 24) of
//                 T = sum_j trunc(x_j 2^F) (Section 2's pieces on the shared
//                 grid): each word adds its truncated magnitude as four signed
//                 24-bit fields into the slots it covers, then one carry pass
//                 from the least significant slot yields the digits;
//   round_column: the m nonoverlapping doubles of X 2^ex, each the value
//                 rounded to nearest (ties to even) of what the previous words
//                 left over (Section 4's final renormalisation, greedy), read
//                 from the two's complement limbs of X without rewriting them.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>
#include <type_traits>

#if defined(__CUDACC__)
#define MW_HD __host__ __device__ __forceinline__
#else
#define MW_HD inline
#endif

namespace mw {
namespace {

MW_HD uint64_t col_bits(double x) {
#if defined(__CUDA_ARCH__)
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t b;
  std::memcpy(&b, &x, sizeof b);
  return b;
#endif
}
MW_HD double col_double(uint64_t b) {
#if defined(__CUDA_ARCH__)
  return __longlong_as_double((long long)b);
#else
  double x;
  std::memcpy(&x, &b, sizeof x);
  return x;
#endif
}
MW_HD int col_clz(uint32_t x) {
#if defined(__CUDA_ARCH__)
  return __clz(x);
#else
  return x ? __builtin_clz(x) : 32;
#endif
}
MW_HD int col_ctz(uint32_t x) {  // x != 0
#if defined(__CUDA_ARCH__)
  return __ffs((int)x) - 1;
#else
  return __builtin_ctz(x);
#endif
}

MW_HD uint32_t col_fshl(uint32_t lo, uint32_t hi, int n) {  // high word of (hi:lo) << n, n < 32
#if defined(__CUDA_ARCH__)
  return __funnelshift_l(lo, hi, n);
#else
  return (uint32_t)(((((uint64_t)hi << 32) | lo) << n) >> 32);
#endif
}
MW_HD uint32_t col_fshr(uint32_t lo, uint32_t hi, int n) {  // low word of (hi:lo) >> n, n < 32
#if defined(__CUDA_ARCH__)
  return __funnelshift_r(lo, hi, n);
#else
  return (uint32_t)((((uint64_t)hi << 32) | lo) >> n);
#endif
}
MW_HD uint64_t col_shr64(uint64_t x, int n) {  // x >> n, zero from n = 64 on
#if defined(__CUDA_ARCH__)
  uint64_t r;
  asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
#else
  return n < 64 ? x >> n : 0;
#endif
}
MW_HD float col_float(uint32_t b) {
#if defined(__CUDA_ARCH__)
  return __uint_as_float(b);
#else
  float f;
  std::memcpy(&f, &b, sizeof f);
  return f;
#endif
}
MW_HD uint32_t col_fbits(float f) {
#if defined(__CUDA_ARCH__)
  return __float_as_uint(f);
#else
  uint32_t b;
  std::memcpy(&b, &f, sizeof b);
  return b;
#endif
}

// bfloat16 bits of an integer |d| <= 2^8 (exact): 1.5 2^23 + d has the float
// bit pattern 0x4B400000 + d, less 1.5 2^23 it is d; a float of at most 8
// significant bits is its top 16 bits.
MW_HD uint16_t small_int_bf16(int32_t d) {
  return (uint16_t)(col_fbits(col_float(0x4B400000u + (uint32_t)d) - 12582912.0f) >> 16);
}

// Slots of the column for S digits of w bits: the 24-bit chunk holding the top
// digit, Ct = w (S-1) / 24, the ones below it and three above it (the highest
// a word's four fields can reach; they stay zero for in-range input).
MW_HD int cut_column_slots(int w, int S) { return w * (S - 1) / 24 + 4; }

// T certainly in range, from the high words without their signs, shifted left by one: of
// the first word (h0) and the largest of the others (h1), on the grid 2^-F below 2^top,
// top = wS - 2 - F.  |x_0| 2^F < 2^(wS-2) and the others log2(MW) binary orders below
// 2^top, so that |T| < 2 2^(wS-2).  Holds for zeros too: entries that need the exact check
// are rare, and a warp with one of them takes both ways (batches of hexa doubles with half
// of their entries zero 220 us while zeros were checked, 193 before there were two ways).
template <int MW> MW_HD bool surely_in_range(uint32_t h0, uint32_t h1, int top) {
  constexpr uint32_t kGap = MW <= 2 ? 1 : MW <= 4 ? 2 : MW <= 8 ? 3 : 4;
  static_assert(MW <= 16, "gap of the later words");
  const uint32_t e1 = (h1 >> 21) + kGap, e = h0 >> 21 > e1 ? h0 >> 21 : e1;
  return (int)e - 1022 <= top;
}

// Balanced digits d_k (k = 0 least significant) of T = sum_j trunc(x_j 2^F):
// d_k in [-2^(w-1), 2^(w-1)) for k < S-1, the top digit d_(S-1) the rest (in
// [-2^(w-1), 2^(w-1)] when T lies in [-2^(wS-1), 2^(wS-1))).  emit(k, d) is
// called once per digit in the order k = 0, 1, ..., S-1.  Returns false when T
// lies outside that range.
// col: this thread's column, slot c at col[c * stride], cut_column_slots(w, S)
// of them, all zero on entry and left zero.  Slot c collects bits 24c .. 24c+23
// of every word plus a signed excess; the carry pass adds the bias
// H = 2^(w-1) (1 + 2^w + ... + 2^(w(S-2))), after which every digit below the
// top one is a plain w-bit field minus 2^(w-1).
// FAST compiles the carry pass twice, without the range's bookkeeping for entries
// that are certainly in range (inner products of octo doubles 515 -> 500 us); kernels
// in which the cut is a small part are faster with one copy (2,000 octo-double series
// products 674 -> 625 us).
template <int MW, int W, bool FAST = true, class Emit>
MW_HD bool cut_column(const double (&x)[MW], int F, int S, uint32_t *col, int stride, Emit emit) {
  static_assert(W == 8 || W == 24, "digit widths 8 and 24");
  constexpr int32_t kHalf = 1 << (W - 1);
  constexpr int32_t kBias = W == 24 ? kHalf : 0x808080;   // H restricted to a full chunk
  const int Ct = W * (S - 1) / 24;
  uint32_t h1 = 0;                                  // largest high word (no sign) after the first
#pragma unroll
  for (int j = 0; j < MW; ++j) {
    const uint64_t b = col_bits(x[j]);
    const uint32_t bh = (uint32_t)(b >> 32);
    if (j) h1 = h1 > (bh << 1) ? h1 : bh << 1;
    const int be = (int)((bh >> 20) & 0x7ff);
    const int sh = (be ? be : 1) - 1075 + F;      // weight of M's last bit on the grid
    // y = trunc(M 2^min(sh, 0)) at bit pos = max(sh, 0), M < 2^53
    uint64_t M = ((uint64_t)((bh & 0xFFFFFu) | (be ? 0x100000u : 0u)) << 32) | (uint32_t)b;
    M = col_shr64(M, sh < 0 ? -sh : 0);
    int pos = sh < 0 ? 0 : sh;
    uint32_t ylo = (uint32_t)M, yhi = (uint32_t)(M >> 32);
    if (pos >= 24 * (Ct + 1)) {                     // only words the exponent does not cover
      ylo = yhi = 0;                                // (non-finite input, flagged elsewhere)
      pos = 0;
    }
    const int c = pos / 24, o = pos - 24 * c;
    const uint32_t w0 = ylo << o, w1 = col_fshl(ylo, yhi, o), w2 = col_fshl(yhi, 0u, o);
    const int32_t f0 = (int32_t)(w0 & 0xFFFFFFu);
    const int32_t f1 = (int32_t)(col_fshr(w0, w1, 24) & 0xFFFFFFu);
    const int32_t f2 = (int32_t)(col_fshr(w1, w2, 16) & 0xFFFFFFu);
    const int32_t f3 = (int32_t)(w2 >> 8);
    const int32_t s = (bh >> 31) ? -1 : 1;
    uint32_t *p = col + c * stride;
    p[0] = (uint32_t)((int32_t)p[0] + s * f0);
    p[stride] = (uint32_t)((int32_t)p[stride] + s * f1);
    p[2 * stride] = (uint32_t)((int32_t)p[2 * stride] + s * f2);
    p[3 * stride] = (uint32_t)((int32_t)p[3 * stride] + s * f3);
  }
  // carry pass.  Where T is not certainly in range, lsign, the sign of the digits below
  // the top one, read off the most significant nonzero one (balanced digits), decides at
  // the edges of the range
  const bool plain = surely_in_range<MW>((uint32_t)(col_bits(x[0]) >> 32) << 1, h1, W * S - 2 - F);
  auto pass = [&](auto check) -> bool {
    constexpr bool kCheck = decltype(check)::value;
    int32_t carry = 0;
    int lsign = 0;
#pragma unroll
    for (int c = 0; c < Ct; ++c) {
      const int32_t v = (int32_t)col[c * stride] + carry + kBias;
      col[c * stride] = 0u;
      carry = v >> 24;
      const int32_t u = v & 0xFFFFFF;
      if (kCheck && u != kBias) lsign = u > kBias ? 1 : -1;
      if (W == 24) {
        emit(c, u - kHalf);
      } else {
        emit(3 * c, (u & 0xFF) - 128);
        emit(3 * c + 1, ((u >> 8) & 0xFF) - 128);
        emit(3 * c + 2, (u >> 16) - 128);
      }
    }
    const int nb = W == 24 ? 0 : S - 1 - 3 * Ct;     // digits of chunk Ct below the top one
    const int32_t v = (int32_t)col[Ct * stride] + carry + (W == 24 ? 0 : (0x808080 & ((1 << (8 * nb)) - 1)));
    for (int i = 0; i < nb; ++i) {
      const int32_t d = ((v >> (8 * i)) & 0xFF) - 128;
      emit(3 * Ct + i, d);
      if (kCheck && d != 0) lsign = d > 0 ? 1 : -1;
    }
    const int32_t top = v >> (W == 24 ? 0 : 8 * nb);
    emit(S - 1, top);
    const uint32_t above = col[(Ct + 1) * stride] | col[(Ct + 2) * stride] | col[(Ct + 3) * stride];
    col[Ct * stride] = 0u;
    col[(Ct + 1) * stride] = 0u;
    col[(Ct + 2) * stride] = 0u;
    col[(Ct + 3) * stride] = 0u;
    // T = top 2^(w(S-1)) + L, |L| < 2^(w(S-1)), L of sign lsign: in range for
    // |top| < 2^(w-1), for top = -2^(w-1) with L >= 0 and top = 2^(w-1) with L < 0
    return !kCheck || (above == 0u && ((top > -kHalf && top < kHalf) || (top == -kHalf && lsign >= 0) ||
                                       (top == kHalf && lsign < 0)));
  };
  if constexpr (FAST)
    if (plain) return pass(std::false_type());
  return pass(std::true_type());
}

// X 2^ex into MW words by greedy rounding to nearest, ties to even: word k is
// the remainder left by words 0 .. k-1 rounded to 53 bits; zeros once the
// remainder vanishes.  U: X in NL32 32-bit limbs, two's complement.  col: this
// thread's column of NL32 words (limb L at col[L * stride]).
// The remainder below the last cut is never written back: with l the lowest
// set bit of X, the magnitude of -X and of each remainder after a word that
// rounded up is X's own bits inverted above l and kept at and below l (the
// negation of a two's complement integer), so one flag, flipped at every
// rounding up, says which of the two readings applies, and the bits below any
// window are nonzero exactly when l lies below it.
template <int MW, int NL32, class Store>
MW_HD void round_column(const uint32_t (&U)[NL32], uint32_t *col, int stride, int ex,
                        Store store) {
  int lw = 0;
  uint32_t lv = U[0];
#pragma unroll
  for (int i = 0; i < NL32; ++i) col[i * stride] = U[i];
  if (lv == 0) {                                    // rare: the last limb is zero
    lw = -1;
#pragma unroll
    for (int i = NL32 - 1; i >= 1; --i)
      if (U[i] != 0) {
        lw = i;
        lv = U[i];
      }
  }
  int k = 0;
  if (lw >= 0) {
    const int ell = 32 * lw + col_ctz(lv);
    const uint32_t inv_l = ~((2u << (ell & 31)) - 1u);    // bits above l in limb lw
    uint32_t flip = (uint32_t)((int32_t)U[NL32 - 1] >> 31);   // all ones: inverted above l
    uint32_t neg = flip & 0x80000000u;
    int cutp = 32 * NL32;                                 // bits at and above are cleared
#pragma unroll 1
    for (; k < MW && ell < cutp; ++k) {
      auto limb = [&](int L) -> uint32_t {                // below the cut
        if (L < 0) return 0u;
        return col[L * stride] ^ (flip & (L > lw ? 0xFFFFFFFFu : (L == lw ? inv_l : 0u)));
      };
      int h = (cutp - 1) >> 5;
      uint32_t a = limb(h);
      if (cutp & 31) a &= (1u << (cutp & 31)) - 1u;
      while (a == 0 && h > lw) a = limb(--h);           // bit l is set: ends at lw at the latest
      const uint32_t b = limb(h - 1), c = limb(h - 2);
      const bool below = ell < 32 * (h - 2);
      const int lz = col_clz(a);
      // the 64 bits from the top one on, then the bits of c below them
      const uint32_t t1 = col_fshl(b, a, lz), t0 = col_fshl(c, b, lz), c_low = c << lz;
      uint64_t mant = ((uint64_t)(t1 >> 11) << 32) | col_fshr(t0, t1, 11);
      const uint32_t rbit = (t0 >> 10) & 1u;
      const bool sticky = ((t0 & 0x3FFu) | c_low) != 0 || below;
      const uint32_t up = rbit & (uint32_t)(sticky | (t0 >> 11 & 1u));
      mant += up;
      const int cut = 32 * h - 21 - lz;                   // weight of the mantissa's last bit
      const int e = ex + cut;
      const int bexp = e + 52 + 1023;                     // mant in [2^52, 2^53]
      double mag;
      if (bexp >= 1 && bexp <= 2045)
        mag = col_double(((uint64_t)bexp << 52) + (mant - (1ull << 52)));
      else
        mag = scalbn((double)mant, e);
      store(k, col_double(col_bits(mag) ^ ((uint64_t)neg << 32)));
      if (up) {
        flip = ~flip;
        neg ^= 0x80000000u;
      }
      cutp = cut;
    }
  }
  for (; k < MW; ++k) store(k, 0.0);
}

}  // namespace
}  // namespace mw

// Fixed-point values of m-double entries in 32-bit limbs (device side): the residue
// split, the inner products and the power series of two and four words cut from them.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

namespace mw {
namespace {

// T += y + (s & 1) on NL limbs, s zero or all ones: one carry chain.
template <int NL>
__device__ __forceinline__ void add_limbs32(uint32_t (&T)[NL], const uint32_t (&y)[NL], uint32_t s);
template <>
__device__ __forceinline__ void add_limbs32<4>(uint32_t (&T)[4], const uint32_t (&y)[4], uint32_t s) {
  asm("{\n" ".reg .u32 c;\n"
      "add.cc.u32 c, %8, %8;\n"
      "addc.cc.u32 %0, %0, %4;\n"
      "addc.cc.u32 %1, %1, %5;\n"
      "addc.cc.u32 %2, %2, %6;\n"
      "addc.u32 %3, %3, %7;\n" "}"
      : "+r"(T[0]), "+r"(T[1]), "+r"(T[2]), "+r"(T[3])
      : "r"(y[0]), "r"(y[1]), "r"(y[2]), "r"(y[3]), "r"(s));
}
template <>
__device__ __forceinline__ void add_limbs32<5>(uint32_t (&T)[5], const uint32_t (&y)[5], uint32_t s) {
  asm("{\n" ".reg .u32 c;\n"
      "add.cc.u32 c, %10, %10;\n"
      "addc.cc.u32 %0, %0, %5;\n"
      "addc.cc.u32 %1, %1, %6;\n"
      "addc.cc.u32 %2, %2, %7;\n"
      "addc.cc.u32 %3, %3, %8;\n"
      "addc.u32 %4, %4, %9;\n" "}"
      : "+r"(T[0]), "+r"(T[1]), "+r"(T[2]), "+r"(T[3]), "+r"(T[4])
      : "r"(y[0]), "r"(y[1]), "r"(y[2]), "r"(y[3]), "r"(y[4]), "r"(s));
}
template <>
__device__ __forceinline__ void add_limbs32<6>(uint32_t (&T)[6], const uint32_t (&y)[6], uint32_t s) {
  asm("{\n" ".reg .u32 c;\n"
      "add.cc.u32 c, %12, %12;\n"
      "addc.cc.u32 %0, %0, %6;\n"
      "addc.cc.u32 %1, %1, %7;\n"
      "addc.cc.u32 %2, %2, %8;\n"
      "addc.cc.u32 %3, %3, %9;\n"
      "addc.cc.u32 %4, %4, %10;\n"
      "addc.u32 %5, %5, %11;\n" "}"
      : "+r"(T[0]), "+r"(T[1]), "+r"(T[2]), "+r"(T[3]), "+r"(T[4]), "+r"(T[5])
      : "r"(y[0]), "r"(y[1]), "r"(y[2]), "r"(y[3]), "r"(y[4]), "r"(y[5]), "r"(s));
}
template <>
__device__ __forceinline__ void add_limbs32<7>(uint32_t (&T)[7], const uint32_t (&y)[7], uint32_t s) {
  asm("{\n" ".reg .u32 c;\n"
      "add.cc.u32 c, %14, %14;\n"
      "addc.cc.u32 %0, %0, %7;\n"
      "addc.cc.u32 %1, %1, %8;\n"
      "addc.cc.u32 %2, %2, %9;\n"
      "addc.cc.u32 %3, %3, %10;\n"
      "addc.cc.u32 %4, %4, %11;\n"
      "addc.cc.u32 %5, %5, %12;\n"
      "addc.u32 %6, %6, %13;\n" "}"
      : "+r"(T[0]), "+r"(T[1]), "+r"(T[2]), "+r"(T[3]), "+r"(T[4]), "+r"(T[5]), "+r"(T[6])
      : "r"(y[0]), "r"(y[1]), "r"(y[2]), "r"(y[3]), "r"(y[4]), "r"(y[5]), "r"(y[6]), "r"(s));
}
template <>
__device__ __forceinline__ void add_limbs32<8>(uint32_t (&T)[8], const uint32_t (&y)[8], uint32_t s) {
  asm("{\n" ".reg .u32 c;\n"
      "add.cc.u32 c, %16, %16;\n"
      "addc.cc.u32 %0, %0, %8;\n"
      "addc.cc.u32 %1, %1, %9;\n"
      "addc.cc.u32 %2, %2, %10;\n"
      "addc.cc.u32 %3, %3, %11;\n"
      "addc.cc.u32 %4, %4, %12;\n"
      "addc.cc.u32 %5, %5, %13;\n"
      "addc.cc.u32 %6, %6, %14;\n"
      "addc.u32 %7, %7, %15;\n" "}"
      : "+r"(T[0]), "+r"(T[1]), "+r"(T[2]), "+r"(T[3]), "+r"(T[4]), "+r"(T[5]), "+r"(T[6]), "+r"(T[7])
      : "r"(y[0]), "r"(y[1]), "r"(y[2]), "r"(y[3]), "r"(y[4]), "r"(y[5]), "r"(y[6]), "r"(y[7]), "r"(s));
}
template <>
__device__ __forceinline__ void add_limbs32<9>(uint32_t (&T)[9], const uint32_t (&y)[9], uint32_t s) {
  asm("{\n" ".reg .u32 c;\n"
      "add.cc.u32 c, %18, %18;\n"
      "addc.cc.u32 %0, %0, %9;\n"
      "addc.cc.u32 %1, %1, %10;\n"
      "addc.cc.u32 %2, %2, %11;\n"
      "addc.cc.u32 %3, %3, %12;\n"
      "addc.cc.u32 %4, %4, %13;\n"
      "addc.cc.u32 %5, %5, %14;\n"
      "addc.cc.u32 %6, %6, %15;\n"
      "addc.cc.u32 %7, %7, %16;\n"
      "addc.u32 %8, %8, %17;\n" "}"
      : "+r"(T[0]), "+r"(T[1]), "+r"(T[2]), "+r"(T[3]), "+r"(T[4]), "+r"(T[5]), "+r"(T[6]), "+r"(T[7]), "+r"(T[8])
      : "r"(y[0]), "r"(y[1]), "r"(y[2]), "r"(y[3]), "r"(y[4]), "r"(y[5]), "r"(y[6]), "r"(y[7]), "r"(y[8]), "r"(s));
}
template <>
__device__ __forceinline__ void add_limbs32<10>(uint32_t (&T)[10], const uint32_t (&y)[10], uint32_t s) {
  asm("{\n" ".reg .u32 c;\n"
      "add.cc.u32 c, %20, %20;\n"
      "addc.cc.u32 %0, %0, %10;\n"
      "addc.cc.u32 %1, %1, %11;\n"
      "addc.cc.u32 %2, %2, %12;\n"
      "addc.cc.u32 %3, %3, %13;\n"
      "addc.cc.u32 %4, %4, %14;\n"
      "addc.cc.u32 %5, %5, %15;\n"
      "addc.cc.u32 %6, %6, %16;\n"
      "addc.cc.u32 %7, %7, %17;\n"
      "addc.cc.u32 %8, %8, %18;\n"
      "addc.u32 %9, %9, %19;\n" "}"
      : "+r"(T[0]), "+r"(T[1]), "+r"(T[2]), "+r"(T[3]), "+r"(T[4]), "+r"(T[5]), "+r"(T[6]), "+r"(T[7]), "+r"(T[8]), "+r"(T[9])
      : "r"(y[0]), "r"(y[1]), "r"(y[2]), "r"(y[3]), "r"(y[4]), "r"(y[5]), "r"(y[6]), "r"(y[7]), "r"(y[8]), "r"(y[9]), "r"(s));
}
template <>
__device__ __forceinline__ void add_limbs32<12>(uint32_t (&T)[12], const uint32_t (&y)[12], uint32_t s) {
  asm("{\n" ".reg .u32 c;\n"
      "add.cc.u32 c, %24, %24;\n"
      "addc.cc.u32 %0, %0, %12;\n"
      "addc.cc.u32 %1, %1, %13;\n"
      "addc.cc.u32 %2, %2, %14;\n"
      "addc.cc.u32 %3, %3, %15;\n"
      "addc.cc.u32 %4, %4, %16;\n"
      "addc.cc.u32 %5, %5, %17;\n"
      "addc.cc.u32 %6, %6, %18;\n"
      "addc.cc.u32 %7, %7, %19;\n"
      "addc.cc.u32 %8, %8, %20;\n"
      "addc.cc.u32 %9, %9, %21;\n"
      "addc.cc.u32 %10, %10, %22;\n"
      "addc.u32 %11, %11, %23;\n" "}"
      : "+r"(T[0]), "+r"(T[1]), "+r"(T[2]), "+r"(T[3]), "+r"(T[4]), "+r"(T[5]), "+r"(T[6]), "+r"(T[7]), "+r"(T[8]), "+r"(T[9]), "+r"(T[10]), "+r"(T[11])
      : "r"(y[0]), "r"(y[1]), "r"(y[2]), "r"(y[3]), "r"(y[4]), "r"(y[5]), "r"(y[6]), "r"(y[7]), "r"(y[8]), "r"(y[9]), "r"(y[10]), "r"(y[11]), "r"(s));
}
// Fixed-point values: two's complement in NL 32-bit limbs.
// T += trunc(x 2^F): the magnitude (53 bits, cut below weight 1) takes three limbs
// from limb sh / 32 on; a barrel of selects over the bits of that limb index puts
// them in place, and a negative word adds the complement of every limb plus one
// (one carry chain either way, no branch on the sign).  Callers start T from the
// bias their digits need.
template <int NL>
__device__ __forceinline__ void add_word32(double x, int F, uint32_t (&T)[NL]) {
  const uint32_t bh = (uint32_t)__double2hiint(x), bl = (uint32_t)__double2loint(x);
  const int be = (int)((bh >> 20) & 0x7ffu);
  int sh = max(be, 1) - 1075 + F;                  // weight of the last mantissa bit
  uint64_t M = ((uint64_t)((bh & 0xFFFFFu) | (be ? 0x100000u : 0u)) << 32) | bl;
  asm("shr.b64 %0, %0, %1;" : "+l"(M) : "r"(max(-sh, 0)));   // zero from 64 bits on
  sh = max(sh, 0);
  uint32_t s = (uint32_t)((int32_t)bh >> 31);
  if (sh >= 32 * NL) {                             // only words the exponent does not cover
    M = 0;                                         // (non-finite input, flagged elsewhere)
    s = 0;
    sh = 0;
  }
  const uint32_t lo = (uint32_t)M, hi = (uint32_t)(M >> 32);
  const uint32_t v0 = (lo << (sh & 31)) ^ s, v1 = __funnelshift_l(lo, hi, sh) ^ s,
                 v2 = __funnelshift_l(hi, 0u, sh) ^ s;
  const bool b0 = sh & 32, b1 = sh & 64, b2 = sh & 128, b3 = sh & 256;
  uint32_t w[4] = {b0 ? s : v0, b0 ? v0 : v1, b0 ? v1 : v2, b0 ? v2 : s};
  uint32_t y[NL];
  auto at1 = [&](int i) { return i >= 0 && i < 4 ? w[i] : s; };
  auto at2 = [&](int i) { return i < 0 || i > 5 ? s : (b1 ? at1(i - 2) : at1(i)); };
  uint32_t q[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) q[i] = at2(i);
  uint32_t h[10];
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    const uint32_t plain = i < 6 ? q[i < 6 ? i : 0] : s, up = i >= 4 ? q[i >= 4 ? i - 4 : 0] : s;
    h[i] = NL > 4 ? (b2 ? up : plain) : plain;
  }
#pragma unroll
  for (int i = 0; i < NL; ++i) {
    const uint32_t plain = i < 10 ? h[i < 10 ? i : 0] : s, up = i >= 8 ? h[i >= 8 ? i - 8 : 0] : s;
    y[i] = NL > 8 ? (b3 ? up : plain) : plain;
  }
  add_limbs32<NL>(T, y, s);                        // carry in: one for a negative word
}

}  // namespace
}  // namespace mw

// Error-free transformations of double additions for kernels bound by the FP64
// pipe (device side): two_sum, fast_two_sum, two_prod.
//
// The FP64 pipe takes 2 lanes a clock and SM, the integer units 64 or more, so
// two_sum orders its operands by integer compares and then needs Dekker's three
// additions instead of Knuth's six: s = fl(a + b) and e = a + b - s exactly is
// the same pair either way.  What else Knuth's form returns is kept: a zero error
// is +0 (y + (x - s) with x - s = +0 is +0 also for y = -0) and a sum that is not
// finite has a NaN error.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

namespace mw {
namespace {

__device__ __forceinline__ double two_sum(double a, double b, double &e) {
  // exponent fields in the high words: |a|'s at least |b|'s is all Dekker's form needs
  const bool ordered = (uint32_t)(__double2hiint(a) << 1) >= (uint32_t)(__double2hiint(b) << 1);
  const double x = ordered ? a : b, y = ordered ? b : a;
  const double s = __dadd_rn(a, b);
  const double r = __dadd_rn(y, __dsub_rn(x, s));
  const bool finite = ((uint32_t)__double2hiint(s) & 0x7FF00000u) != 0x7FF00000u;
  e = __hiloint2double(finite ? __double2hiint(r) : 0x7FF80000, __double2loint(r));
  return s;
}
// Dekker: the same for |a| >= |b|.
__device__ __forceinline__ double fast_two_sum(double a, double b, double &e) {
  const double s = __dadd_rn(a, b);
  e = __dsub_rn(b, __dsub_rn(s, a));
  return s;
}
// p = fl(a b), e = a b - p exactly (one fused multiply-add; the same p and e as
// Dekker's splitting, which needs no fma).
__device__ __forceinline__ double two_prod(double a, double b, double &e) {
  const double p = __dmul_rn(a, b);
  e = __fma_rn(a, b, -p);
  return p;
}

}  // namespace
}  // namespace mw

// What the float64 block inverses share about a pivot: when it is usable, and
// its reciprocal without float64 instructions.
#pragma once

#include <cstdint>

namespace dm {

// not for pivot_recip: zero, below 2^-1022 (whose reciprocal overflows or is
// near it), at or above 2^1022 (whose reciprocal is not a normal number) or not
// finite
__device__ __forceinline__ bool pivot_unusable(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
  return b < 0x0010000000000000ull || b >= 0x7fd0000000000000ull;
}

// 1/x for a usable pivot x (2^-1022 <= |x| < 2^1022) in integer arithmetic,
// within 0.52 units in the last place.  x = X 2^(E - 52), X its 53-bit
// significand; Y 2^-24 = y0 ~ 2^52 / X from the float32 reciprocal of X's
// leading bits, relative error |h| < 2^-21.  The residual h = 1 - X y0 2^-52 =
// H 2^-76 is exact in the low 64 bits of X Y, and 1/X = y0 2^-52 (1 + h + h^2)
// up to h^3 (a Householder step of third order).  No float64 instruction: a
// third of the pivot chain would be the three a float64 refinement takes.
__device__ __forceinline__ double pivot_recip(double x) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(bits >> 52) & 0x7ff;
  const uint32_t xh = ((uint32_t)(bits >> 32) & 0xfffffu) | 0x100000u, xl = (uint32_t)bits;
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(0x3f800000u | (xh << 12 >> 9) | (xl >> 29))));
  const uint32_t rb = __float_as_uint(r);
  const uint32_t Y = ((rb & 0x7fffffu) | 0x800000u) << ((rb >> 23) - 126u & 1u);  // r in [1/2, 1]
  const unsigned long long XY = (unsigned long long)xl * Y + ((unsigned long long)(xh * Y) << 32);
  const long long H = (long long)(0ull - XY);  // 2^76 - X Y, |H| < 2^55
  const int Hh = (int)(H >> 24);
  const long long c = H + (((long long)Hh * Hh) >> 28);  // (h + h^2) 2^76
  const long long ch = c >> 16;                          // |ch| < 2^40
  const long long cy = (long long)(int)(ch >> 24) * (int)Y * (1ll << 24) + (long long)((uint32_t)ch & 0xffffffu) * Y;
  const unsigned long long y = ((unsigned long long)Y << 36) + (unsigned long long)(cy >> 24);  // 2^60 / (X 2^-52)
  const unsigned long long mant = (y + 64) >> 7;  // leading bit at 52, or 2^53
  return __longlong_as_double((long long)((bits & 0x8000000000000000ull) +
                                          ((unsigned long long)(2044 - ex) << 52) + mant));
}

// The same for every pivot that has a finite reciprocal, 0 for the others.
static __device__ __noinline__ double pivot_recip_any(double x) {
  const double r = 1.0 / x;
  return fabs(x) > 0.0 && isfinite(x) && isfinite(r) ? r : 0.0;
}

__device__ __forceinline__ uint32_t abs_hi(double v) { return (uint32_t)__double2hiint(v) & 0x7fffffffu; }

}  // namespace dm

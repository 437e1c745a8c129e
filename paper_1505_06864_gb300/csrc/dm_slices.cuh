// Exact digit slices of float64 values for products on the bf16 tensor
// cores (Ozaki's error-free splitting; the digit extraction from the float64
// bits is this library's), and the way back from their integer sums.
#pragma once

#include <cstdint>

namespace dm {

constexpr int kBalSlices = 7;

// Row pitch (elements) of the slices of an m x m block: 16-byte rows.
__host__ __device__ constexpr int slice_pitch(int m) { return (m + 7) & ~7; }

// v 2^(55 - e) rounded to the nearest integer (halves away from zero), |v| < 2^e.
__device__ __forceinline__ long long scaled_integer(unsigned long long bits, int e) {
  const int ex = (int)((bits >> 52) & 0x7ff);
  const unsigned long long mant = (bits & 0xfffffffffffffull) | (ex ? (1ull << 52) : 0ull);
  // (mant 8 >> n) / 2, rounded: |v| < 2^e leaves n >= 0, and from n = 56 on nothing is left
  // (nor of a subnormal v where e < -1021)
  const int n = (int)min((unsigned)(e + 1022 - (ex ? ex : 1)), 62u);
  const unsigned long long Y = (((mant << 3) >> n) + 1) >> 1;
  return (long long)((bits >> 63) ? 0ull - Y : Y);
}

// S balanced digits of v, |v| < 2^e, in base 2^8 (S = 7) or 2^7 (S = 8):
// v = 2^(e+1) sum_{s=1..S} d_s base^(-s), rounded to the nearest multiple of
// 2^(e-55), every d_s an integer of at most base / 2 in magnitude and so exact
// in bf16 (bit patterns in the high half of each word, the low half ignored).
// Integer and float32 operations only: a digit d < 2^23 becomes the float d
// exactly as (2^23 + d) - 2^23, and a float with at most 8 significant bits is
// its own bf16 truncation.  The
// scaled integer is biased by base / 2 in every digit, so that each digit is a
// bit field minus base / 2.  NaN or infinity: the first digit is NaN, the
// others finite.
template <int S>
__device__ __forceinline__ void digits(unsigned long long bits, int e, uint32_t (&q)[S]) {
  static_assert(S == 7 || S == 8, "base 2^8 or 2^7");
  const long long Y = scaled_integer(bits, e);
  if constexpr (S == 7) {
    const unsigned long long Z = (unsigned long long)Y + 0x0080808080808080ull;
    const uint32_t hi = (uint32_t)(Z >> 32), lo = (uint32_t)Z;
    const uint32_t w[7] = {0x4b000000u | (hi >> 16),
                           __byte_perm(hi, 0x4b000000u, 0x7541),
                           __byte_perm(hi, 0x4b000000u, 0x7540),
                           __byte_perm(lo, 0x4b000000u, 0x7543),
                           __byte_perm(lo, 0x4b000000u, 0x7542),
                           __byte_perm(lo, 0x4b000000u, 0x7541),
                           __byte_perm(lo, 0x4b000000u, 0x7540)};
#pragma unroll
    for (int k = 0; k < 7; ++k) q[k] = __float_as_uint(__uint_as_float(w[k]) - 8388736.0f);
  } else {
    const unsigned long long Z = (unsigned long long)Y + 0x0081020408102040ull;  // 64 in every 7-bit digit
    const uint32_t hi = (uint32_t)(Z >> 32), lo = (uint32_t)Z;
    const uint32_t mid = __funnelshift_r(lo, hi, 28);  // bits 28 .. 59
    const uint32_t w[8] = {hi >> 17,          (hi >> 10) & 127u, (hi >> 3) & 127u, (mid >> 0) & 127u,
                           (lo >> 21) & 127u, (lo >> 14) & 127u, (lo >> 7) & 127u, lo & 127u};
#pragma unroll
    for (int k = 0; k < 8; ++k) q[k] = __float_as_uint(__uint_as_float(0x4b000000u | w[k]) - 8388672.0f);
  }
  if ((bits >> 52 & 0x7ff) == 0x7ff) q[0] = 0x7fc00000u;
}

// T 2^s rounded to float64 (to nearest, halves up), |T| < 2^63, by integer
// operations; `odd` is set when the result is outside the normal range (then
// the value is not the result).
__device__ __forceinline__ double round_scaled(long long T, int s, bool& odd) {
  const unsigned long long a = (unsigned long long)(T < 0 ? -T : T);
  const int lz = __clzll(a);
  const unsigned long long an = a << (lz & 63);                   // leading bit at 63
  const unsigned long long mant = (an >> 11) + ((an >> 10) & 1);  // leading bit at 52 (or 2^53)
  const int ex = 1022 + 63 - lz + s;                              // the leading bit adds one to the exponent
  odd = odd || (a != 0 && (unsigned)ex > 2044u);
  const unsigned long long r = ((unsigned long long)T & 0x8000000000000000ull) + ((unsigned long long)ex << 52) + mant;
  return __longlong_as_double(a == 0 ? 0ll : (long long)r);
}

// v 2^k exactly (rounded where the result is subnormal), without float64
// instructions while it is a normal number.
__device__ __forceinline__ double scale_pow2(double v, int k) {
  const int hi = __double2hiint(v), lo = __double2loint(v), ex = (hi >> 20) & 0x7ff;
  if ((unsigned)(ex - 1) < 2046u && (unsigned)(ex + k - 1) < 2046u) return __hiloint2double(hi + k * (1 << 20), lo);
  return ((hi << 1) | lo) == 0 ? v : ldexp(v, k);
}

// Two bf16 values (high halves of a and b) in one register, a first.
__device__ __forceinline__ uint32_t pack_hi(uint32_t a, uint32_t b) { return __byte_perm(a, b, 0x7632); }

// Exponent e with |v| < 2^e for every v whose high word (sign cleared) is at
// most hmax; subnormal or zero maxima share e = -1021.
__device__ __forceinline__ int scale_exponent(uint32_t hmax) {
  const int E = (int)(hmax >> 20);
  return E == 0 ? -1021 : E - 1022;
}

// Key of the high word of an entry with shift s: keys are compared, and an
// entry of key K is below 2^(K - 1022).
constexpr int kNoKey = -(1 << 20);
__device__ __forceinline__ int scale_key(uint32_t hi, int s) {
  const int h = (int)(hi & 0x7fffffffu);
  return h == 0 ? kNoKey : max(h >> 20, 1) + s;
}
__device__ __forceinline__ int key_exponent(int key) { return key == kNoKey ? 0 : key - 1022; }

}  // namespace dm

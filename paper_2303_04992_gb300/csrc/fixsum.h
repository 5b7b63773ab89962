// Sums of binary64 values by 64-bit integer arithmetic, for stencils on a GPU
// whose FP64 pipe (two lanes per SM and cycle) is the bound: every value is
// aligned to the largest exponent among them (58 significant bits below it,
// truncated: within 2^-57 of the largest value, sixteen times finer than a
// binary64 rounding of it), the sum is exact, and its conversion back is
// rounded to nearest even.
//
// Plain C++ (host and device): the CPU test suite compiles this header with
// g++ and compares the sums with long-double ones.
#pragma once

#include "fastcvt.h"

namespace kfbim {

// Biased exponent of a binary64 encoding.
KFBIM_CVT_HD int fix_exp(uint64_t b) { return (int)((b >> 52) & 0x7ffu); }

// The largest biased exponent, and kFixMin at least, as fix_of and fix_value take it:
// it starts there.  Below it (values under 1e-289) the unit no longer shrinks.
constexpr int kFixMin = 64;

// The value of encoding b in units of 2^(E - 1080), E >= its biased exponent and
// E >= kFixMin: |result| < 2^58.  A zero's shift is 63, which leaves nothing.
KFBIM_CVT_HD int64_t fix_of(uint64_t b, int E) {
  const int sh = E - fix_exp(b);
  const uint64_t m = (((b & 0xfffffffffffffull) | 0x10000000000000ull) << 5) >> (sh < 63 ? sh : 63);
  const uint64_t s = (uint64_t)((int64_t)b >> 63);
  return (int64_t)((m ^ s) - s);
}

KFBIM_CVT_HD int fix_clz(uint64_t a) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)a);
#else
  return __builtin_clzll(a);
#endif
}

// S 2^(E - 1080) rounded to nearest even (|S| < 2^63).  E = 2047, the exponent of
// infinities and NaN, gives NaN; results below the normal range give zero.
KFBIM_CVT_HD double fix_value(int64_t S, int E) {
  if (E == 2047) return cvt_from_bits64(0x7ff8000000000000ull);
  if (S == 0) return 0.0;
  const uint64_t sign = (uint64_t)S & 0x8000000000000000ull;
  uint64_t a = S < 0 ? (uint64_t)(-S) : (uint64_t)S;
  const int lz = fix_clz(a);
  a <<= lz;                                         // in [2^63, 2^64)
  const uint64_t rest = a & 0x7ffu;
  uint64_t m = a >> 11;                             // 53 bits, the leading one included
  m += (rest > 0x400u || (rest == 0x400u && (m & 1u))) ? 1u : 0u;
  const int e = E + 6 - lz;                         // biased exponent of the leading one
  if (e <= 0) return cvt_from_bits64(sign);
  if (e >= 2047) return cvt_from_bits64(sign | 0x7ff0000000000000ull);
  // the leading one adds one to the exponent field, as does a carry out of the rounding
  return cvt_from_bits64(sign | (((uint64_t)(e - 1) << 52) + m));
}

}  // namespace kfbim

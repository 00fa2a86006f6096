// Fixed-point trigonometric values and exact sums of their products with integers.
#pragma once

#include <cstdint>

namespace ilg {

// A 128-bit integer as the record holds it.
struct I128 {
  unsigned long long lo = 0;
  long long hi = 0;
};

// v * 2^-62 rounded once to double (round to nearest even).
__device__ inline double i128_to_double_2m62(I128 v) {
  const bool neg = v.hi < 0;
  unsigned long long lo = v.lo, hi = (unsigned long long)v.hi;
  if (neg) {  // two's complement negation
    lo = ~lo + 1ull;
    hi = ~hi + (lo == 0 ? 1ull : 0ull);
  }
  double mag;
  if (hi == 0) {
    mag = __ull2double_rn(lo);
  } else {
    // keep the top 64 bits, fold the rest into a sticky bit: one correct rounding
    const int k = 64 - __clzll((long long)hi);  // significant bits of hi, 1..64
    unsigned long long m = k == 64 ? hi : ((hi << (64 - k)) | (lo >> k));
    const unsigned long long dropped = k == 64 ? lo : (lo << (64 - k));
    if (dropped) m |= 1ull;
    mag = ldexp(__ull2double_rn(m), k);
  }
  const double r = ldexp(mag, -62);
  return neg ? -r : r;
}

// 2^62 v rounded to the nearest integer (|v| <= 1).
__device__ __forceinline__ long long fixed62(double v) { return __double2ll_rn(v * 4611686018427387904.0); }

}  // namespace ilg

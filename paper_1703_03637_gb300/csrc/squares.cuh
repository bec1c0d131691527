// Sum of the squares of a few fp32 values as fp64, in integer arithmetic.
//
// In fp64 each value would cost a conversion and a multiply-add, at 1/64 of the fp32 rate.
// Instead the 24-bit significands are squared as integers (exact, 48 bits), aligned to the
// group's largest exponent in 64 bits and added; the group then takes one conversion and one
// exact power-of-two scale.  The largest square stands at 2^58 or above, so what the alignment
// drops is below 2^-58 of it per value: the conversion's rounding, 2^-53, is the only other one,
// where the fp64 sum rounds once per value.  Groups with an infinity or NaN, or whose values are
// all below 2^-63 (their subnormals count), take the fp64 sum.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#include "gauss.cuh"

namespace hphi {

HPHI_HD uint32_t float_bits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t b;
  memcpy(&b, &x, 4);
  return b;
#endif
}

template <int N>
HPHI_HD double sum_squares(const float* x) {
  static_assert(N >= 1 && N <= 8, "the sum of N squares below 2^60 must fit 63 bits");
  constexpr uint32_t kExp = 0x7f800000u;
  uint32_t top = 0;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const uint32_t e = float_bits(x[k]) & kExp;
    top = e > top ? e : top;
  }
  if (top >= (64u << 23) && top != kExp) {
    int64_t s = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const uint32_t b = float_bits(x[k]);
      const uint32_t d = (top - (b & kExp)) >> 22;  // twice the exponent's distance from the largest
      const uint64_t m = ((b << 6) & 0x1fffffc0u) | 0x20000000u;  // significand << 6 (zero, subnormal: d > 63)
      s += (int64_t)((m * m) >> (d < 63u ? d : 63u));
    }
    return int_to_double(s) * pow2_double(2 * (int)(top >> 23) - 312);
  }
  double s = 0.0;
#pragma unroll 1
  for (int k = 0; k < N; ++k) s = fma((double)x[k], (double)x[k], s);
  return s;
}

}  // namespace hphi

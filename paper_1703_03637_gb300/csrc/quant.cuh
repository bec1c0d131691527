// The fixed point of the fp64 gather paths: one rounding for every kernel that writes a copy.
#pragma once

#include <stdint.h>
#include <string.h>

#include "gauss.cuh"

namespace hphi {

// q = round(x 2^(1078 - E)), halves away from zero, by integer operations on the bits of x; |q| < 2^56
// when the exponent field of x is at most E.  Subnormals give zero.
HPHI_HD long long quant_one(double x, int E) {
#ifdef __CUDA_ARCH__
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
#else
  uint64_t bits;
  memcpy(&bits, &x, 8);
  const int hi = (int)(uint32_t)(bits >> 32);
  const unsigned lo = (unsigned)bits;
#endif
  const int ex = (hi >> 20) & 0x7ff;
  long long q = 0;
  if (ex != 0) {
    const long long M = ((long long)((hi & 0xfffff) | 0x100000) << 32) | (long long)lo;  // x = M 2^(ex-1075)
    const int sh = E - ex - 3;                                                           // q = M 2^-sh
    if (sh <= 0) q = M << (-sh);
    else if (sh < 62) q = (M + (1ll << (sh - 1))) >> sh;
    if (hi < 0) q = -q;
  }
  return q;
}

}  // namespace hphi

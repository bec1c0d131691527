// Box-Muller pairs from two 53-bit integers in integer arithmetic.
//
// GB300 issues fp64 at 1/64 of its integer rate, so the transform's logarithm, square root,
// sine and cosine run in 64-bit fixed point (high halves of 64 x 64-bit products) and only
// the last step, one conversion and one exact power-of-two scale per number, is fp64.  With
// u_a = A / 2^54 and u_b = B / 2^54 taken exactly:
//   -ln u_a   u_a = m 2^-n, m in [1, 2]; a table of reciprocals rc_j / 1024 of m's 257 nearest
//             centres makes r = m rc_j / 1024 - 1 an exact integer, |r| < 2^-8.6, and
//             -ln u_a = n ln 2 - ln(1024 / rc_j) - ln(1 + r), the last by its Taylor series
//             to r^7.  For u_a next to 1 the first two terms cancel exactly and the series is
//             taken on a normalised r, so the result keeps its relative accuracy.
//   sqrt      two Newton steps from the fp32 reciprocal square root
//   cos, sin  the nearest of 256 table angles, the Taylor series of the remaining angle
//             |phi| <= pi / 256 (to phi^7 and phi^6) and one rotation; next to an axis the small
//             component is sin phi on a normalised angle
// A result is within 3 2^-53 of the exact transform of (u_a, u_b), relative to itself: one
// rounding, 2^-53 where the logarithm's three terms nearly cancel (-ln u_a near 2^-10) and 2^-60
// of the radius from the rotation, whose components are at least pi / 256.
// Bound by integer issue.  Measured on GB300, 155,117,520 fp64 elements: 1.7 ms, against
// 10.4 ms with fp64 log, sqrt and sincospi (the floor of its writes is 0.19 ms).
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define HPHI_HD __host__ __device__ __forceinline__
#else
#define HPHI_HD inline
#endif

namespace hphi {

// ------------------------------------------------------------------ tables (compile time)
struct GaussTables {
  uint64_t lnc[257];    // ln(1024 / rc_j), Q63
  int64_t cs[256][2];   // cos, sin of 2 pi i / 256, Q62
  uint32_t rc[257];     // round(1024 / (1 + j / 256))
};

namespace gauss_detail {
using u128 = unsigned __int128;

// ln(1024 / rc) = 2 atanh(t), t = (1024 - rc) / (1024 + rc) <= 1/3, in Q100; rounded to Q63
constexpr uint64_t ln_entry(unsigned rc) {
  const u128 p = 1024 - rc, q = 1024 + rc;
  u128 pw = (p << 100) / q, sum = 0;
  for (unsigned k = 1; pw != 0; k += 2) {
    sum += pw / k;
    pw = pw * (p * p) / (q * q);
  }
  return (uint64_t)((2 * sum + ((u128)1 << 36)) >> 37);
}

constexpr u128 mul100(u128 a, u128 b) {  // Q100 product of values below 2
  const u128 m = ((u128)1 << 50) - 1, a1 = a >> 50, a0 = a & m, b1 = b >> 50, b0 = b & m;
  return a1 * b1 + ((a1 * b0 + a0 * b1) >> 50) + ((a0 * b0) >> 100);
}

// sin (odd) or cos of i pi / 128, 0 <= i <= 32, by Taylor series in Q100; rounded to Q62
constexpr int64_t trig_entry(unsigned i, bool sine) {
  const u128 pi = ((u128)0x3243F6A8885A3ull << 52) | 0x08D313198A2E0ull;  // 3.243F6A88... in Q100
  const u128 x = pi * i / 128, x2 = mul100(x, x);
  u128 t = sine ? x : (u128)1 << 100, pos = 0, neg = 0;
  for (unsigned k = sine ? 1 : 0, n = 0; t != 0; k += 2, ++n) {
    if (n & 1) neg += t;
    else pos += t;
    t = mul100(t, x2) / ((k + 1) * (k + 2));
  }
  return (int64_t)((pos - neg + ((u128)1 << 37)) >> 38);
}

constexpr GaussTables make_tables() {
  GaussTables g{};
  for (unsigned j = 0; j <= 256; ++j) {
    g.rc[j] = (2 * 1024 * 256 + (256 + j)) / (2 * (256 + j));
    g.lnc[j] = ln_entry(g.rc[j]);
  }
  for (unsigned i = 0; i < 256; ++i) {
    const unsigned oct = i / 32, k = i % 32;  // octant and angle inside it
    const int64_t c = trig_entry((oct & 1) ? 32 - k : k, false), s = trig_entry((oct & 1) ? 32 - k : k, true);
    const int64_t x = ((oct + 1) & 2) ? s : c, y = ((oct + 1) & 2) ? c : s;
    g.cs[i][0] = (oct >= 2 && oct < 6) ? -x : x;
    g.cs[i][1] = (oct >= 4) ? -y : y;
  }
  return g;
}
}  // namespace gauss_detail

// ------------------------------------------------------------------ arithmetic
HPHI_HD uint64_t mulhi_u(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
HPHI_HD int64_t mulhi_s(int64_t a, int64_t b) {
#ifdef __CUDA_ARCH__
  return __mul64hi(a, b);
#else
  return (int64_t)(((__int128)a * b) >> 64);
#endif
}
HPHI_HD uint32_t mulhi32(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
HPHI_HD int32_t mulhi32_s(int32_t a, int32_t b) { return (int32_t)(((int64_t)a * b) >> 32); }
HPHI_HD int clz64(uint64_t x) {  // x != 0
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return __builtin_clzll(x);
#endif
}
HPHI_HD float rsqrt32(float x) {
#ifdef __CUDA_ARCH__
  return rsqrtf(x);
#else
  return 1.0f / sqrtf(x);
#endif
}
HPHI_HD double int_to_double(int64_t x) {
#ifdef __CUDA_ARCH__
  return __ll2double_rn(x);
#else
  return (double)x;
#endif
}
HPHI_HD double pow2_double(int e) {
  const int64_t b = (int64_t)(e + 1023) << 52;
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double d;
  memcpy(&d, &b, 8);
  return d;
#endif
}

// k + 1/2 as fp64 rounds it (ties to even), times 2: the numerator A of u = A / 2^54
HPHI_HD uint64_t gauss_numerator(uint64_t k) {
  return k < (1ull << 52) ? 2 * k + 1 : 2 * (k + (k & 1));
}

// sqrt(-2 ln(A / 2^54)) = rad 2^-62 2^ex, rad in [2^62, 2^63) (0 for A = 2^54)
HPHI_HD uint64_t gauss_radius(uint64_t A, const GaussTables& t, int& ex) {
  if (A >> 54) {  // u = 1: no logarithm to normalise
    ex = 0;
    return 0;
  }
  const int nz = clz64(A);
  const int n = nz - 9;                                    // u = m 2^-n, m = M / 2^53 in [1, 2)
  const uint64_t M = A << (nz - 10);
  const uint32_t j = ((uint32_t)(M >> 44) + 1) / 2 - 256;  // nearest centre 1 + j / 256
  const int64_t r0 = (int64_t)(M * t.rc[j] - (1ull << 63));  // r, Q63, exact
  const int64_t r = r0 * 128;                              // Q70
  const int32_t r32 = (int32_t)((r + (1ll << 31)) >> 32);  // Q38
  // ln(1 + r) = r - r^2 h2, h2 = 1/2 - r h3, h3 = 1/3 - r h4, h4 = 1/4 - r (1/5 - r (1/6 - r / 7))
  int32_t h = 357913941 - (mulhi32_s(r32, 306783378) >> 6);  // 1/6 - r / 7, Q31
  h = 429496730 - (mulhi32_s(r32, h) >> 6);                  // Q31
  h = 1073741824 - (mulhi32_s(r32, h) >> 5);                 // h4, Q32
  const int64_t h3 = 1537228672809129301ll - (((int64_t)r32 * h) >> 8);  // Q62
  const int64_t h2 = (1ll << 62) - (mulhi_s(r, h3) >> 5);                // Q63
  const int64_t g = mulhi_s(r, h2);                                      // r h2, Q69
  uint64_t X;  // -ln u = X 2^-q
  int q;
  if (n == 1 && j == 256) {  // n ln 2 - ln c_j = 0 and r < 0
    const int s = clz64((uint64_t)(-r0)) - 1;
    const int64_t rn = -r0 * (int64_t)(1ull << s);  // |r|, Q(63 + s), below 2^63
    X = (uint64_t)rn + (uint64_t)(mulhi_s(rn, -g) >> 5);
    q = 63 + s;
  } else {
    const int64_t L = r - (mulhi_s(r, g) >> 5);  // ln(1 + r), Q70
    const int sft = n > 1 ? 64 - clz64((uint64_t)(n - 1)) : 0;  // keeps X below 2^63
    X = (uint64_t)n * (t.lnc[256] >> sft) - (t.lnc[j] >> sft) - (uint64_t)(L >> (7 + sft));
    q = 63 - sft;
  }
  // 2 X 2^-q = w 2^-62 4^k with w in [2^62, 2^64)
  const int z = clz64(X);
  const int e2 = 64 - z - q;                        // 2 X 2^-q = (X << z) 2^-63 2^e2
  const uint64_t w = (X << z) >> ((e2 & 1) ? 0 : 1);  // odd: [2, 4) in Q62, else [1, 2)
  ex = (e2 - (e2 & 1)) / 2;
  const float y = rsqrt32((float)(uint32_t)(w >> 32) * (1.0f / 1073741824.0f));
  const uint32_t Y = (uint32_t)fminf(y * 4294967296.0f, 4294967040.0f);  // 1 / sqrt(w), Q32
  uint64_t s = mulhi_u(w, (uint64_t)Y << 32);       // Q62
  int64_t d = (int64_t)((w >> 2) - mulhi_u(s, s));  // w - s^2, Q60
  s += (uint64_t)(mulhi_s(d, (int64_t)((uint64_t)Y << 31)) * 4);  // + d y / 2
  d = (int64_t)((w >> 2) - mulhi_u(s, s));
  s += (uint64_t)((d * (int64_t)(Y >> 2)) >> 29);   // |d| < 2^20 now
  return s;
}

// cos and sin of 2 pi B / 2^54: c 2^-(62 + kc), s 2^-(62 + ks).  Next to an axis (a table angle
// that is a multiple of a quarter turn) the small one is sin phi itself, taken on the normalised
// angle so that it keeps its relative accuracy (kc or ks > 0).
HPHI_HD void gauss_direction(uint64_t B, const GaussTables& t, int64_t& c, int64_t& s, int& kc, int& ks) {
  const uint64_t th = B << 10;  // turns, Q64
  const uint32_t i = (uint32_t)((th + (1ull << 55)) >> 56) & 255u;
  const int64_t d = (int64_t)(th - ((uint64_t)i << 56));       // turns, Q64, |d| <= 2^55
  const int64_t f = mulhi_s(d * 256, 7244019458077122843ll);   // phi = 2 pi d, Q68
  const uint64_t fa = (uint64_t)(f < 0 ? -f : f);
  const uint64_t z = mulhi_u(fa * 4, fa * 4);                  // phi^2, Q76
  const uint32_t z32 = (uint32_t)(z >> 32);                    // Q44
  // sin phi = phi (1 - P), P = phi^2 (1/6 - phi^2 / 120 + phi^4 / 5040)
  const uint32_t v = mulhi32(z32, 2290649225u - mulhi32(z32, 13315u));               // Q50
  const uint64_t P = mulhi_u(z, 3074457345618258603ull - ((uint64_t)v << 14));       // Q76
  const uint64_t fp = mulhi_u(fa, P) >> 12;                                          // Q68
  const int64_t sp = f - (f < 0 ? -(int64_t)fp : (int64_t)fp);                       // sin phi, Q68
  // cos phi = 1 - C, C = phi^2 (1/2 - phi^2 / 24 + phi^4 / 720)
  const uint32_t v2 = mulhi32(z32, 2863311531u - mulhi32(z32, 23302u));              // Q48
  const int64_t C = (int64_t)(mulhi_u(z, (1ull << 63) - ((uint64_t)v2 << 16)) >> 1);  // Q75
  const int64_t ci = t.cs[i][0], si = t.cs[i][1];
  c = ci - (((mulhi_s(ci, C) >> 7) + mulhi_s(si, sp)) >> 4);
  s = si - (((mulhi_s(si, C) >> 7) - mulhi_s(ci, sp)) >> 4);
  kc = 0;
  ks = 0;
  if ((i & 63u) == 0 && d != 0) {
    const uint64_t da = (uint64_t)(d < 0 ? -d : d);
    const int k = clz64(da) - 1;
    const uint64_t F = mulhi_u(da << k, 14488038916154245685ull);  // |phi|, Q(61 + k): pi / 4 in Q64
    const int64_t w = (int64_t)(F - (mulhi_u(F, P) >> 12));        // |sin phi|, Q(61 + k)
    // sine of 0 + phi, -sine of 1/2 + phi, -cosine of 1/4 + phi, cosine of 3/4 + phi (in turns)
    const bool neg = (d < 0) != (i == 64 || i == 128);
    if (i & 64u) {
      c = neg ? -w : w;
      kc = k - 1;
    } else {
      s = neg ? -w : w;
      ks = k - 1;
    }
  }
}

// g0 = sqrt(-2 ln u_a) cos(2 pi u_b), g1 = sqrt(-2 ln u_a) sin(2 pi u_b), u = (k + 1/2) / 2^53
HPHI_HD void gauss_pair(uint64_t a, uint64_t b, const GaussTables& t, double& g0, double& g1) {
  int ex;
  const uint64_t rad = gauss_radius(gauss_numerator(a), t, ex);
  int64_t c, s;
  int kc, ks;
  gauss_direction(gauss_numerator(b), t, c, s, kc, ks);
  g0 = int_to_double(mulhi_s((int64_t)rad, c)) * pow2_double(ex - 60 - kc);
  g1 = int_to_double(mulhi_s((int64_t)rad, s)) * pow2_double(ex - 60 - ks);
}

}  // namespace hphi

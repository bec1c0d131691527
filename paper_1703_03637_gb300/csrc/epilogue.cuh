// Helpers shared by the H v kernels: per-column CTA reductions, element access, the exact
// fixed-point accumulator for fp64 gather sums and the fused Lanczos / mTPQ epilogues.
#pragma once

#include "common.cuh"
#include "reduce.cuh"

namespace hphi {

// Per-column CTA reduction in a fixed tree order; partials[(block * nvec + c) * kMaxRedQ + q].
// NT is the CTA size; sm holds NT * kMaxRedQ doubles.
template <bool F64, int NT = kThreads, int NQ = kMaxRedQ>
__device__ void block_finish(const Red<F64, NQ>& red, int nq, int nvec, double* __restrict__ partials, double* sm) {
  const int tid = threadIdx.x;
  for (int q = 0; q < nq; ++q) sm[q * NT + tid] = red.get(q);
  __syncthreads();
  for (int off = NT / 2; off >= nvec; off >>= 1) {
    if (tid < off) {
      for (int q = 0; q < nq; ++q) sm[q * NT + tid] += sm[q * NT + tid + off];
    }
    __syncthreads();
  }
  if (tid < nvec) {
    for (int q = 0; q < nq; ++q) partials[((size_t)blockIdx.x * nvec + tid) * kMaxRedQ + q] = sm[q * NT + tid];
  }
}

// ------------------------------------------------------------------ element access
template <class S>
__device__ __forceinline__ void ld(const S* __restrict__ p, int64_t i, typename Traits<S>::R& re,
                                   typename Traits<S>::R& im) {
  if constexpr (Traits<S>::kCplx) {
    const S x = p[i];
    re = x.x;
    im = x.y;
  } else {
    re = p[i];
    im = 0;
  }
}

template <class S>
__device__ __forceinline__ void st(S* __restrict__ p, int64_t i, typename Traits<S>::R re, typename Traits<S>::R im) {
  if constexpr (Traits<S>::kCplx) {
    S x;
    x.x = re;
    x.y = im;
    p[i] = x;
  } else {
    p[i] = re;
  }
}

// m * 2^eoff rounded to nearest even: the hardware int64 -> fp64 conversion (round to
// nearest even) and an exact power-of-two scale.  Measured on GB300, this runs three
// times faster than assembling the result's bits with 64-bit integer operations.
__device__ __forceinline__ double fix_to_double(long long m, int eoff) {
  const double d = __ll2double_rn(m);
  if (eoff >= -1022 && eoff <= 1023) return d * __longlong_as_double((long long)(eoff + 1023) << 52);
  return ldexp(d, eoff);
}

// a 128-bit integer as the nearest-ish fp64 (two roundings: relative error below 2^-52)
__device__ __forceinline__ double i128_to_double(__int128 v) {
  const long long hi = (long long)(v >> 64);
  const unsigned long long lo = (unsigned long long)v;
  return fma(__ll2double_rn(hi), 18446744073709551616.0, __ull2double_rn(lo));
}

// 4- or 8-byte asynchronous copy to shared memory, and 16-byte ones past L1
template <int B>
__device__ __forceinline__ void copy_async(void* dst, const void* src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  if constexpr (B == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(B) : "memory");
}

// ------------------------------------------------------------------ gather sums
// fp64 terms are summed in an exact-alignment fixed-point accumulator: every term's
// 53-bit significand is shifted to the running largest exponent and added as a 64-bit
// integer (2 guard bits), so the sum runs on the integer pipes, which GB300 issues at 64x
// the fp64 rate.  Truncation below the grid 2^(e_max - 1077) costs at most one unit per
// term, i.e. <= n 2^-54 |largest term|, the same order as fp64 summation's error bound.
// Terms below 2^-1022 (subnormals) are dropped.
struct FixAcc {
  long long m;   // signed sum of aligned significands, units of 2^(e - 1077)
  int e;         // biased exponent of the largest term so far (0: empty)
  int n;         // terms since the last overflow flush
  double spill;  // flushed part (only after 128 terms)
  bool sp;       // spill holds something
  __device__ __forceinline__ void zero() { m = 0; e = 0; n = 0; spill = 0.0; sp = false; }
  __device__ __forceinline__ double value() const {
    const double r = fix_to_double(m, e - 1077);
    return sp ? r + spill : r;
  }
  __device__ __forceinline__ void add(double x, bool neg) {
    const int hi = __double2hiint(x);
    const unsigned lo = (unsigned)__double2loint(x);
    const int ex = (hi >> 20) & 0x7ff;
    if (ex == 0) return;
    if (++n == 128) {  // keep |m| < 2^63: 127 terms of < 2^55 each
      spill = value();
      sp = true;
      m = 0;
      e = 0;
      n = 1;
    }
    long long mant = ((long long)((hi & 0xfffff) | 0x100000) << 34) | ((long long)lo << 2);
    if (ex > e) {
      const int d = ex - e;
      m = (d >= 63) ? 0 : (m >> d);
      e = ex;
    }
    const int sh = e - ex;
    mant = (sh >= 63) ? 0 : (mant >> sh);
    if ((hi < 0) != neg) m -= mant;
    else m += mant;
  }
};

struct F32Acc {
  float s;
  __device__ __forceinline__ void zero() { s = 0.f; }
  __device__ __forceinline__ float value() const { return s; }
  __device__ __forceinline__ void add(float x, bool neg) { s += neg ? -x : x; }
};

// exact sums of 64-bit fixed-point terms (the quantised fp64 path; no overflow below
// 128 terms of magnitude < 2^56)
struct IntAcc {
  long long s;
  __device__ __forceinline__ void zero() { s = 0; }
  __device__ __forceinline__ long long value() const { return s; }
  __device__ __forceinline__ void add(long long x, bool neg) { s += neg ? -x : x; }
};

template <class R> struct SumAcc;
template <> struct SumAcc<double> { using T = FixAcc; };
template <> struct SumAcc<float> { using T = F32Acc; };
template <> struct SumAcc<long long> { using T = IntAcc; };

// (ar, ai) += phase(code) * (xr, xi), code: 1 (+1), 2 (+i), 3 (-1), 4 (-i)
template <class A, class R>
__device__ __forceinline__ void acc_phase(int code, R xr, R xi, A& ar, A& ai) {
  switch (code) {
    case 1: ar.add(xr, false); ai.add(xi, false); break;
    case 2: ar.add(xi, true); ai.add(xr, false); break;
    case 3: ar.add(xr, true); ai.add(xi, true); break;
    default: ar.add(xi, false); ai.add(xr, true); break;
  }
}

// ------------------------------------------------------------------ epilogues
// The scalars of a fused step in the vectors' precision, converted once per thread: the opaque
// copy keeps the compiler from converting the kernel's fp64 arguments again for every element
// (three fp64-pipe conversions an element in the fp32 mTPQ step, at 1/64 of the fp32 rate).
template <class R>
__device__ __forceinline__ R opaque(R x) {
  if constexpr (sizeof(R) == 8) asm volatile("" : "+d"(x));
  else asm volatile("" : "+f"(x));
  return x;
}

template <class R>
struct EpiScalars {
  R c1, c2;  // Lanczos pass 1; c1: the shift c
  R l, ins;  // mTPQ: l and 1 / N_s
};

template <class R, Epi E>
__device__ __forceinline__ EpiScalars<R> epi_scalars(const FusedArgs& fa) {
  EpiScalars<R> es{(R)0, (R)0, (R)0, (R)0};
  if constexpr (E == Epi::kLanczos1) {
    es.c1 = opaque((R)fa.scal[0]);
    es.c2 = opaque((R)fa.scal[1]);
  } else if constexpr (E == Epi::kShift) {
    es.c1 = opaque((R)fa.scal[0]);
  } else if constexpr (E == Epi::kTpq) {
    es.l = opaque((R)fa.l);
    es.ins = opaque((R)fa.inv_ns);
  }
  return es;
}

// inv: 1 / |X_k| of this column (mTPQ only)
template <class S, Epi E, int NQ = kMaxRedQ>
__device__ __forceinline__ void epilogue(int64_t idx, typename Traits<S>::R sr, typename Traits<S>::R si,
                                         typename Traits<S>::R hr, typename Traits<S>::R hi, S* __restrict__ w,
                                         const FusedArgs& fa, const EpiScalars<typename Traits<S>::R>& es,
                                         typename Traits<S>::R inv, Red<Traits<S>::kF64, NQ>& red) {
  using R = typename Traits<S>::R;
  constexpr bool C = Traits<S>::kCplx;
  if constexpr (E == Epi::kStore) {
    st<S>(w, idx, hr, hi);
  } else if constexpr (E == Epi::kLanczos1) {
    // P <- sigma_k * (H C) - beta_k sigma_{k-1} * P ;  partial <C, H C>
    S* P = reinterpret_cast<S*>(fa.out);
    const S* Pin = fa.in ? reinterpret_cast<const S*>(fa.in) : P;
    R pr, pi;
    ld<S>(Pin, idx, pr, pi);
    st<S>(P, idx, es.c1 * hr - es.c2 * pr, es.c1 * hi - es.c2 * pi);
    red.add(0, sr, hr);
    if constexpr (C) red.add(0, si, hi);
    red.tick();
  } else if constexpr (E == Epi::kTpq) {
    // X_{k+1} = (l X_k - H X_k / N_s) / |X_k| ; partials <X, HX>, |HX|^2.  |X_{k+1}|^2 follows
    // from them (section 3.5's norm, deferred): l^2 - 2 l u_k + <H^2>_k.
    S* Xn = reinterpret_cast<S*>(fa.out);
    const R nr = inv * (es.l * sr - hr * es.ins);
    const R ni = inv * (es.l * si - hi * es.ins);
    st<S>(Xn, idx, nr, ni);
    red.add(0, sr, hr);
    red.add(1, hr, hr);
    if constexpr (C) {
      red.add(0, si, hi);
      red.add(1, hi, hi);
    }
    red.tick();
  } else if constexpr (E == Epi::kShift) {
    // H x stored; partial <x, (H + c) x>, element by element: with x near an eigenvector the sums of
    // <x, H x> and c <x, x> would cancel, and their roundings with them be all that is left
    st<S>(reinterpret_cast<S*>(fa.out), idx, hr, hi);
    red.add(0, sr, fma(es.c1, sr, hr));
    if constexpr (C) red.add(0, si, fma(es.c1, si, hi));
    red.tick();
  } else {  // kRefine: Hx stored; partials <x, Hx>, <x, x>, <Hx, Hx>
    st<S>(reinterpret_cast<S*>(fa.out), idx, hr, hi);
    red.add(0, sr, hr);
    red.add(1, sr, sr);
    red.add(2, hr, hr);
    if constexpr (C) {
      red.add(0, si, hi);
      red.add(1, si, si);
      red.add(2, hi, hi);
    }
    red.tick();
  }
}

// The refinement's element in folded units (x = xr 2^eoff, hv = hvu 2^e2): two fp64 conversions,
// one scale and three multiply-adds an element instead of about ten operations.
template <int NQ>
__device__ __forceinline__ void refine_folded(double hvu, double xr, double s_e2, int64_t idx, const FusedArgs& fa,
                                              Red<true, NQ>& red) {
  reinterpret_cast<double*>(fa.out)[idx] = hvu * s_e2;
  red.add(0, xr, hvu);
  red.add(1, xr, xr);
  red.add(2, hvu, hvu);
}

// The shifted product's element in folded units; cs = c 2^-k, hv = hvu 2^(eoff + k), x = xr 2^eoff.
template <int NQ>
__device__ __forceinline__ void shift_folded(double hvu, double xr, double cs, double s_e2, int64_t idx,
                                             const FusedArgs& fa, Red<true, NQ>& red) {
  reinterpret_cast<double*>(fa.out)[idx] = hvu * s_e2;
  red.add(0, xr, fma(cs, xr, hvu));
}

// A sum of folded products back in plain units: quantity 0 is x hv, 1 x x and 2 hv hv.
__device__ __forceinline__ double folded_sum(double x, int q, double s_eoff, double s_e2) {
  const double a = q == 2 ? s_e2 : s_eoff, b = q == 1 ? s_eoff : s_e2;
  return (x * a) * b;
}

template <Epi E> __host__ __device__ constexpr int n_red() {
  return E == Epi::kStore ? 0 : (E == Epi::kLanczos1 || E == Epi::kShift ? 1 : (E == Epi::kTpq ? 2 : 3));
}

}  // namespace hphi

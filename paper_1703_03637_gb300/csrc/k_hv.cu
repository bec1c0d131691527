// Matrix-free H v over the bit-string basis (section 3.3), fused with the Lanczos
// (section 3.4) and mTPQ (section 3.5) vector updates and their reductions.
//
// Gather form: each thread owns one output element (row r, vector c) and sums
//     w[r] = diag(s_r) v[r] + sum_patterns coef * phase * v[rank(s_r ^ mask)],
// so every write is coalesced and no atomics are needed.  The diagonal is an integer bit
// count per coefficient class (popcounts), then one multiply-add per class.  Off-diagonal
// patterns that share a coefficient up to a phase in {+1, +i, -1, -i} are summed first
// and multiplied once per class.  Fermion signs are popcount parities of the bits between
// the two hopping sites.  Reductions for the fused steps are per-thread partial sums
// (fp64, or error-free fp32 TwoSum chunks flushed to fp64) reduced per CTA in a fixed
// order and written to a partials array, so results are bit-reproducible run to run.
#include <algorithm>
#include <type_traits>

#include "basis.cuh"
#include "common.cuh"
#include "reduce.cuh"
#include "epilogue.cuh"

namespace hphi {

namespace {

// ------------------------------------------------------------------ spin kernel
// One thread per output element.  Patterns are visited in unrolled batches of kBatch:
// the active test, rank and address of every pattern in a batch are computed first and
// the batch's loads are issued together (predicated on the phase code), so each thread
// keeps kBatch gathers in flight instead of one.  Class boundaries are the same for every
// thread (patterns are sorted by class), so class flushes never diverge.
constexpr int kBatch = 8;

// largest hi with hi_off[hi] <= r, by one warp (32 probes a round)
__device__ __forceinline__ uint64_t warp_find_hi(const SectorTables& t, uint64_t r, uint64_t hmax) {
  const int lane = threadIdx.x & 31;
  uint64_t lo = 0, hi = hmax;
  while (lo < hi) {
    const uint64_t step = (hi - lo + 31) >> 5;
    const uint64_t m = lo + step * (uint64_t)(lane + 1);
    const bool in = m <= hi && __ldg(t.hi_off + (m <= hi ? m : hi)) <= r;
    const int c = __popc(__ballot_sync(0xffffffffu, in));  // hi_off does not decrease
    lo += step * (uint64_t)c;
    hi = min(hi, lo + step - 1);
  }
  return lo;
}

//
// The entries are merged by flip mask (SpinMerged): one gather serves both entries of a bond
// whose two patterns carry conjugate coefficients, which fall into two classes; a row adds the
// value to the sums of the one class its bits select.  St is the configuration's type, 32 bits
// up to 32 sites.
//
// QT (fp64): the gathers read the input quantised to 64-bit integers, one scale per vector
// column (q = round(x 2^(1078 - E_c)), |q| < 2^56), so every class sum of at most 127 terms
// is an exact integer sum (two integer instructions a term instead of the per-term
// alignment of the fixed-point accumulator), converted to fp64 once per class.
//
// 22-site ring with Dzyaloshinskii-Moriya exchange, S^z = 0 (705,432 rows c128), Lanczos step on
// GB300: 94 us instead of 173 us (one entry at a time, a binary search by one thread per 256 rows,
// conversions per class); bound by issue (47 %), the fp64 pipe (37 %) and latency together.
template <class S, Epi E, bool QT, class St>
__global__ void __launch_bounds__(kThreads, (Traits<S>::kF64 && !QT) ? 2 : 3) k_hv_spin(const SpinDev md, const S* __restrict__ v, S* __restrict__ w,
                                                         int nvec, int lg_nvec, FusedArgs fa,
                                                         const long long* __restrict__ Q, const int* __restrict__ Ec) {
  using R = typename Traits<S>::R;
  static_assert(!QT || Traits<S>::kF64, "quantised gathers are an fp64 path");
  using A = std::conditional_t<QT, IntAcc, typename SumAcc<R>::T>;
  using T = std::conditional_t<QT, long long, R>;  // gathered scalar
  constexpr bool C = Traits<S>::kCplx;
  constexpr bool F64 = Traits<S>::kF64;
  __shared__ SpinMerged s_ent[kMaxSpinEntries];
  __shared__ R s_cr[kMaxClasses], s_ci[kMaxClasses];
  __shared__ St s_lm[kMaxLin];
  __shared__ R s_lc[kMaxLin], s_pcoef[kMaxPairGroups];
  __shared__ PairEntry s_pair[kMaxPairs];
  __shared__ R s_inv[kMaxNvec];
  __shared__ uint64_t s_hi[2];
  __shared__ double s_red[(E == Epi::kStore) ? 1 : kThreads * (n_red<E>() > 0 ? n_red<E>() : 1)];

  if (fa.done != nullptr && *fa.done) return;
  const int tid = threadIdx.x;
  const int n_ent = md.n_merged;
  for (int k = tid; k < n_ent; k += kThreads) s_ent[k] = md.merged[k];
  for (int k = tid; k < md.n_classes; k += kThreads) {
    const double2 cc = md.cls_coef[k];
    s_cr[k] = (R)cc.x;
    s_ci[k] = (R)cc.y;
  }
  for (int k = tid; k < md.n_lin; k += kThreads) {
    s_lm[k] = (St)md.lin[k].mask;
    s_lc[k] = (R)md.lin[k].coef;
  }
  for (int k = tid; k < md.n_pairs; k += kThreads) s_pair[k] = md.pairs[k];
  for (int k = tid; k < md.n_pair_groups; k += kThreads) s_pcoef[k] = (R)md.pair_coef[k];
  if constexpr (E == Epi::kTpq) {
    for (int k = tid; k < nvec; k += kThreads) s_inv[k] = (R)fa.scal[k];
  }
  const EpiScalars<R> es = epi_scalars<R, E>(fa);
  const R c0 = opaque((R)md.c0);
  // one vector: the fixed point's scale goes into the class coefficients (an exact power of two
  // unless a product leaves the normal range), so a sum is one conversion and its multiply-adds
  bool pre = false;
  if constexpr (QT) {
    __syncthreads();
    bool ok = nvec == 1 && Ec[0] >= 1078 - 1022;
    const double sc = ok ? __longlong_as_double((long long)(Ec[0] - 1078 + 1023) << 52) : 1.0;
    for (int k = tid; k < md.n_classes; k += kThreads)
      ok = ok && (s_cr[k] == 0.0 || fabs(s_cr[k] * sc) >= 1e-290) && (s_ci[k] == 0.0 || fabs(s_ci[k] * sc) >= 1e-290);
    pre = __syncthreads_and(ok ? 1 : 0) != 0;
    if (pre)
      for (int k = tid; k < md.n_classes; k += kThreads) {
        s_cr[k] *= sc;
        s_ci[k] *= sc;
      }
  }
  __syncthreads();

  constexpr int kNQ = n_red<E>() > 0 ? n_red<E>() : 1;
  Red<F64, kNQ> red;
  red.zero();
  const int64_t total = md.dim * (int64_t)nvec;
  __shared__ int64_t s_item;
  const uint64_t hmax = md.sector ? ((1ull << md.t.H) - 1ull) : 0ull;
  const int tL = md.t.L;
  const St lomask = (St)(((uint64_t)1 << tL) - 1);

  // plain H v: chunks of kThreads elements are handed out in order from a counter, so
  // resident CTAs stay on neighbouring rows and share the rows they gather through L2.
  // Fused steps keep the static assignment (chunk = CTA + k * grid): each CTA's partial sums
  // then cover the same elements in the same order every run (bit-reproducible reductions).
  constexpr bool kDyn = (E == Epi::kStore);
  int64_t next = blockIdx.x;
  for (;;) {
    if constexpr (kDyn) {
      __syncthreads();
      if (tid == 0) s_item = (int64_t)atomicAdd(md.counter, 1ull);
      __syncthreads();
      next = s_item;
    }
    const int64_t base = next * kThreads;
    if constexpr (!kDyn) next += gridDim.x;
    if (base >= total) break;
    const int64_t idx = base + tid;
    const bool act = idx < total;
    int64_t r;
    int c;
    if (lg_nvec >= 0) {
      r = idx >> lg_nvec;
      c = (int)(idx & (nvec - 1));
    } else {
      r = idx / nvec;
      c = (int)(idx - r * nvec);
    }
    uint64_t s64 = (uint64_t)r;
    if (md.sector) {
      __syncthreads();
      if (tid < 64) {  // warp 0: the first row's high part, warp 1: the last row's
        const int64_t e = tid < 32 ? base : (base + kThreads < total ? base + kThreads : total) - 1;
        const uint64_t f = warp_find_hi(md.t, (uint64_t)(e / nvec), hmax);
        if ((tid & 31) == 0) s_hi[tid >> 5] = f;
      }
      __syncthreads();
      if (act) s64 = sector_state_in(md.t, (uint64_t)r, sector_find_hi(md.t, (uint64_t)r, s_hi[0], s_hi[1]));
    }
    if (!act) continue;
    const St s = (St)s64;
    auto pop = [](St x) -> int {
      if constexpr (sizeof(St) == 4) return __popc(x);
      else return __popcll(x);
    };

    // diagonal: integer bit counts per coefficient class
    R d = c0;
    for (int g = 0; g < md.n_lin; ++g) d += s_lc[g] * (R)pop(s & s_lm[g]);
    if (md.n_pairs) {
      int grp = s_pair[0].grp, cnt = 0;
      for (int p = 0; p < md.n_pairs; ++p) {
        const PairEntry pe = s_pair[p];
        if (pe.grp != grp) {
          d += s_pcoef[grp] * (R)cnt;
          cnt = 0;
          grp = pe.grp;
        }
        cnt += (int)((s >> pe.i) & (s >> pe.j) & (St)1);
      }
      d += s_pcoef[grp] * (R)cnt;
    }
    R sr, si;
    ld<S>(v, idx, sr, si);
    R hr = d * sr, hi = d * si;
    const int eoff = QT ? Ec[c] - 1078 : 0;

    A ar[2], ai[2];  // the sums of the two classes
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      ar[q].zero();
      ai[q].zero();
    }
    uint32_t cur = n_ent ? s_ent[0].cls : 0u;
    auto flush = [&]() {
      if constexpr (QT && C) {
        // the two patterns of a complex exchange: a + i b and, in its quadrant, b + i a =
        // i (a - i b); their sums meet as integers, half the conversions' multiply-adds
        const int p = (int)(cur & 0xffffu), o = (int)(cur >> 16);
        if (pre && o != 0xffff && md.max_run <= 63 && s_cr[o] == s_ci[p] && s_ci[o] == s_cr[p]) {
          const double a = s_cr[p], b = s_ci[p];
          hr = fma(a, __ll2double_rn(ar[0].s - ai[1].s), fma(b, __ll2double_rn(ar[1].s - ai[0].s), hr));
          hi = fma(a, __ll2double_rn(ai[0].s + ar[1].s), fma(b, __ll2double_rn(ar[0].s + ai[1].s), hi));
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            ar[q].zero();
            ai[q].zero();
          }
          return;
        }
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int cls = q ? (int)(cur >> 16) : (int)(cur & 0xffffu);
        if (q && cls == 0xffff) break;  // no second class
        const R cx = s_cr[cls], cy = s_ci[cls];
        R vr, vi;
        if constexpr (QT) {
          vr = pre ? __ll2double_rn(ar[q].value()) : fix_to_double(ar[q].value(), eoff);
          vi = !C ? 0.0 : pre ? __ll2double_rn(ai[q].value()) : fix_to_double(ai[q].value(), eoff);
        } else {
          vr = (R)ar[q].value();
          vi = (R)ai[q].value();
        }
        if constexpr (C) {
          hr += cx * vr;
          hi += cx * vi;
          if (cy != R(0)) {
            hr -= cy * vi;
            hi += cy * vr;
          }
        } else {
          hr += cx * vr;
        }
        ar[q].zero();
        ai[q].zero();
      }
    };
    for (int e0 = 0; e0 < n_ent; e0 += kBatch) {
      T xr[kBatch], xi[kBatch];
      int code[kBatch];  // phase, plus 8 for the second class
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const int k = e0 + j;
        code[j] = 0;
        xr[j] = 0;
        xi[j] = 0;
        if (k < n_ent) {
          const SpinMerged en = s_ent[k];
          const int sel = (int)((s >> en.i) & (St)1) | ((int)((s >> en.j) & (St)1) << 1);
          code[j] = (int)((en.phases >> (4 * sel)) & 15u);
          if (code[j]) {
            const St s2 = s ^ (St)en.mask;
            uint64_t r2 = (uint64_t)s2;
            if (md.sector) r2 = __ldg(md.t.hi_off + (s2 >> tL)) + (uint64_t)__ldg(md.t.lo_rank + (s2 & lomask));
            if constexpr (QT) {
              const int64_t o = (int64_t)r2 * nvec + c;
              if constexpr (C) {
                const longlong2 t = __ldg(reinterpret_cast<const longlong2*>(Q) + o);
                xr[j] = t.x;
                xi[j] = t.y;
              } else {
                xr[j] = __ldg(Q + o);
              }
            } else {
              ld<S>(v, (int64_t)r2 * nvec + c, xr[j], xi[j]);
            }
          }
        }
      }
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const int k = e0 + j;
        if (k < n_ent) {
          const uint32_t cls = s_ent[k].cls;
          if (cls != cur) {  // the entries are shared: the same for all threads
            flush();
            cur = cls;
          }
          if (code[j] & 8) {
            if constexpr (C) acc_phase<A, T>(code[j] & 7, xr[j], xi[j], ar[1], ai[1]);
            else ar[1].add(xr[j], code[j] != 9);
          } else if (code[j]) {
            if constexpr (C) acc_phase<A, T>(code[j], xr[j], xi[j], ar[0], ai[0]);
            else ar[0].add(xr[j], code[j] != 1);
          }
        }
      }
    }
    if (n_ent) flush();
    epilogue<S, E, kNQ>(idx, sr, si, hr, hi, w, fa, es, E == Epi::kTpq ? s_inv[c] : R(0), red);
  }
  if constexpr (E != Epi::kStore) block_finish<F64, kThreads, kNQ>(red, n_red<E>(), nvec, fa.partials, s_red);
}

// ------------------------------------------------------------------ Hubbard kernel
// Work item = (down-spin row d, chunk of kThreads consecutive (up, vector) elements).
// Down-spin hops depend only on d, so warp 0 builds the row's compacted neighbour list
// (source row, sign, direction, class) in shared memory once per item and every thread
// walks it uniformly in batches of kBatch coalesced loads.  Up-spin hops depend on each
// thread's up configuration and are visited in predicated batches of kBatch.
template <class S, Epi E>
__global__ void __launch_bounds__(kThreads) k_hv_hub(const HubDev md, const S* __restrict__ v, S* __restrict__ w,
                                                     int nvec, int lg_nvec, FusedArgs fa) {
  using R = typename Traits<S>::R;
  using A = typename SumAcc<R>::T;
  constexpr bool C = Traits<S>::kCplx;
  constexpr bool F64 = Traits<S>::kF64;
  __shared__ HopEntry s_hop[kMaxHops];
  __shared__ double2 s_cls[kMaxClasses];
  __shared__ LinGroup s_ulin[kMaxLin];
  __shared__ LinGroup s_mlin[kMaxLin];
  __shared__ PairEntry s_pair[kMaxPairs];
  __shared__ double s_pcoef[kMaxPairGroups];
  __shared__ R s_inv[kMaxNvec];
  __shared__ int64_t s_dl_src[kMaxHops];   // source element offset of neighbour row d'
  __shared__ uint32_t s_dl_meta[kMaxHops];  // bit 0 negative sign, bit 1 direction b, class << 2
  __shared__ int s_dl_n;
  __shared__ double s_red[(E == Epi::kStore) ? 1 : kThreads * kMaxRedQ];

  if (fa.done != nullptr && *fa.done) return;
  const int tid = threadIdx.x;
  const int n_up = md.n_up_hops, n_dn = md.n_dn_hops;
  const int n_hops = n_up + n_dn;
  for (int k = tid; k < n_hops; k += kThreads) s_hop[k] = md.hops[k];
  for (int k = tid; k < md.n_classes; k += kThreads) s_cls[k] = md.cls_coef[k];
  for (int k = tid; k < md.n_ulin; k += kThreads) s_ulin[k] = md.ulin[k];
  for (int k = tid; k < md.n_mulin; k += kThreads) s_mlin[k] = md.mulin[k];
  for (int k = tid; k < md.n_pairs; k += kThreads) s_pair[k] = md.pairs[k];
  for (int k = tid; k < md.n_pair_groups; k += kThreads) s_pcoef[k] = md.pair_coef[k];
  if constexpr (E == Epi::kTpq) {
    for (int k = tid; k < nvec; k += kThreads) s_inv[k] = (R)fa.scal[k];
  }
  const EpiScalars<R> es = epi_scalars<R, E>(fa);
  __syncthreads();

  constexpr int kNQ = n_red<E>() > 0 ? n_red<E>() : 1;
  Red<F64, kNQ> red;
  red.zero();
  const int64_t row_elems = md.dim_up * (int64_t)nvec;
  const int64_t nchunk = (row_elems + kThreads - 1) / kThreads;
  const int64_t n_items = nchunk * md.dim_dn;

  __shared__ int64_t s_item;
  constexpr bool kDyn = (E == Epi::kStore);  // see k_hv_spin: fused steps stay static
  int64_t next = blockIdx.x;
  for (;;) {
    if constexpr (kDyn) {
      __syncthreads();
      if (tid == 0) s_item = (int64_t)atomicAdd(md.counter, 1ull);
      __syncthreads();
      next = s_item;
    }
    const int64_t item = next;
    if constexpr (!kDyn) next += gridDim.x;
    if (item >= n_items) break;
    const int64_t d = item / nchunk;
    const int64_t e = (item - d * nchunk) * kThreads + tid;
    const uint32_t dn = md.sector ? __ldg(md.list_dn + d) : (uint32_t)d;
    // neighbour list of row d (ordered, so classes stay grouped)
    __syncthreads();
    if (tid < 32) {
      int cnt = 0;
      for (int k0 = 0; k0 < n_dn; k0 += 32) {
        const int k = k0 + tid;
        bool on = false;
        int64_t src = 0;
        uint32_t meta = 0;
        if (k < n_dn) {
          const HopEntry h = s_hop[n_up + k];
          const uint32_t bi = (dn >> h.i) & 1u, bj = (dn >> h.j) & 1u;
          if (bi != bj) {
            on = true;
            const uint32_t b2 = dn ^ h.mask;
            const int64_t d2 = md.sector ? (int64_t)__ldg(md.rank + b2) : (int64_t)b2;
            src = d2 * md.dim_up * nvec;
            meta = (uint32_t)(__popc(dn & h.between) & 1) | ((bi ? 0u : 1u) << 1) | ((uint32_t)h.cls << 2);
          }
        }
        const unsigned bal = __ballot_sync(0xffffffffu, on);
        if (on) {
          const int pos = cnt + __popc(bal & ((1u << tid) - 1u));
          s_dl_src[pos] = src;
          s_dl_meta[pos] = meta;
        }
        cnt += __popc(bal);
      }
      if (tid == 0) s_dl_n = cnt;
    }
    __syncthreads();
    if (e >= row_elems) continue;
    int64_t u;
    int c;
    if (lg_nvec >= 0) {
      u = e >> lg_nvec;
      c = (int)(e & (nvec - 1));
    } else {
      u = e / nvec;
      c = (int)(e - u * nvec);
    }
    const uint32_t up = md.sector ? __ldg(md.list_up + u) : (uint32_t)u;
    const int64_t row_base = d * md.dim_up;
    const int64_t idx = (row_base + u) * nvec + c;

    // diagonal
    R dg = (R)md.c0;
    for (int g = 0; g < md.n_ulin; ++g) dg += (R)s_ulin[g].coef * (R)__popc(up & dn & (uint32_t)s_ulin[g].mask);
    for (int g = 0; g < md.n_mulin; ++g) {
      const uint32_t m = (uint32_t)s_mlin[g].mask;
      dg += (R)s_mlin[g].coef * (R)(__popc(up & m) + __popc(dn & m));
    }
    if (md.n_pairs) {
      int grp = s_pair[0].grp, cnt = 0;
      for (int p = 0; p < md.n_pairs; ++p) {
        const PairEntry pe = s_pair[p];
        if (pe.grp != grp) {
          dg += (R)s_pcoef[grp] * (R)cnt;
          cnt = 0;
          grp = pe.grp;
        }
        const int ni = (int)((up >> pe.i) & 1u) + (int)((dn >> pe.i) & 1u);
        const int nj = (int)((up >> pe.j) & 1u) + (int)((dn >> pe.j) & 1u);
        cnt += ni * nj;
      }
      dg += (R)s_pcoef[grp] * (R)cnt;
    }
    R sr, si;
    ld<S>(v, idx, sr, si);
    R hr = dg * sr, hi = dg * si;

    // coef * a + conj(coef) * b for one class
    A ar, ai, br, bi_;
    ar.zero(); ai.zero(); br.zero(); bi_.zero();
    auto flush = [&](int cls) {
      const double2 cc = s_cls[cls];
      if constexpr (C) {
        const R a_r = (R)ar.value(), a_i = (R)ai.value(), b_r = (R)br.value(), b_i = (R)bi_.value();
        hr += (R)cc.x * (a_r + b_r) - (R)cc.y * (a_i - b_i);
        hi += (R)cc.x * (a_i + b_i) + (R)cc.y * (a_r - b_r);
        br.zero();
        bi_.zero();
      } else {
        hr += (R)cc.x * (R)ar.value();
      }
      ar.zero();
      ai.zero();
    };

    // up hops: predicated batches
    int cur = n_up ? s_hop[0].cls : 0;
    for (int k0 = 0; k0 < n_up; k0 += kBatch) {
      R xr[kBatch], xi[kBatch];
      uint32_t fl[kBatch];  // bit 0 active, bit 1 negative, bit 2 direction b
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const int k = k0 + j;
        fl[j] = 0;
        xr[j] = 0;
        xi[j] = 0;
        if (k < n_up) {
          const HopEntry h = s_hop[k];
          const uint32_t bi = (up >> h.i) & 1u, bj = (up >> h.j) & 1u;
          if (bi != bj) {
            const uint32_t b2 = up ^ h.mask;
            const int64_t u2 = md.sector ? (int64_t)__ldg(md.rank + b2) : (int64_t)b2;
            ld<S>(v, (row_base + u2) * nvec + c, xr[j], xi[j]);
            fl[j] = 1u | ((uint32_t)(__popc(up & h.between) & 1) << 1) | ((bi ? 0u : 1u) << 2);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const int k = k0 + j;
        if (k < n_up) {
          const int cls = s_hop[k].cls;
          if (cls != cur) {
            flush(cur);
            cur = cls;
          }
          if (fl[j] & 1u) {
            const bool neg = (fl[j] & 2u) != 0;
            if constexpr (C) {
              if (!(fl[j] & 4u)) { ar.add(xr[j], neg); ai.add(xi[j], neg); }
              else { br.add(xr[j], neg); bi_.add(xi[j], neg); }
            } else {
              ar.add(xr[j], neg);
            }
          }
        }
      }
    }
    if (n_up) flush(cur);

    // down hops: row-uniform compacted list, batches of coalesced loads
    const int ndl = s_dl_n;
    const int64_t off = u * nvec + c;
    cur = ndl ? (int)(s_dl_meta[0] >> 2) : 0;
    for (int q0 = 0; q0 < ndl; q0 += kBatch) {
      R xr[kBatch], xi[kBatch];
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        xr[j] = 0;
        xi[j] = 0;
        if (q0 + j < ndl) ld<S>(v, s_dl_src[q0 + j] + off, xr[j], xi[j]);
      }
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const int q = q0 + j;
        if (q < ndl) {
          const uint32_t meta = s_dl_meta[q];
          const int cls = (int)(meta >> 2);
          if (cls != cur) {
            flush(cur);
            cur = cls;
          }
          const bool neg = (meta & 1u) != 0;
          if constexpr (C) {
            if (!(meta & 2u)) { ar.add(xr[j], neg); ai.add(xi[j], neg); }
            else { br.add(xr[j], neg); bi_.add(xi[j], neg); }
          } else {
            ar.add(xr[j], neg);
          }
        }
      }
    }
    if (ndl) flush(cur);
    epilogue<S, E, kNQ>(idx, sr, si, hr, hi, w, fa, es, E == Epi::kTpq ? s_inv[c] : R(0), red);
  }
  if constexpr (E != Epi::kStore) block_finish<F64, kThreads, kNQ>(red, n_red<E>(), nvec, fa.partials, s_red);
}

template <class S, Epi E>
int occupancy_t(bool hub) {
  static int cache[2] = {0, 0};
  int& b = cache[hub ? 1 : 0];
  if (b == 0) {
    int n = 0;
    cudaError_t e = hub ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_hv_hub<S, E>, kThreads, 0)
                        : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_hv_spin<S, E, Traits<S>::kF64, uint32_t>, kThreads, 0);
    if (e != cudaSuccess || n < 1) {
      cudaGetLastError();
      n = 2;
    }
    b = n;
  }
  return b;
}

template <Epi E>
int occupancy_e(bool hub, int prec, bool cplx) {
  if (prec == HPHI_FP64) return cplx ? occupancy_t<double2, E>(hub) : occupancy_t<double, E>(hub);
  return cplx ? occupancy_t<float2, E>(hub) : occupancy_t<float, E>(hub);
}

template <class S, Epi E>
Status launch_t(bool hub, const void* md, const void* v, void* w, int nvec, const FusedArgs& fa, int grid,
                void* scratch, cudaStream_t st) {
  int lg = -1;
  if ((nvec & (nvec - 1)) == 0) {
    lg = 0;
    while ((1 << lg) < nvec) ++lg;
  }
  unsigned long long* counter = hub ? reinterpret_cast<const HubDev*>(md)->counter
                                   : reinterpret_cast<const SpinDev*>(md)->counter;
  HPHI_CUDA_TRY(cudaMemsetAsync(counter, 0, sizeof(unsigned long long), st));
  if (hub) {
    k_hv_hub<S, E><<<grid, kThreads, 0, st>>>(*reinterpret_cast<const HubDev*>(md), reinterpret_cast<const S*>(v),
                                             reinterpret_cast<S*>(w), nvec, lg, fa);
  } else {
    const SpinDev& sd = *reinterpret_cast<const SpinDev*>(md);
    const S* vs = reinterpret_cast<const S*>(v);
    S* ws = reinterpret_cast<S*>(w);
    const bool narrow = sd.n_sites <= 32;
    long long* q = nullptr;
    int* e = nullptr;
    if constexpr (Traits<S>::kF64) {
      if (spin_quantised(sd, HPHI_FP64, nvec) && scratch != nullptr) {
        constexpr int ncomp = Traits<S>::kCplx ? 2 : 1;
        q = reinterpret_cast<long long*>(scratch);
        e = reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(scratch) + (size_t)sd.dim * nvec * sizeof(S));
        Status qs = launch_quant_cols(reinterpret_cast<const double*>(v), sd.dim, nvec, ncomp, q, e, st);
        if (qs.code) return qs;
        if (narrow) k_hv_spin<S, E, true, uint32_t><<<grid, kThreads, 0, st>>>(sd, vs, ws, nvec, lg, fa, q, e);
        else k_hv_spin<S, E, true, uint64_t><<<grid, kThreads, 0, st>>>(sd, vs, ws, nvec, lg, fa, q, e);
      }
    }
    if (q == nullptr) {
      if (narrow) k_hv_spin<S, E, false, uint32_t><<<grid, kThreads, 0, st>>>(sd, vs, ws, nvec, lg, fa, q, e);
      else k_hv_spin<S, E, false, uint64_t><<<grid, kThreads, 0, st>>>(sd, vs, ws, nvec, lg, fa, q, e);
    }
  }
  HPHI_CUDA_TRY(cudaGetLastError());
  return {};
}

template <Epi E>
Status launch_e(bool hub, const void* md, int prec, bool cplx, const void* v, void* w, int nvec, const FusedArgs& fa,
                int grid, void* scratch, cudaStream_t st) {
  if (prec == HPHI_FP64) {
    return cplx ? launch_t<double2, E>(hub, md, v, w, nvec, fa, grid, scratch, st)
                : launch_t<double, E>(hub, md, v, w, nvec, fa, grid, scratch, st);
  }
  return cplx ? launch_t<float2, E>(hub, md, v, w, nvec, fa, grid, scratch, st)
              : launch_t<float, E>(hub, md, v, w, nvec, fa, grid, scratch, st);
}

}  // namespace

int hv_grid(int nvec) {
  (void)nvec;
  return num_sms() * (2048 / kThreads);
}

int hv_resident_grid(bool hubbard, int prec, bool cplx, Epi epi) {
  int b = 2;
  switch (epi) {
    case Epi::kStore: b = occupancy_e<Epi::kStore>(hubbard, prec, cplx); break;
    case Epi::kLanczos1: b = occupancy_e<Epi::kLanczos1>(hubbard, prec, cplx); break;
    case Epi::kTpq: b = occupancy_e<Epi::kTpq>(hubbard, prec, cplx); break;
    case Epi::kRefine: b = occupancy_e<Epi::kRefine>(hubbard, HPHI_FP64, cplx); break;
    case Epi::kShift: b = cplx ? occupancy_t<double2, Epi::kShift>(hubbard) : occupancy_t<double, Epi::kShift>(hubbard); break;
  }
  return num_sms() * b;
}

bool spin_quantised(const SpinDev& md, int prec, int nvec) {
  return prec == HPHI_FP64 && md.max_run <= 127 && nvec >= 1 && nvec <= kMaxNvec && (nvec & (nvec - 1)) == 0;
}

size_t spin_scratch_bytes(const SpinDev& md, int prec, bool cplx, int nvec) {
  if (!spin_quantised(md, prec, nvec)) return 0;
  return (size_t)md.dim * nvec * 8 * (cplx ? 2 : 1) + sizeof(int) * (size_t)nvec;
}

Status launch_hv(bool hubbard, const void* md, int prec, bool cplx, const void* v, void* w, int nvec, Epi epi,
                 const FusedArgs& fa, int grid, void* scratch, cudaStream_t st) {
  switch (epi) {
    case Epi::kStore: return launch_e<Epi::kStore>(hubbard, md, prec, cplx, v, w, nvec, fa, grid, scratch, st);
    case Epi::kLanczos1:
      return launch_e<Epi::kLanczos1>(hubbard, md, prec, cplx, v, w, nvec, fa, grid, scratch, st);
    case Epi::kTpq: return launch_e<Epi::kTpq>(hubbard, md, prec, cplx, v, w, nvec, fa, grid, scratch, st);
    case Epi::kRefine:
      if (prec != HPHI_FP64) return {HPHI_ERR_INVALID_ARG, "refinement runs in fp64"};
      return launch_e<Epi::kRefine>(hubbard, md, prec, cplx, v, w, nvec, fa, grid, scratch, st);
    case Epi::kShift:
      if (prec != HPHI_FP64) return {HPHI_ERR_INVALID_ARG, "refinement runs in fp64"};
      return cplx ? launch_t<double2, Epi::kShift>(hubbard, md, v, w, nvec, fa, grid, scratch, st)
                  : launch_t<double, Epi::kShift>(hubbard, md, v, w, nvec, fa, grid, scratch, st);
  }
  return {HPHI_ERR_INVALID_ARG, "unknown epilogue"};
}

// ------------------------------------------------------------------ one-cluster Lanczos
// The whole recurrence of section 3.4 in one thread-block cluster when both Lanczos vectors fit
// in the cluster's shared memory (real spin models up to kClMaxDim rows): no launch per step,
// no trip through HBM.  CTA c of the cluster owns rows [c R, (c + 1) R) of C and P in its shared
// memory; a thread owns rows of its CTA's slice.  H C gathers C[r'] from whichever CTA owns r'
// through distributed shared memory.  GB300 issues fp64 at 1/64 of its fp32 rate, so one SM
// alone would be bound by the fp64 work of the diagonal and exchange sums: the cluster spreads
// it over kClCtas SMs.  Per step: P = c1 H C - c2 P with the partial (C, H C), cluster barrier,
// alpha, P -= gamma C with |P|^2, cluster barrier, beta, swap C and P.
//
// What does not change from step to step is worked out once: each row's diagonal element and the
// cluster address of every element it gathers, with the element's signed coefficient in the
// address's low bits (kClCoef codes).  Models with more coefficients, or rows with more elements
// than the shared memory left (cap), decode their terms in every step instead.
//
// A sum over the cluster: every warp writes its sum into every CTA's slot for it before the
// barrier; behind it one warp of each CTA adds the slots in one fixed order (the same bits in
// every CTA), works out the step's scalars and hands them to its CTA.  One warp, because every
// fp64 instruction of a warp holds its scheduler's fp64 unit for 64 cycles: eight warps repeating
// the scalar work cost more than the hand-over.  The two slot arrays alternate, so each barrier
// also ends the reads of the other.
// Scalars follow k_lz_fin's conventions (C unnormalised, sigma = 1 / |C|), so k_tridiag reads the
// same arrays.  Bound by latency (two barriers, two sums and about 14 dependent fp64 operations a
// step); measured on GB300: 6.1 us a step on the 12-site ring's 4,096 rows instead of 11.5 us.
namespace {
constexpr int kClThreads = 256;
constexpr int kClWarps = kClThreads / 32;
constexpr int kClCoef = 8;  // distinct signed coefficients a gather address can carry

// cluster barrier (all threads of all CTAs; shared-memory writes before it are visible after)
__device__ __forceinline__ void cl_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// cluster shared-memory address of this CTA's variable p as it lies in CTA `rank`
__device__ __forceinline__ uint32_t cl_map(const void* p, unsigned rank) {
  uint32_t out;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return out;
}
__device__ __forceinline__ double cl_load(uint32_t a) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a));  // ordered against cl_sync
  return v;
}
__device__ __forceinline__ void cl_store(uint32_t a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

// first half of a cluster sum: this warp's sum of x into its slot of every CTA
__device__ __forceinline__ void cl_put(double x, double* slots, unsigned rank, int ncta) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
  x = __shfl_sync(0xffffffffu, x, 0);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane < ncta) cl_store(cl_map(slots + rank * kClWarps + wid, (unsigned)lane), x);
}
// second half, behind the barrier
__device__ __forceinline__ double cl_take(const double* slots, int ncta) {
  const int lane = threadIdx.x & 31;
  double v = 0.0;
  for (int k = lane; k < ncta * kClWarps; k += 32) v += slots[k];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  // lanes may hold differently rounded sums; lane 0's is the same in every CTA, and the loop's
  // exit test must see one value everywhere
  return __shfl_sync(0xffffffffu, v, 0);
}

__device__ __forceinline__ unsigned cl_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// list: cap slots per row, slot k of local row i at list[k R + i]
__global__ void __launch_bounds__(kClThreads, 1) k_lz_cl(const SpinDev md, LzDev lz, int steps, double brk,
                                                         const double* __restrict__ C0, int R, int ncta, int cap) {
  extern __shared__ __align__(16) double sm_v[];  // [2][R] this CTA's slices, [R] diagonal, lists
  __shared__ double s_slot[2][16 * kClWarps];
  __shared__ double s_coef[kClCoef];
  __shared__ double s_sc[3];  // gamma; c1 = sigma and c2 of the next step
  __shared__ int s_over, s_ncoef, s_done;
  __shared__ SpinEntry s_ent[kMaxSpinEntries];
  __shared__ double s_cls[kMaxClasses];
  __shared__ LinGroup s_lin[kMaxLin];
  __shared__ PairEntry s_pair[kMaxPairs];
  __shared__ double s_pcoef[kMaxPairGroups];
  const int tid = threadIdx.x;
  const unsigned rank = cl_rank();
  const int64_t n = md.dim;
  const int64_t r0 = (int64_t)rank * R;
  const int64_t left = n - r0;
  const int nloc = left <= 0 ? 0 : (left < (int64_t)R ? (int)left : R);
  double* A = sm_v;
  double* B = sm_v + R;
  double* D = sm_v + 2 * R;
  uint32_t* list = reinterpret_cast<uint32_t*>(sm_v + 3 * R);
  uint8_t* s_cnt = reinterpret_cast<uint8_t*>(list + (size_t)cap * R);
  for (int k = tid; k < md.n_entries; k += kClThreads) s_ent[k] = md.entries[k];
  for (int k = tid; k < md.n_classes; k += kClThreads) s_cls[k] = md.cls_coef[k].x;
  for (int k = tid; k < md.n_lin; k += kClThreads) s_lin[k] = md.lin[k];
  for (int k = tid; k < md.n_pairs; k += kClThreads) s_pair[k] = md.pairs[k];
  for (int k = tid; k < md.n_pair_groups; k += kClThreads) s_pcoef[k] = md.pair_coef[k];
  if (tid == 0) {
    // +c of class k at code 2k, -c at 2k + 1
    s_ncoef = 2 * md.n_classes;
    s_over = s_ncoef > kClCoef ? 1 : 0;
  }
  __syncthreads();
  if (tid < kClCoef) s_coef[tid] = tid < s_ncoef ? ((tid & 1) ? -s_cls[tid >> 1] : s_cls[tid >> 1]) : 0.0;
  auto state = [&](int i) -> uint64_t {
    return md.sector ? sector_state(md.t, (uint64_t)(r0 + i)) : (uint64_t)(r0 + i);
  };
  const uint32_t a_off = (uint32_t)__cvta_generic_to_shared(A);
  for (int i = tid; i < nloc; i += kClThreads) {
    A[i] = C0[r0 + i];
    B[i] = 0.0;
    const uint64_t s = state(i);
    // diagonal: integer bit counts per coefficient group, one multiply-add per group
    double d = md.c0;
    for (int g = 0; g < md.n_lin; ++g) d += s_lin[g].coef * (double)__popcll(s & s_lin[g].mask);
    if (md.n_pairs) {
      int grp = s_pair[0].grp, cnt = 0;
      for (int q = 0; q < md.n_pairs; ++q) {
        const PairEntry pe = s_pair[q];
        if (pe.grp != grp) {
          d += s_pcoef[grp] * (double)cnt;
          cnt = 0;
          grp = pe.grp;
        }
        cnt += (int)((s >> pe.i) & (s >> pe.j) & 1ull);
      }
      d += s_pcoef[grp] * (double)cnt;
    }
    D[i] = d;
    int c = 0;
    if (s_ncoef <= kClCoef) {
      for (int e = 0; e < md.n_entries; ++e) {
        const SpinEntry en = s_ent[e];
        const int sel = (int)((s >> en.i) & 1ull) | ((int)((s >> en.j) & 1ull) << 1);
        const int code = (en.phases >> (3 * sel)) & 7;
        if (!code) continue;
        if (c < cap) {
          const uint64_t s2 = s ^ en.mask;
          const int64_t r2 = md.sector ? (int64_t)sector_rank(md.t, s2) : (int64_t)s2;
          const unsigned owner = (unsigned)(r2 / R);
          list[(size_t)c * R + i] = cl_map(A + (r2 - (int64_t)owner * R), owner) | (uint32_t)(2 * en.cls + (code == 1 ? 0 : 1));
        }
        ++c;
      }
      if (c > min(cap, 255)) s_over = 1;  // (any thread: the value is the same)
    }
    s_cnt[i] = (uint8_t)min(c, 255);
  }
  // k_lz_init / its finaliser have set sigma_0, c1, c2 and the flags
  double sg = lz.sig[0];
  double c1 = lz.s[0], c2 = lz.s[1];
  int done = *lz.done;
  bool cur_a = true;  // C is A (else B)
  int k = 0;
  cl_sync();  // every CTA has staged its slice of C_0 and its flag
  bool over = false;
  for (int c = 0; c < ncta; ++c) {
    int f;
    asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(f) : "r"(cl_map(&s_over, (unsigned)c)) : "memory");
    over = over || f != 0;
  }
  for (; k < steps && !done; ++k) {
    double* C = cur_a ? A : B;
    double* P = cur_a ? B : A;
    const uint32_t shift = cur_a ? 0u : (uint32_t)(R * sizeof(double));
    double xh = 0.0;
    for (int i = tid; i < nloc; i += kClThreads) {
      const double x = C[i];
      double hv = D[i] * x;
      if (!over) {
        const int cnt = s_cnt[i];
        for (int e0 = 0; e0 < cnt; e0 += 8) {
          double y[8];
          uint32_t ad[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) ad[j] = e0 + j < cnt ? list[(size_t)(e0 + j) * R + i] : a_off;
#pragma unroll
          for (int j = 0; j < 8; ++j) y[j] = e0 + j < cnt ? cl_load((ad[j] & ~7u) + shift) : 0.0;
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (e0 + j < cnt) hv = fma(s_coef[ad[j] & 7u], y[j], hv);
        }
      } else {
        // signed sums per coefficient class (entries are sorted by class), gathers in batches of
        // eight so their distributed-shared-memory loads overlap
        const uint64_t s = state(i);
        double acc = 0.0;
        int cur = md.n_entries ? s_ent[0].cls : 0;
        for (int e0 = 0; e0 < md.n_entries; e0 += 8) {
          double y[8];
          int sg8[8], cl8[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            y[j] = 0.0;
            sg8[j] = 0;
            cl8[j] = cur;
            const int e = e0 + j;
            if (e < md.n_entries) {
              const SpinEntry en = s_ent[e];
              cl8[j] = en.cls;
              const int sel = (int)((s >> en.i) & 1ull) | ((int)((s >> en.j) & 1ull) << 1);
              const int code = (en.phases >> (3 * sel)) & 7;
              if (code) {
                const uint64_t s2 = s ^ en.mask;
                const int64_t r2 = md.sector ? (int64_t)sector_rank(md.t, s2) : (int64_t)s2;
                const unsigned owner = (unsigned)(r2 / R);
                y[j] = cl_load(cl_map(C + (r2 - (int64_t)owner * R), owner));
                sg8[j] = code == 1 ? 1 : -1;  // real models: codes +1 / -1 only
              }
            }
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if (cl8[j] != cur) {
              hv = fma(s_cls[cur], acc, hv);
              acc = 0.0;
              cur = cl8[j];
            }
            if (sg8[j] > 0) acc += y[j];
            else if (sg8[j] < 0) acc -= y[j];
          }
        }
        if (md.n_entries) hv = fma(s_cls[cur], acc, hv);
      }
      xh = fma(x, hv, xh);
      P[i] = c1 * hv - c2 * P[i];
    }
    cl_put(xh, s_slot[0], rank, ncta);
    cl_sync();  // P written everywhere (so C is no longer read), sums of alpha in their slots
    double a = 0.0;
    if (tid < 32) {
      const double xs = cl_take(s_slot[0], ncta);
      a = xs * sg * sg;  // alpha_k = (H v_k, v_k)
      if (tid == 0) s_sc[0] = a * sg;
    }
    __syncthreads();
    const double gm = s_sc[0];
    double pp = 0.0;
    for (int i = tid; i < nloc; i += kClThreads) {
      const double pv = fma(-gm, C[i], P[i]);
      P[i] = pv;
      pp = fma(pv, pv, pp);
    }
    cl_put(pp, s_slot[1], rank, ncta);
    cl_sync();  // the new vector complete everywhere, sums of beta in their slots
    if (tid < 32) {
      const double ps = cl_take(s_slot[1], ncta);
      const double b = sqrt(ps), sn = 1.0 / b;
      if (tid == 0) {
        const bool stop = !(b > brk * fmax(1.0, fabs(a)));
        s_done = stop ? 1 : 0;
        s_sc[1] = sn;
        s_sc[2] = b * sg;
        if (rank == 0) {
          lz.alpha[k] = a;
          lz.beta[k] = b;
          if (!stop) lz.sig[k + 1] = sn;
        }
      }
    }
    __syncthreads();
    if (s_done) {
      done = 1;
    } else {
      c1 = s_sc[1];
      c2 = s_sc[2];
      sg = c1;
      cur_a = !cur_a;
    }
  }
  if (rank == 0 && tid == 0) {
    *lz.steps_done = k;
    *lz.done = 1;
  }
  cl_sync();  // no CTA leaves while another may still read its shared memory
}

constexpr int kClCtas = 16;       // CTAs per cluster (non-portable size; 8 if 16 cannot launch)
constexpr int64_t kClMaxDim = 32768;
constexpr int kClSmem = 190000;   // dynamic shared memory of a CTA (besides ~26 KB static)

}  // namespace

// dynamic shared memory of one cluster CTA, or 0 when the model does not take the path
size_t lz_cta_smem(const SpinDev& md) {
  if (md.dim > kClMaxDim) return 0;
  const int64_t R = (md.dim + kClCtas - 1) / kClCtas;
  return 3 * sizeof(double) * (size_t)R;
}

Status launch_lz_cta(const SpinDev& md, const LzDev& lz, int steps, double brk, const double* C0, cudaStream_t st) {
  for (int cs : {kClCtas, 8}) {
    const int R = (int)((md.dim + cs - 1) / cs);
    // two slices and the diagonal, a count and `cap` list slots per row
    const size_t fixed = (3 * sizeof(double) + 1) * (size_t)R;
    const int cap = (int)std::max<int64_t>(0, std::min<int64_t>(md.n_entries, ((int64_t)kClSmem - (int64_t)fixed) / (4 * (int64_t)R)));
    const size_t smem = fixed + 4 * (size_t)cap * (size_t)R;
    HPHI_CUDA_TRY(cudaFuncSetAttribute(k_lz_cl, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (cs > 8) HPHI_CUDA_TRY(cudaFuncSetAttribute(k_lz_cl, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs, 1, 1);
    cfg.blockDim = dim3(kClThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nclusters = 0;
    if (cudaOccupancyMaxActiveClusters(&nclusters, k_lz_cl, &cfg) != cudaSuccess || nclusters < 1) {
      cudaGetLastError();
      continue;
    }
    HPHI_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_lz_cl, md, lz, steps, brk, C0, R, cs, cap));
    return {};
  }
  return {HPHI_ERR_CUDA, "one-cluster Lanczos: no cluster of 16 or 8 CTAs can be scheduled"};
}

}  // namespace hphi

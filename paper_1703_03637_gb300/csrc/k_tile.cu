// H v over rows of many vectors in the full 2^N basis, N <= 32, by tiles of rows in shared
// memory (the batched mTPQ starts of section 3.5; section 4.3's idea of making every term act on
// local data, with a tile as the local memory).
//
// A term flips one or two sites, so a set of t sites closes a tile: the 2^t rows that agree on
// all other sites hold every partner of the terms whose flipped sites lie in the set.  The
// terms are covered by a few site sets (batch_tile_plan; three sets of ten sites hold the 48
// terms of the 24-site Kitaev cluster in a field).  One pass per set: a CTA stages a tile of
// 2^t rows x 16 U bytes (64 KB), sums the set's terms out of it and adds the sums to the output
// block, which is also the accumulator; the last pass adds the diagonal and runs the epilogue.
// Against gathers from L2 (one 512-byte row per term and row), a step's memory traffic falls
// from (terms) to (3 passes - 1) blocks.
//
// A 64 KB tile is 4,096 units of 16 bytes (two c64, four fp32, one c128 or two fp64 numbers).
// Thread tid owns unit tid mod U of 16 rows: the low t - 4 local row bits come from tid, the
// four high ones number its rows, which share their columns, and for most terms their phase.
// A warp's partner reads are XOR images of its own consecutive units, so they never conflict.
//
// fp32 multiplies each value by its phase times the class coefficient; where the element is zero it
// reads a zero unit behind the tile, so an infinity stays in the rows coupled to it.
//
// fp64 quantises the rows while staging them (one scale per column, q = round(x 2^(1078 - E_c))),
// sums each class's run exactly in 64-bit integers and multiplies the sums by the class
// coefficients in fixed point (rounded high halves of 64 x 64-bit products, tile_fix).  The partial sums
// stay integers from pass to pass; the last one converts once, so an element is rounded twice, in
// the conversion and with the diagonal, whatever the number of classes and passes.
//
// Measured on GB300, one mTPQ step of 64 starts against the gather kernel: 2^24 rows c64 26.3 ms
// instead of 49.4 ms (three passes; bound by shared-memory wavefronts, 73 %, with DRAM at 48 %),
// 2^18 rows c128 1.62 ms instead of 1.99 ms (two passes: 0.48 ms, issue 59 % and integer pipe 56 %, and
// 1.08 ms with the diagonal and the epilogue, fp64 pipe 69 %; 1.81 ms with a conversion per class and pass);
// 16 starts, 2^24 rows c64 28.2 instead of 156 ms for four steps.
#include <math.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "epilogue.cuh"
#include "quant.cuh"
#include "reduce.cuh"

namespace hphi {

namespace {

constexpr int kTileUnits = 4096;     // units of 16 bytes per tile
constexpr int kTileBytes = kTileUnits * 16;  // a zero unit follows
constexpr int kTileSteps = kTileUnits / kThreads;  // rows per thread
static_assert(kTileSteps == 16, "a thread's rows are numbered by four local bits");
constexpr int kTileRows = 1024;      // most rows per tile (U >= 4)

template <class S> struct TileUnit {
  static constexpr bool kF64 = Traits<S>::kF64;
  using T = std::conditional_t<kF64, long long, float>;  // staged scalar
  static constexpr int NC = 16 / (int)sizeof(S);         // columns per unit
};

// change of an entry's phase index on the thread's row r (its two bits per row bit, host-made)
__device__ __forceinline__ uint32_t tile_flip(const TileEntry& en, int r) {
  return (((r & 1) ? en.flip : 0u) ^ ((r & 2) ? en.flip >> 2 : 0u) ^ ((r & 4) ? en.flip >> 4 : 0u)) & 3u;
}

// a b / 2^64, rounded to nearest (so a zero sum stays zero)
__device__ __forceinline__ long long tile_mul(long long a, long long b) {
  return (long long)(((__int128)a * b + ((__int128)1 << 63)) >> 64);
}

// (ar, ai) += phase(code) * (xr, xi) of NR rows; one branch for all of them
template <int NR>
__device__ __forceinline__ void tile_phase(int code, const long long (*x)[2], long long (*a)[2], bool cplx) {
  if (!cplx) {
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      if (code == 1) {
        a[r][0] += x[r][0];
        a[r][1] += x[r][1];
      } else if (code) {
        a[r][0] -= x[r][0];
        a[r][1] -= x[r][1];
      }
    }
    return;
  }
  switch (code) {
    case 1:
#pragma unroll
      for (int r = 0; r < NR; ++r) { a[r][0] += x[r][0]; a[r][1] += x[r][1]; }
      break;
    case 2:
#pragma unroll
      for (int r = 0; r < NR; ++r) { a[r][0] -= x[r][1]; a[r][1] += x[r][0]; }
      break;
    case 3:
#pragma unroll
      for (int r = 0; r < NR; ++r) { a[r][0] -= x[r][0]; a[r][1] -= x[r][1]; }
      break;
    case 4:
#pragma unroll
      for (int r = 0; r < NR; ++r) { a[r][0] += x[r][1]; a[r][1] -= x[r][0]; }
      break;
    default: break;
  }
}

template <class R>
__device__ __forceinline__ R tile_diag(const SpinDev& md, uint32_t s) {
  R d = (R)md.c0;
  for (int g = 0; g < md.n_lin; ++g) {
    const LinGroup lg = md.lin[g];
    d += (R)lg.coef * (R)__popc(s & (uint32_t)lg.mask);
  }
  int grp = md.n_pairs ? md.pairs[0].grp : 0, cnt = 0;
  for (int p = 0; p < md.n_pairs; ++p) {
    const PairEntry pe = md.pairs[p];
    if (pe.grp != grp) {
      d += (R)md.pair_coef[grp] * (R)cnt;
      cnt = 0;
      grp = pe.grp;
    }
    cnt += (int)((s >> pe.i) & (s >> pe.j) & 1u);
  }
  if (md.n_pairs) d += (R)md.pair_coef[grp] * (R)cnt;
  return d;
}

// HOLES (fp32): some entry of the pass is zero for some settings of its bits
template <class S, Epi E, bool LAST, bool HOLES>
__global__ void __launch_bounds__(kThreads, 3)
    k_hv_tile(const SpinDev md, const TilePass tp, const S* __restrict__ v, S* out, int nvec, FusedArgs fa,
              const int* __restrict__ Ec) {
  using R = typename Traits<S>::R;
  using T = typename TileUnit<S>::T;
  constexpr bool C = Traits<S>::kCplx, F64 = Traits<S>::kF64;
  constexpr int NC = TileUnit<S>::NC, NW = 16 / (int)sizeof(T);  // columns, scalars per unit
  constexpr int NR = (F64 || LAST) ? 4 : 8;                      // rows in flight per thread
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ TileEntry s_ent[kTileMaxEntries];
  __shared__ float2 s_ph[F64 ? 1 : kTileMaxEntries][4];  // entry's class coefficient times its phase, by row bits
  __shared__ R s_d[LAST ? kTileRows : 1];          // diagonal element of the tile's rows

  if (fa.done != nullptr && *fa.done) return;
  const int tid = threadIdx.x;
  const int ne = tp.n_ent;
  if (tid < 4) reinterpret_cast<uint32_t*>(smem_raw + kTileBytes)[tid] = 0u;
  for (int k = tid; k < ne; k += kThreads) s_ent[k] = tp.ents[k];
  if constexpr (!F64) {
    for (int k = tid; k < ne * 4; k += kThreads) {
      const TileEntry en = tp.ents[k >> 2];
      const double2 c = md.cls_coef[en.cls];
      const int code = (en.phases >> (3 * (k & 3))) & 7;  // 0 (none), 1 (+1), 2 (+i), 3 (-1), 4 (-i)
      double re = 0.0, im = 0.0;
      if (code == 1) { re = c.x; im = c.y; }
      if (code == 2) { re = -c.y; im = c.x; }
      if (code == 3) { re = -c.x; im = -c.y; }
      if (code == 4) { re = c.y; im = -c.x; }
      s_ph[k >> 2][k & 3] = make_float2((float)re, (float)im);
    }
  }
  const int t = tp.t, lgU = 12 - t, U = 1 << lgU, lb = t - 4;
  const int h = tid & (U - 1), lrow = tid >> lgU;
  const int nch = nvec / (U * NC);
  const int ch = (int)(blockIdx.x % (unsigned)nch);
  const int col = (ch * U + h) * NC;  // first column of this thread
  const int64_t n_sets = md.dim >> t;
  const int64_t step = gridDim.x / (unsigned)nch;
  uint32_t rlow = 0u;
  for (int b = 0; b < lb; ++b) rlow |= ((uint32_t)(lrow >> b) & 1u) << tp.pos[b];
  const uint32_t kb0 = 1u << tp.pos[lb], kb1 = 1u << tp.pos[lb + 1], kb2 = 1u << tp.pos[lb + 2], kb3 = 1u << tp.pos[lb + 3];
  auto kbits = [&](int k) -> uint32_t {
    return (k & 1 ? kb0 : 0u) | (k & 2 ? kb1 : 0u) | (k & 4 ? kb2 : 0u) | (k & 8 ? kb3 : 0u);
  };
  const uint32_t rowb = 16u << lgU;  // bytes per tile row
  const uint32_t off0 = (uint32_t)lrow * rowb + 16u * (uint32_t)h;
  const uint32_t kstride = rowb << lb;  // byte distance of a thread's consecutive rows
  unsigned char* tb = smem_raw;
  int eq[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) eq[q] = F64 ? Ec[col + q] : 0;
  using H = std::conditional_t<F64, long long, float>;  // a row's sums, fp64 in units of 2^(fix_exp + eq - 1078)
  const EpiScalars<R> es = epi_scalars<R, E>(fa);
  R inv[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) inv[q] = (LAST && E == Epi::kTpq) ? opaque((R)fa.scal[col + q]) : (R)0;
  // fp64: X_{k+1} = (inv l) x - (inv / N_s) h, one product and one multiply-add a number
  R il[NC], in_[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    il[q] = F64 ? inv[q] * es.l : (R)0;
    in_[q] = F64 ? inv[q] * es.ins : (R)0;
  }
  constexpr int NQ = n_red<E>() > 0 ? n_red<E>() : 1;
  Red<F64, NQ> red[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) red[q].zero();

  for (int64_t set = blockIdx.x / (unsigned)nch; set < n_sets; set += step) {
    const uint32_t vi = (uint32_t)(set << t);
    const uint32_t rbase = __ldg(tp.dep + (vi & 255u)) | __ldg(tp.dep + 256 + ((vi >> 8) & 255u)) |
                           __ldg(tp.dep + 512 + ((vi >> 16) & 255u)) | __ldg(tp.dep + 768 + (vi >> 24));
    const uint32_t s0 = rbase | rlow;
    __syncthreads();  // the previous tile is no longer read
    if constexpr (!F64) {
#pragma unroll
      for (int k = 0; k < kTileSteps; ++k)
        copy_async<16>(tb + off0 + k * kstride, v + (int64_t)(s0 | kbits(k)) * nvec + col);
    } else {
#pragma unroll 4
      for (int k = 0; k < kTileSteps; ++k) {
        const double2 x = __ldg(reinterpret_cast<const double2*>(v + (int64_t)(s0 | kbits(k)) * nvec + col));
        longlong2 q;
        q.x = quant_one(x.x, eq[0]);
        q.y = quant_one(x.y, eq[NC - 1]);
        *reinterpret_cast<longlong2*>(tb + off0 + k * kstride) = q;
      }
    }
    if constexpr (LAST) {
      for (int i = tid; i < (1 << t); i += kThreads) {
        uint32_t s = rbase;
        for (int b = 0; b < t; ++b) s |= ((uint32_t)(i >> b) & 1u) << tp.pos[b];
        s_d[i] = tile_diag<R>(md, s);
      }
    }
    if constexpr (!F64) asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    for (int k0 = 0; k0 < kTileSteps; k0 += NR) {
      H hs[NR][NW];  // the row's sums: NW scalars (re, im pairs or columns)
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        if (tp.first) {
#pragma unroll
          for (int e = 0; e < NW; ++e) hs[r][e] = (H)0;
        } else {
          const uint4 p = __ldcs(reinterpret_cast<const uint4*>(out + (int64_t)(s0 | kbits(k0 + r)) * nvec + col));
          memcpy(&hs[r][0], &p, 16);
        }
      }
      T ac[F64 ? NR : 1][2];
      auto flush = [&](int cls) {
        if constexpr (F64) {
          const longlong2 cf = __ldg(tp.fix + cls);
#pragma unroll
          for (int r = 0; r < NR; ++r) {
            const long long v0 = ac[r][0] << tp.fix_shift, v1 = ac[r][1] << tp.fix_shift;
            hs[r][0] += tile_mul(v0, cf.x);
            hs[r][1] += tile_mul(v1, cf.x);
            if (C && cf.y != 0) {
              hs[r][0] -= tile_mul(v1, cf.y);
              hs[r][1] += tile_mul(v0, cf.y);
            }
          }
#pragma unroll
          for (int r = 0; r < NR; ++r)
#pragma unroll
            for (int e = 0; e < 2; ++e) ac[r][e] = 0;
        }
      };
      if constexpr (F64) {
#pragma unroll
        for (int r = 0; r < NR; ++r)
#pragma unroll
          for (int e = 0; e < 2; ++e) ac[r][e] = 0;
      }
      const uint32_t g0 = off0 + (uint32_t)k0 * kstride;
      const uint32_t sg = s0 | kbits(k0);
      int cur = ne ? s_ent[0].cls : 0;
      for (int n = 0; n < ne; ++n) {
        const TileEntry en = s_ent[n];
        if (F64 && en.cls != cur) {  // the entries are the same for all threads
          flush(cur);
          cur = en.cls;
        }
        T x[NR][NW];
        const uint32_t sel = ((sg >> en.i) & 1u) | (((sg >> en.j) & 1u) << 1);
#pragma unroll
        for (int r = 0; r < NR; ++r) {
          uint32_t o = (g0 + (uint32_t)r * kstride) ^ (en.lmask << (4 + lgU));
          if (HOLES && !((en.flags >> (kTileLive + (sel ^ tile_flip(en, r)))) & 1)) o = (uint32_t)kTileBytes;
          const uint4 p = *reinterpret_cast<const uint4*>(tb + o);
          memcpy(&x[r][0], &p, 16);
        }
        const bool per_row = (en.flags & (NR == 8 ? kTilePerRow8 : kTilePerRow4)) != 0;
        if constexpr (!F64) {
          const float2* tab = s_ph[n];
          float2 ph = tab[sel];
          const bool real = (en.flags & kTileReal) != 0;
#pragma unroll
          for (int r = 0; r < NR; ++r) {
            if (r > 0 && per_row) ph = tab[sel ^ tile_flip(en, r)];
            if (!C || real) {
#pragma unroll
              for (int e = 0; e < NW; ++e) hs[r][e] = fmaf(ph.x, x[r][e], hs[r][e]);
            } else {
              hs[r][0] = fmaf(ph.x, x[r][0], fmaf(-ph.y, x[r][1], hs[r][0]));
              hs[r][1] = fmaf(ph.x, x[r][1], fmaf(ph.y, x[r][0], hs[r][1]));
              hs[r][2] = fmaf(ph.x, x[r][2], fmaf(-ph.y, x[r][3], hs[r][2]));
              hs[r][3] = fmaf(ph.x, x[r][3], fmaf(ph.y, x[r][2], hs[r][3]));
            }
          }
        } else if (!per_row) {
          tile_phase<NR>((en.phases >> (3 * sel)) & 7, x, ac, C);
        } else {
#pragma unroll
          for (int r = 0; r < NR; ++r)
            tile_phase<1>((en.phases >> (3 * (sel ^ tile_flip(en, r)))) & 7, x + r, ac + r, C);
        }
      }
      if (F64 && ne) flush(cur);
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const int64_t idx = (int64_t)(sg | kbits(r)) * nvec + col;
        if constexpr (LAST) {
          R x0[NW];  // the row's own value: exact in fp64 (read again), from the tile in fp32
          {
            uint4 p;
            if constexpr (F64) p = __ldg(reinterpret_cast<const uint4*>(v + idx));
            else p = *reinterpret_cast<const uint4*>(tb + g0 + (uint32_t)r * kstride);
            memcpy(x0, &p, 16);
          }
          const R d = s_d[lrow + ((k0 + r) << lb)];
          R hv[NW];
#pragma unroll
          for (int e = 0; e < NW; ++e) {
            if constexpr (F64) hv[e] = fma(d, x0[e], fix_to_double(hs[r][e], eq[C ? 0 : e] + tp.fix_exp - 1078));
            else hv[e] = fma(d, x0[e], hs[r][e]);
          }
          if constexpr (E == Epi::kTpq) {
#pragma unroll
            for (int e = 0; e < NW; ++e) {
              const int q = C ? e / 2 : e;
              red[q].add(0, x0[e], hv[e]);
              red[q].add(1, hv[e], hv[e]);
              if constexpr (F64) hv[e] = fma(-in_[q], hv[e], il[q] * x0[e]);
              else hv[e] = inv[q] * (es.l * x0[e] - hv[e] * es.ins);
            }
#pragma unroll
            for (int q = 0; q < NC; ++q) red[q].tick();
          }
          uint4 p;
          memcpy(&p, &hv[0], 16);
          *reinterpret_cast<uint4*>(out + idx) = p;
        } else {
          uint4 p;
          memcpy(&p, &hs[r][0], 16);
          __stcs(reinterpret_cast<uint4*>(out + idx), p);
        }
      }
    }
  }
  if constexpr (LAST && E == Epi::kTpq) {
    // per-column sums in a fixed order; columns of other CTAs' chunks get zeros from this one
    double* s_red = reinterpret_cast<double*>(smem_raw);
    const int cw = U * NC, rows = kThreads >> lgU;
#pragma unroll
    for (int k = 0; k < n_red<E>(); ++k) {
      __syncthreads();
#pragma unroll
      for (int q = 0; q < NC; ++q) s_red[lrow * cw + h * NC + q] = red[q].get(k);
      __syncthreads();
      for (int c = tid; c < nvec; c += kThreads) {
        double sum = 0.0;
        const int l = c - ch * cw;
        if (l >= 0 && l < cw)
          for (int r = 0; r < rows; ++r) sum += s_red[r * cw + l];
        fa.partials[((size_t)blockIdx.x * nvec + c) * kMaxRedQ + k] = sum;
      }
    }
  }
}

constexpr size_t kTileSmem = kTileBytes + 16;

template <class S, Epi E, bool LAST, bool HOLES>
Status launch_holes(const SpinDev& md, const TilePass& tp, const void* v, void* out, int nvec, const FusedArgs& fa,
                   int grid, const int* Ec, cudaStream_t st) {
  HPHI_CUDA_TRY(cudaFuncSetAttribute(k_hv_tile<S, E, LAST, HOLES>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTileSmem));
  k_hv_tile<S, E, LAST, HOLES><<<grid, kThreads, kTileSmem, st>>>(md, tp, reinterpret_cast<const S*>(v),
                                                           reinterpret_cast<S*>(out), nvec, fa, Ec);
  HPHI_CUDA_TRY(cudaGetLastError());
  return {};
}

template <class S, Epi E, bool LAST>
Status launch_pass(const SpinDev& md, const TilePass& tp, const void* v, void* out, int nvec, const FusedArgs& fa,
                   int grid, const int* Ec, cudaStream_t st) {
  if constexpr (!Traits<S>::kF64)
    if (tp.holes) return launch_holes<S, E, LAST, true>(md, tp, v, out, nvec, fa, grid, Ec, st);
  return launch_holes<S, E, LAST, false>(md, tp, v, out, nvec, fa, grid, Ec, st);
}

template <class S>
Status launch_s(const SpinDev& md, const TilePlan& plan, const void* v, void* w, void* scratch, int nvec, Epi epi,
                const FusedArgs& fa, int grid, cudaStream_t st) {
  int* Ec = nullptr;
  if constexpr (Traits<S>::kF64) {
    Ec = reinterpret_cast<int*>(scratch);
    Status s = launch_maxexp_cols(reinterpret_cast<const double*>(v), md.dim, nvec, Traits<S>::kCplx ? 2 : 1, Ec, st);
    if (s.code) return s;
  }
  void* out = epi == Epi::kTpq ? fa.out : w;
  for (int p = 0; p < plan.n_pass; ++p) {
    TilePass tp = plan.pass[p];
    tp.first = p == 0;
    Status s;
    if (p + 1 < plan.n_pass) s = launch_pass<S, Epi::kStore, false>(md, tp, v, out, nvec, fa, grid, Ec, st);
    else if (epi == Epi::kTpq) s = launch_pass<S, Epi::kTpq, true>(md, tp, v, out, nvec, fa, grid, Ec, st);
    else s = launch_pass<S, Epi::kStore, true>(md, tp, v, out, nvec, fa, grid, Ec, st);
    if (s.code) return s;
  }
  return {};
}

}  // namespace

// The integers of fp64.  A class sum S of a pass is below 2^56 times its longest run, so
// S 2^shift fits 63 bits with shift = 7 - log2(run); the coefficients times 2^s fit 63 bits with
// s = 62 - log2(c_max); and the sum of all products over 2^64 must stay below 2^62, which lowers
// first the shift, then s.  Products are rounded to nearest (with a shift of two or more those with
// c_max = 2^k are exact); against the whole vector that is below the rounding of the elements (rms over
// the norm, 18-site Heisenberg ring in a field of 1e-3: 0.60 2^-53, the gather kernel 0.77).  Rows that
// only a coefficient c reaches lose a further c_max / (12 c) of their own rounding, so models whose
// coefficients span more than 1,024 keep to the gather kernels.
static void tile_fix(const std::vector<SpinEntry>& ents, const std::vector<double2>& cls, TileHost* out) {
  double cmax = 0.0, cmin = 1e308, sum = 0.0;
  for (const SpinEntry& e : ents) {
    for (double c : {fabs(cls[e.cls].x), fabs(cls[e.cls].y)}) {
      if (c == 0.0) continue;
      cmax = std::max(cmax, c);
      cmin = std::min(cmin, c);
      sum += c;
    }
  }
  int run = 1;
  for (int p = 0; p < out->n_pass; ++p)
    for (int k = out->e0[p], r = 0; k < out->e0[p + 1]; ++k) {
      r = (k > out->e0[p] && out->ents[k].cls == out->ents[k - 1].cls) ? r + 1 : 1;
      run = std::max(run, r);
    }
  out->fix.assign(cls.size(), longlong2{0, 0});
  out->f64 = run <= 127 && cmax > 0.0 && cmin >= cmax / 1024 && cmax < 1e300 && cmin > 1e-290;
  if (!out->f64) return;
  const int lg = std::ilogb(cmax);
  int s = 62 - lg, run2 = 0, sum2 = 0;
  while ((1 << run2) < run) ++run2;
  while (std::ldexp(cmax, sum2) < sum * 1.001) ++sum2;  // sum <= 2^(lg + 1 + sum2)
  out->fix_shift = std::min(7 - run2, 7 - sum2);
  if (out->fix_shift < 0) {
    s += out->fix_shift;
    out->fix_shift = 0;
  }
  out->fix_exp = 64 - s - out->fix_shift;
  for (size_t k = 0; k < cls.size(); ++k)
    out->fix[k] = longlong2{std::llrint(std::ldexp(cls[k].x, s)), std::llrint(std::ldexp(cls[k].y, s))};
}

// Covers the flip masks by site sets of at most t sites: the set grows by the mask that covers
// most new masks per added site (ties: the one whose new sites fewest masks touch, which walks
// chains from their ends), those that touch the set first, until none fits.  False when more than kMaxPasses sets, more than
// kTileMaxEntries entries in one, or a mask wider than t sites; below 13 sites no block of vectors
// has enough tiles (tile_choose).
bool batch_tile_plan(int n_sites, int t, const std::vector<SpinEntry>& ents, const std::vector<double2>& cls, TileHost* out) {
  out->ents.clear();
  out->dep.clear();
  out->n_pass = 0;
  if (t < 8 || t > 10 || n_sites < 13 || n_sites > 32 || ents.empty() || (int)ents.size() > 512) return false;
  auto pc = [](uint32_t x) { return __builtin_popcount(x); };
  // distinct masks of the entries not placed yet, in the entries' order, with their counts
  uint32_t masks[512];
  int counts[512], n_masks = 0;
  for (const SpinEntry& e : ents) {
    int k = 0;
    while (k < n_masks && masks[k] != (uint32_t)e.mask) ++k;
    if (k == n_masks) {
      masks[n_masks] = (uint32_t)e.mask;
      counts[n_masks++] = 0;
    }
    ++counts[k];
  }
  std::vector<int> pass_of(ents.size(), -1);
  while (n_masks > 0) {
    if (out->n_pass >= kMaxPasses) return false;
    uint32_t S = 0;
    for (int cov0 = 0;;) {
      double bg = -1.0;
      int bd = 0, bc = 0;
      uint32_t bU = 0;
      for (int near = S ? 1 : 0; near >= 0 && bg < 0.0; --near) {
        for (int k = 0; k < n_masks; ++k) {
          const uint32_t U = S | masks[k];
          if (U == S || (near && !(masks[k] & S)) || pc(U) > t) continue;
          const uint32_t out_of_U = ~U, added = U & ~S;
          int cov = 0, deg = 0;
          for (int o = 0; o < n_masks; ++o) {
            cov += (masks[o] & out_of_U) == 0u ? counts[o] : 0;
            deg += (masks[o] & added) != 0u ? counts[o] : 0;
          }
          const double gain = (double)(cov - cov0) / (pc(U) - pc(S));
          if (gain > bg || (gain == bg && deg < bd)) {
            bg = gain;
            bd = deg;
            bc = cov;
            bU = U;
          }
        }
      }
      if (bg < 0.0) break;
      S = bU;
      cov0 = bc;
    }
    if (S == 0) return false;  // a mask wider than t sites
    const int p = out->n_pass++;
    out->e0[p] = (int)out->ents.size();
    for (size_t k = 0; k < ents.size(); ++k)
      if (pass_of[k] < 0 && ((uint32_t)ents[k].mask & ~S) == 0) pass_of[k] = p;
    int kept = 0;
    for (int k = 0; k < n_masks; ++k)
      if (masks[k] & ~S) {
        masks[kept] = masks[k];
        counts[kept++] = counts[k];
      }
    n_masks = kept;
    for (int b = 0; b < n_sites && pc(S) < t; ++b) S |= 1u << b;  // whole tiles
    // local positions: the four highest bits number a thread's rows, the first of them innermost,
    // so the sites that fewest of the pass's entries read go there (the phase is then the same
    // for a thread's rows), the least read first
    std::vector<std::pair<int, int>> use;
    for (int b = 0; b < n_sites; ++b)
      if ((S >> b) & 1u) {
        int n = 0;
        for (size_t k = 0; k < ents.size(); ++k) n += pass_of[k] == p && (ents[k].i == b || ents[k].j == b);
        use.emplace_back(-n, b);
      }
    std::stable_sort(use.begin(), use.end());
    std::reverse(use.end() - 4, use.end());
    for (int l = 0; l < t; ++l) out->pos[p][l] = (uint8_t)use[l].second;
    for (size_t k = 0; k < ents.size(); ++k) {  // input is class-sorted; keep that order
      if (pass_of[k] != p) continue;
      TileEntry e{};
      for (int l = 0; l < t; ++l)
        if ((ents[k].mask >> use[l].second) & 1ull) e.lmask |= 1u << l;
      e.i = ents[k].i;
      e.j = ents[k].j;
      e.phases = ents[k].phases;
      e.cls = ents[k].cls;
      bool real = true;
      int live = e.i == e.j ? 6 : 0;  // (settings that a one-site term never reads)
      for (int s = 0; s < 4; ++s) {
        const int code = (ents[k].phases >> (3 * s)) & 7;
        real = real && (code == 0 || code == 1 || code == 3);
        if (code) live |= 1 << s;
      }
      e.flags |= (uint16_t)(live << kTileLive);
      if (live != 15) out->holes[p] = 1;
      if (real && cls[ents[k].cls].y == 0.0) e.flags |= kTileReal;
      for (int b = 0; b < 3; ++b) {
        const int site = use[t - 4 + b].second;
        const uint32_t f = (e.i == site ? 1u : 0u) | (e.j == site ? 2u : 0u);
        e.flip |= f << (2 * b);
        if (f && b < 2) e.flags |= kTilePerRow4;
        if (f) e.flags |= kTilePerRow8;
      }
      out->ents.push_back(e);
    }
    if ((int)out->ents.size() - out->e0[p] > kTileMaxEntries) return false;
    // visit index bit -> row bit: the set's sites first, then the others
    int pos[32], n = 0;
    for (int l = 0; l < t; ++l) pos[n++] = out->pos[p][l];
    for (int b = 0; b < n_sites; ++b)
      if (!((S >> b) & 1u)) pos[n++] = b;
    const size_t d0 = out->dep.size();
    out->dep.resize(d0 + 1024, 0u);
    for (int byte = 0; byte < 4; ++byte)
      for (int val = 1; val < 256; ++val) {  // the value without its lowest bit, and that bit
        const int bit = byte * 8 + __builtin_ctz((unsigned)val);
        out->dep[d0 + byte * 256 + val] = out->dep[d0 + byte * 256 + (val & (val - 1))] | (bit < n_sites ? 1u << pos[bit] : 0u);
      }
  }
  out->e0[out->n_pass] = (int)out->ents.size();
  tile_fix(ents, cls, out);
  return true;
}

bool tile_applies(const SpinDev& md, int prec, bool cplx, int nvec, Epi epi) {
  const int esz = (prec == HPHI_FP64 ? 8 : 4) * (cplx ? 2 : 1);
  return md.sector == 0 && md.n_sites >= 13 && md.n_sites <= 32 && nvec >= 2 && (nvec & (nvec - 1)) == 0 &&
         nvec <= kMaxNvec && nvec * esz >= 64 && (epi == Epi::kStore || epi == Epi::kTpq);
}

// Tiles of one pass of the plan (t sites): row sets times column chunks.
static int64_t tile_count(const SpinDev& md, int t, int nvec, int esz) {
  return (md.dim >> t) * ((int64_t)nvec * esz / (16 << (12 - t)));
}

// The plan of fewest block transfers (3 passes - 1, a tenth more for 64-byte row pieces), among
// those whose row piece divides the row, that have two tiles for every SM; null: the gather
// kernels.  Below that the passes are too short to fill the chip.  Smallest cases above the line,
// four mTPQ steps with their start block on GB300, tiles against gathers: 2^16 rows x 64 c64 (512
// tiles) 0.49 against 0.71 ms, x 32 c128 1.24 against 1.56 ms,
// 2^18 rows x 16 c64 0.59 against 2.03 ms, 2^20 rows x 8 c64 1.02 against 4.16 ms.
const TilePlan* tile_choose(const TilePlan* plans, const SpinDev& md, int prec, bool cplx, int nvec, Epi epi) {
  if (!tile_applies(md, prec, cplx, nvec, epi)) return nullptr;
  const int esz = (prec == HPHI_FP64 ? 8 : 4) * (cplx ? 2 : 1);
  const TilePlan* best = nullptr;
  double bc = 1e30;
  for (int t = 8; t <= 10; ++t) {
    const TilePlan& pl = plans[t - 8];
    if (pl.n_pass == 0 || (16 << (12 - t)) > nvec * esz) continue;
    if (prec == HPHI_FP64 && !pl.f64) continue;
    if (tile_count(md, t, nvec, esz) < 2 * num_sms()) continue;
    const double c = (3.0 * pl.n_pass - 1.0) * (t == 10 ? 1.1 : 1.0);
    if (c < bc) {
      bc = c;
      best = &pl;
    }
  }
  return best;
}

// three resident CTAs per SM, a whole number of CTAs per column chunk
int tile_grid(const TilePlan& plan, const SpinDev& md, int prec, bool cplx, int nvec) {
  const int esz = (prec == HPHI_FP64 ? 8 : 4) * (cplx ? 2 : 1);
  const int t = plan.pass[0].t, nch = nvec * esz / (16 << (12 - t));
  const int64_t per = std::min<int64_t>(md.dim >> t, std::max(1, 3 * num_sms() / nch));
  return (int)(per * nch);
}

size_t tile_scratch_bytes(int prec, int nvec) { return prec == HPHI_FP64 ? sizeof(int) * (size_t)nvec : 0; }

Status launch_tile(const SpinDev& md, const TilePlan& plan, int prec, bool cplx, const void* v, void* w, void* scratch,
                   int nvec, Epi epi, const FusedArgs& fa, int grid, cudaStream_t st) {
  if (prec == HPHI_FP64)
    return cplx ? launch_s<double2>(md, plan, v, w, scratch, nvec, epi, fa, grid, st)
                : launch_s<double>(md, plan, v, w, scratch, nvec, epi, fa, grid, st);
  return cplx ? launch_s<float2>(md, plan, v, w, scratch, nvec, epi, fa, grid, st)
              : launch_s<float>(md, plan, v, w, scratch, nvec, epi, fa, grid, st);
}

}  // namespace hphi

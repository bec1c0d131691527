// Two-pass H v for Hubbard models with real hopping and one hopping value per spin
// species (the half-filled square-lattice workloads): section 3.3's on-the-fly product,
// laid out for GB300's memory hierarchy.
//
// The amplitudes form a matrix X[d][u] (down-spin rank d, up-spin rank u).  Down-spin
// hops combine whole rows (W[d][:] = sum_q +-X[d'_q][:]) and up-spin hops act inside a row
// (sum_q +-X[d][u'_q]).  So:
//   pass D  walks column stripes in stripe-major order; the stripe of every row stays in
//           L2 while all rows of that stripe are combined, so X is read from HBM about once.
//           W receives the plain signed sums.
//   pass U  stages K whole rows of X in shared memory, applies the up-spin gather table
//           (built once per sector on the device) to all K rows at once, adds diag * X and
//           coef * W, and runs the fused Lanczos / mTPQ epilogue.
// fp64 sums use the exact fixed-point accumulator (integer pipes); fp32 sums are plain.
#include <algorithm>
#include <mutex>
#include <string>
#include <type_traits>

#include "common.cuh"
#include "epilogue.cuh"
#include "gather.cuh"
#include "quant.cuh"
#include "reduce.cuh"

namespace hphi {

// ------------------------------------------------------------------ allocation-free scratch
// Scratch of hphi_apply_H_noalloc: the int64 copy of the input, the int64 down-spin sums and
// the scale word of the fixed-point fp64 path (16 bytes per row + 256).  It is a file-scope
// device array, so every GPU that loads this library holds these 64 MiB until the process
// exits, and every call on a device shares it.  Host code must not use the symbol as a
// pointer: its device address comes from cudaGetSymbolAddress (noalloc_scratch below).
constexpr size_t kNoAllocScratchBytes = (size_t)64 << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

namespace {

// 16-byte pieces per lane of pass D unless hphi_autotune has chosen (a warp's stripe is 32 times
// that wide): two, or one where wider stripes would leave fewer than two rounds of warps (4x3
// torus, 6 + 5 electrons, fp64 product 0.052 against 0.057 ms)
constexpr int kDnPieces = 2;

// K consecutive values of a shared-memory row tile with the widest aligned accesses
template <class R, int K>
__device__ __forceinline__ void load_k(const R* p, R* out) {
  if constexpr (sizeof(R) * K == 16) {
    if constexpr (sizeof(R) == 4) {
      const float4 t = *reinterpret_cast<const float4*>(p);
      out[0] = t.x; out[1] = t.y; out[2] = t.z; out[3] = t.w;
    } else {
      const longlong2 t = *reinterpret_cast<const longlong2*>(p);
      out[0] = t.x; out[1] = t.y;
    }
  } else if constexpr (sizeof(R) * K == 8 && sizeof(R) == 4) {
    const float2 t = *reinterpret_cast<const float2*>(p);
    out[0] = t.x; out[1] = t.y;
  } else {
#pragma unroll
    for (int m = 0; m < K; ++m) out[m] = p[m];
  }
}

constexpr int kZeroBytes = 128;      // gather_lanes(4 .. 16) entries
constexpr int kSmemBudget = 208000;  // shared-memory bytes of the row tile (plus its zero entries and ~7 KB static)

// neighbour table of one species: the q-th active hop target of state k (rank | sign << 31) at
// nbr[q * n + k] for the up species (threads of consecutive states read consecutive words) and
// at nbr[k * maxdeg_dn + q] for the down species (a warp reads one state's list)
__global__ void k_hub_nbr(const HubDev md, int species, uint32_t* __restrict__ nbr, uint8_t* __restrict__ deg,
                          uint8_t* __restrict__ npos) {
  const int64_t n = species ? md.dim_dn : md.dim_up;
  const int e0 = species ? md.n_up_hops : 0;
  const int ne = species ? md.n_dn_hops : md.n_up_hops;
  const uint32_t* list = species ? md.list_dn : md.list_up;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t b = md.sector ? list[k] : (uint32_t)k;
    // positive-sign targets first, then negative ones (hop order within each group)
    int cnt = 0, np = 0;
    for (int pass = 0; pass < 2; ++pass) {
      for (int q = 0; q < ne; ++q) {
        const HopEntry h = md.hops[e0 + q];
        if (((b >> h.i) ^ (b >> h.j)) & 1u) {
          const uint32_t sg = (uint32_t)(__popc(b & h.between) & 1);
          if ((int)sg != pass) continue;
          const uint32_t b2 = b ^ h.mask;
          const uint32_t r2 = md.sector ? md.rank[b2] : b2;
          nbr[species ? k * md.maxdeg_dn + cnt : (int64_t)cnt * n + k] = r2 | (sg << 31);
          ++cnt;
        }
      }
      if (pass == 0) np = cnt;
    }
    deg[k] = (uint8_t)cnt;
    if (npos != nullptr) npos[k] = (uint8_t)np;
  }
}

// Pass D: W[d][u] = sum over down-spin neighbours d' of d of +-X[d'][u].  A warp item is one row
// and a stripe of 32 * P 16-byte pieces; items run stripe by stripe, claimed in order from a
// counter, so all CTAs stay on neighbouring rows of one stripe and that stripe of all rows stays
// in L2.  Lane q holds the row's neighbour q and shuffles broadcast it; the list is sign-sorted,
// entries [0, npos) add and the rest subtract.  VEC: rows start on 16 bytes, one load a piece;
// otherwise element by element.
//
// Bound by the loads from L2 (17 neighbours a row on average: 13.6 TB/s).  Measured on GB300
// against 256 single elements a CTA and claim: 16 sites, 8 + 8 electrons, int64 1.65 ms instead of
// 2.37 ms; 7 + 6 electrons, fp32 0.37 instead of 0.50 ms; 18 sites, 9 + 9, fp32 11.8 instead of
// 16.1 ms.
template <class R, int P, bool VEC>
__global__ void __launch_bounds__(kThreads) k_hub_dn(const HubDev md, const R* __restrict__ X, R* __restrict__ W,
                                                     const int* __restrict__ done,
                                                     unsigned long long* __restrict__ next_item, int claim) {
  if (done != nullptr && *done) return;
  constexpr int PV = 16 / (int)sizeof(R), NE = P * PV, SW = 32 * NE;
  constexpr int kWarps = kThreads / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t dim_up = md.dim_up, dim_dn = md.dim_dn;
  const int64_t n_items = ((dim_up + SW - 1) / SW) * dim_dn;
  __shared__ int64_t s_item;
  for (bool first = true;; first = false) {
    int64_t base = (int64_t)blockIdx.x * kWarps;
    if (claim > 0) {
      __syncthreads();
      if (tid == 0) s_item = (int64_t)atomicAdd(next_item, (unsigned long long)(kWarps * claim));
      __syncthreads();
      base = s_item;
    }
    if (base >= n_items || (claim == 0 && !first)) break;
    int64_t s = base / dim_dn, d = base - s * dim_dn + warp;  // the CTA's warps on neighbouring rows
    for (int it = 0; it < max(claim, 1); ++it, d += kWarps) {
      while (d >= dim_dn) {  // (the warp's offset or the next round runs into the next stripe)
        d -= dim_dn;
        ++s;
      }
      const int64_t u0 = s * SW;
      if (u0 >= dim_up) break;
      const int deg = __ldg(md.deg_dn + d), npos = __ldg(md.npos_dn + d);
      const bool full = u0 + SW <= dim_up;
      // first column of element j of this lane
      auto col = [&](int j) -> int64_t { return u0 + (VEC ? ((j / PV) * 32 + lane) * PV + j % PV : j * 32 + lane); };
      R acc[NE];
#pragma unroll
      for (int j = 0; j < NE; ++j) acc[j] = (R)0;
      for (int qb = 0; qb < deg; qb += 32) {
        const int nq = min(32, deg - qb);
        const uint32_t mine = lane < nq ? __ldg(md.nbr_dn + d * md.maxdeg_dn + qb + lane) : 0u;
        for (int q0 = 0; q0 < nq; q0 += 4) {
          R x[4][NE];
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const uint32_t e = __shfl_sync(0xffffffffu, mine, (q0 + t) & 31);
            const bool on = q0 + t < nq;
            const R* src = X + (int64_t)(e & 0x7fffffffu) * dim_up;
            if constexpr (VEC) {
#pragma unroll
              for (int j = 0; j < P; ++j) {
                uint4 p = make_uint4(0u, 0u, 0u, 0u);
                if (on && (full || col(j * PV) < dim_up)) p = __ldg(reinterpret_cast<const uint4*>(src + col(j * PV)));
                memcpy(&x[t][j * PV], &p, 16);
              }
            } else {
#pragma unroll
              for (int j = 0; j < NE; ++j) x[t][j] = (on && (full || col(j) < dim_up)) ? __ldg(src + col(j)) : (R)0;
            }
          }
          const int left = npos - (qb + q0);  // of these four, so many add
          if (left >= 4) {
#pragma unroll
            for (int j = 0; j < NE; ++j) acc[j] += (x[0][j] + x[1][j]) + (x[2][j] + x[3][j]);
          } else if (left <= 0) {
#pragma unroll
            for (int j = 0; j < NE; ++j) acc[j] -= (x[0][j] + x[1][j]) + (x[2][j] + x[3][j]);
          } else {
#pragma unroll
            for (int t = 0; t < 4; ++t)
#pragma unroll
              for (int j = 0; j < NE; ++j) acc[j] += t < left ? x[t][j] : -x[t][j];
          }
        }
      }
      R* dst = W + d * dim_up;
      if constexpr (VEC) {
#pragma unroll
        for (int j = 0; j < P; ++j)
          if (full || col(j * PV) < dim_up) {
            uint4 p;
            memcpy(&p, &acc[j * PV], 16);
            __stcs(reinterpret_cast<uint4*>(dst + col(j * PV)), p);
          }
      } else {
#pragma unroll
        for (int j = 0; j < NE; ++j)
          if (full || col(j) < dim_up) __stcs(dst + col(j), acc[j]);
      }
    }
  }
}

// ------------------------------------------------------------------ fp64 via fixed point
// fp64 vectors take the gather passes as 64-bit integers on one scale per vector:
// q = round(x * 2^(1078 - E)), E = the largest exponent field of x, so |q| < 2^56 and the
// signed sums of up to 127 terms are exact integer additions (two instructions a term on
// the integer pipes instead of one fp64 add each at 1/64 rate).  Each element is rounded
// once, by at most 2^-57 max|x|; the final sums convert back to fp64 exactly rounded.

__global__ void __launch_bounds__(kThreads) k_maxexp(const double* __restrict__ X, int64_t n, int* __restrict__ E,
                                                      const int* __restrict__ done) {
  if (done != nullptr && *done) return;
  int mx = 0;
  for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads)
    mx = max(mx, (__double2hiint(__ldg(X + i)) >> 20) & 0x7ff);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) mx = max(mx, __shfl_down_sync(0xffffffffu, mx, off));
  if ((threadIdx.x & 31) == 0 && mx > 0) atomicMax(E, mx);
}

// Exponent scan and quantisation of a short vector in one CTA: one launch instead of three (the
// exponent slot's reset among them), which is what a few thousand elements wait for.  On the
// 8-site cluster (4,900 rows), with pass D's counter gone too, a product takes 20.0 us instead of
// 24.4 (three launches instead of six).  Sixteen elements a thread is what the one CTA holds in
// registers; above that the grid's bandwidth is worth more than two launches.
constexpr int kShortQuant = 16384;
__global__ void __launch_bounds__(1024) k_quant_short(const double* __restrict__ X, long long* __restrict__ Q, int n,
                                                      int* __restrict__ Ep, const int* __restrict__ done, int extra) {
  if (done != nullptr && *done) return;
  __shared__ int s_mx[32];
  constexpr int kPer = kShortQuant / 1024;
  const int tid = threadIdx.x;
  double x[kPer];
  int mx = 0;
#pragma unroll
  for (int k = 0; k < kPer; ++k) x[k] = tid + k * 1024 < n ? __ldg(X + tid + k * 1024) : 0.0;
#pragma unroll
  for (int k = 0; k < kPer; ++k) mx = max(mx, (__double2hiint(x[k]) >> 20) & 0x7ff);
  mx = (int)__reduce_max_sync(0xffffffffu, (unsigned)mx);
  if ((tid & 31) == 0) s_mx[tid >> 5] = mx;
  __syncthreads();
  mx = (int)__reduce_max_sync(0xffffffffu, (unsigned)s_mx[tid & 31]);
  if (tid == 0) *Ep = mx;
#pragma unroll
  for (int k = 0; k < kPer; ++k)
    if (tid + k * 1024 < n) Q[tid + k * 1024] = quant_one(x[k], mx + extra);
}

// extra: headroom bits; q = round(x 2^(1078 - E - extra)), |q| < 2^(56 - extra)
__global__ void __launch_bounds__(kThreads) k_quant(const double* __restrict__ X, long long* __restrict__ Q, int64_t n,
                                                     const int* __restrict__ Ep, const int* __restrict__ done,
                                                     int extra) {
  if (done != nullptr && *done) return;
  const int E = *Ep + extra;
  for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads) {
    Q[i] = quant_one(__ldg(X + i), E);
  }
}

// Pass U: up-spin hops on K rows staged in shared memory, the diagonal, + c_dn W and the fused
// epilogue.  T is float (fp32 vectors) or long long (fp64 vectors on the fixed-point copy; the
// diagonal term and the reductions take the row's own value from the same quantised tile).
//
// The K rows are interleaved (tile[u * K + m] = X[d0 + m][u]), so one load per neighbour
// fetches the value of all K rows, and every thread's terms come from a gather table
// (gather.cuh): four 16-bit targets per 8-byte record, ordered against bank conflicts, the
// signs a warp-uniform property of the slot.  W and, in Lanczos steps, the previous vector are
// loaded before the gathers.
//
// Measured on GB300, against one 4-byte signed target per term in state order: 16 sites, 8 + 8
// electrons (165,636,900 rows), fp64 Lanczos step, two rows a tile: 2.13 ms instead of 4.16 ms,
// bound by shared-memory wavefronts (71 %) and instruction issue (61 %); 7 + 6 electrons, fp32
// product, four rows: 0.55 instead of 0.90 ms; 18 sites, 9 + 9 (2,363,904,400 rows), fp32 mTPQ
// step, one 194 KB row: 26.6 instead of 64.3 ms, bound by instruction issue.  There whole chunks of
// slots that add skip the tests of each group (*; 28.1 ms without; 1 % slower with two or four rows,
// whose groups carry more work per test).
template <class T, int K, Epi E, int NT>
__global__ void __launch_bounds__(NT, (NT >= 1024) ? 1 : 2) k_hub_up(const HubDev md, const T* __restrict__ X, const T* W,
                                               const int* __restrict__ Ep, void* w, FusedArgs fa) {
  constexpr bool FIX = sizeof(T) == 8;
  using R = std::conditional_t<FIX, double, float>;
  constexpr int kWidth = K * (int)sizeof(T) >= 16 ? 2 : (K * (int)sizeof(T) >= 8 ? 1 : 0);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* tile = reinterpret_cast<T*>(smem_raw);
  __shared__ LinGroup s_ulin[kMaxLin];
  __shared__ LinGroup s_mlin[kMaxLin];
  __shared__ PairEntry s_pair[kMaxPairs];
  __shared__ R s_uc[kMaxLin], s_mc[kMaxLin], s_pcoef[kMaxPairGroups];  // coefficients in R
  __shared__ double s_red[(NT / 32) * kMaxRedQ];
  __shared__ R s_dtab[33];
  __shared__ int s_dti[33];

  if (fa.done != nullptr && *fa.done) return;
  const int tid = threadIdx.x;
  for (int k = tid; k < md.n_ulin; k += NT) { s_ulin[k] = md.ulin[k]; s_uc[k] = (R)md.ulin[k].coef; }
  for (int k = tid; k < md.n_mulin; k += NT) { s_mlin[k] = md.mulin[k]; s_mc[k] = (R)md.mulin[k].coef; }
  for (int k = tid; k < md.n_pairs; k += NT) s_pair[k] = md.pairs[k];
  for (int k = tid; k < md.n_pair_groups; k += NT) s_pcoef[k] = (R)md.pair_coef[k];
  const EpiScalars<R> es = epi_scalars<R, E>(fa);
  const R inv = E == Epi::kTpq ? opaque((R)fa.scal[0]) : (R)0;
  int same_flag = md.c_up == md.c_dn ? 1 : 0;
  asm volatile("" : "+r"(same_flag));  // one fp64 comparison per thread, not per element
  const bool same_c = same_flag != 0;
  // Fixed point.  One hopping value of magnitude 2^k (t = 1 in particular): c * fix(a) =
  // fix(+-a) 2^k, an exponent shift instead of an fp64 multiply per element; the element is
  // then computed in units of 2^e2, e2 = eoff + k: hv = (dg 2^-k xr + (+-(acc + wq))) 2^e2 with
  // xr = q as fp64, so the two per-element power-of-two scalings fold into the diagonal table,
  // the Lanczos coefficient and the per-CTA partial sum (both scales must be normal numbers).
  const int eoff = FIX ? *Ep - 1078 : 0;
  const long long cbits = __double_as_longlong(md.c_up);
  const int cexp = (int)((cbits >> 52) & 0x7ff);
  const bool c_p2 = FIX && same_c && (cbits & 0xfffffffffffffll) == 0 && cexp > 0 && cexp < 0x7ff;
  const bool c_neg = cbits < 0;
  const int c_l2 = cexp - 1023;
  const int e2 = eoff + c_l2;
  const bool fold = c_p2 && eoff >= -1022 && eoff <= 1023 && e2 >= -1022 && e2 <= 1023 &&
                    E != Epi::kTpq;
  const double s_eoff = fold ? __longlong_as_double((long long)(eoff + 1023) << 52) : 1.0;
  const double s_e2 = fold ? __longlong_as_double((long long)(e2 + 1023) << 52) : 1.0;
  const double r_k = fold ? __longlong_as_double((long long)(1023 - c_l2) << 52) : 1.0;  // 2^-k
  // diagonal = c0 + U * popcount(up & dn & mask) in the common single-group case: table
  const bool dtab = md.n_ulin == 1 && md.n_mulin == 0 && md.n_pairs == 0;
  // the diagonal an integer multiple of the hopping (md.dint): the whole element is one exact
  // int64 sum d q +- S and <x, H x> adds the exact products q (d q +- S) in 128 bits, moved to
  // fp64 every 64 elements, so an element costs three fp64 operations instead of six
  const bool dint = fold && dtab && md.dint;
  if (dtab && tid <= 32) {
    const double v = (md.c0 + md.ulin[0].coef * (double)tid) * r_k;
    s_dtab[tid] = (R)v;
    s_dti[tid] = dint ? (int)__double2ll_rn(v) : 0;
  }
  const R c_up = opaque((R)md.c_up), c_dn = opaque((R)md.c_dn);
  const int dim_up = (int)md.dim_up;
  const int64_t dim_dn = md.dim_dn;
  // the zero entries after the row that unused slots read
  for (int k = tid; k < gather_lanes(K * (int)sizeof(T)) * K; k += NT) tile[(size_t)dim_up * K + k] = (T)0;
  constexpr int NQ = n_red<E>() > 0 ? n_red<E>() : 1;
  Red<FIX, NQ> red;
  red.zero();
  __int128 ia = 0;
  int ic = 0;
  int pmx = 0;  // fp64 Lanczos: largest exponent field of the P values written (fa.pexp)
  const int64_t n_tiles = (dim_dn + K - 1) / K;
  const uint2* rec = md.up_rec[kWidth];
  const uint4* hdr = md.up_hdr[kWidth];
  const int64_t stride = md.up_stride;

  for (int64_t t = blockIdx.x; t < n_tiles; t += gridDim.x) {
    const int64_t d0 = t * K;
    const int nk = (int)((dim_dn - d0 < K) ? (dim_dn - d0) : K);
    __syncthreads();
    const T* rows = X + d0 * dim_up;
    if (K == 1 && (reinterpret_cast<uintptr_t>(rows) & 15u) == 0) {  // one row: 16-byte pieces
      constexpr int kPer = 16 / (int)sizeof(T);
      const int nv = dim_up / kPer;
      for (int u = tid; u < nv; u += NT) copy_async<16>(tile + u * kPer, rows + u * kPer);
      for (int u = nv * kPer + tid; u < dim_up; u += NT) copy_async<(int)sizeof(T)>(tile + u, rows + u);
    } else {
      for (int u = tid; u < dim_up; u += NT) {
#pragma unroll
        for (int m = 0; m < K; ++m) {
          if (m < nk) copy_async<(int)sizeof(T)>(tile + u * K + m, rows + (int64_t)m * dim_up + u);
          else tile[u * K + m] = (T)0;
        }
      }
    }
    uint32_t dn[K];
#pragma unroll
    for (int m = 0; m < K; ++m) dn[m] = (m < nk) ? (md.sector ? __ldg(md.list_dn + d0 + m) : (uint32_t)(d0 + m)) : 0u;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // Whole warps run to the padded row length: the table's padding reads zero entries.  The
    // records come from L2, so they are streamed a chunk of kGatherChunk groups ahead, across
    // states: while a chunk's targets are gathered the next chunk (of this state or the next)
    // and the next state's header are on their way.
    uint2 cur[kGatherChunk];
    uint32_t hx = 0u;
    if (tid < (int)stride) {
      hx = __ldg(&hdr[tid >> 5].x);
#pragma unroll
      for (int j = 0; j < kGatherChunk; ++j) cur[j] = __ldg(rec + tid + j * stride);
    }
    for (int u = tid; u < (int)stride; u += NT) {
      const int np = (int)(hx & 0xffffu), ns = (int)(hx >> 16);  // slots [0, np) add, [np, ns) subtract
      const int ng = (ns + 3) >> 2;
      const int un = u + NT < (int)stride ? u + NT : u;
      hx = __ldg(&hdr[un >> 5].x);
      const bool on = u < dim_up;
      T wv[K];
      R pin[K];
#pragma unroll
      for (int m = 0; m < K; ++m) {
        const int64_t idx = (d0 + m) * dim_up + u;
        wv[m] = (on && m < nk) ? W[idx] : (T)0;
        if constexpr (E == Epi::kLanczos1 && FIX)
          pin[m] = (on && m < nk) ? reinterpret_cast<const R*>(fa.in ? fa.in : fa.out)[idx] : (R)0;
      }
      const uint32_t up = md.sector ? __ldg(md.list_up + (on ? u : 0)) : (uint32_t)u;
      T acc[K];
#pragma unroll
      for (int m = 0; m < K; ++m) acc[m] = (T)0;
      int c0 = 0;
      do {
        const uint2* q = c0 + kGatherChunk < ng ? rec + u + (int64_t)(c0 + kGatherChunk) * stride : rec + un;
        uint2 nxt[kGatherChunk];
#pragma unroll
        for (int j = 0; j < kGatherChunk; ++j) nxt[j] = __ldg(q + j * stride);
        if (K == 1 && 4 * (c0 + kGatherChunk) <= np) {  // a chunk that only adds: no tests per group (*)
          T cs = (T)0;
#pragma unroll
          for (int j = 0; j < kGatherChunk; ++j) {
            const uint2 r = cur[j];
            cs += (tile[r.x & 0xffffu] + tile[r.x >> 16]) + (tile[r.y & 0xffffu] + tile[r.y >> 16]);
          }
          acc[0] += cs;
        } else {
#pragma unroll
          for (int j = 0; j < kGatherChunk; ++j) {
            if (c0 + j < ng) {
              const uint2 r = cur[j];
              T v[4][K];
              load_k<T, K>(tile + (r.x & 0xffffu) * K, v[0]);
              load_k<T, K>(tile + (r.x >> 16) * K, v[1]);
              load_k<T, K>(tile + (r.y & 0xffffu) * K, v[2]);
              load_k<T, K>(tile + (r.y >> 16) * K, v[3]);
              const int left = np - 4 * (c0 + j);  // slots of this group that add
              if (left >= 4) {
#pragma unroll
                for (int m = 0; m < K; ++m) acc[m] += (v[0][m] + v[1][m]) + (v[2][m] + v[3][m]);
              } else if (left <= 0) {
#pragma unroll
                for (int m = 0; m < K; ++m) acc[m] -= (v[0][m] + v[1][m]) + (v[2][m] + v[3][m]);
              } else {
#pragma unroll
                for (int s = 0; s < 4; ++s)
#pragma unroll
                  for (int m = 0; m < K; ++m) acc[m] += s < left ? v[s][m] : -v[s][m];
              }
            }
          }
        }
#pragma unroll
        for (int j = 0; j < kGatherChunk; ++j) cur[j] = nxt[j];
        c0 += kGatherChunk;
      } while (c0 < ng);
      if (!on) continue;
#pragma unroll
      for (int m = 0; m < K; ++m) {
        if (m >= nk) break;
        const int64_t idx = (d0 + m) * dim_up + u;
        const T xq = tile[u * K + m];
        if constexpr (FIX) {
          if (dint) {
            const long long S = acc[m] + wv[m];
            const long long hq = (long long)s_dti[__popc(up & dn[m] & (uint32_t)s_ulin[0].mask)] * xq + (c_neg ? -S : S);
            const double hvu = __ll2double_rn(hq);  // hv = hvu 2^e2
            if constexpr (E == Epi::kStore) {
              reinterpret_cast<double*>(w)[idx] = hvu * s_e2;
            } else if constexpr (E == Epi::kLanczos1) {
              const double pv = fma(es.c1 * s_e2, hvu, -(es.c2 * pin[m]));
              reinterpret_cast<double*>(fa.out)[idx] = pv;
              pmx = max(pmx, (int)((__double_as_longlong(pv) >> 52) & 0x7ff));
              ia += (__int128)xq * (__int128)hq;
              if (++ic == 64) {
                red.add(0, i128_to_double(ia), 1.0);
                ia = 0;
                ic = 0;
              }
            } else if constexpr (E == Epi::kRefine) {
              refine_folded(hvu, __ll2double_rn(xq), s_e2, idx, fa, red);
            } else if constexpr (E == Epi::kShift) {
              shift_folded(hvu, __ll2double_rn(xq), es.c1 * r_k, s_e2, idx, fa, red);
            }
            continue;
          }
        }
        // diagonal: integer counts times the class coefficients (times 2^-k when folding)
        R dg;
        if (dtab) {
          dg = s_dtab[__popc(up & dn[m] & (uint32_t)s_ulin[0].mask)];
        } else {
          dg = (R)md.c0;
          for (int g = 0; g < md.n_ulin; ++g) dg += s_uc[g] * (R)__popc(up & dn[m] & (uint32_t)s_ulin[g].mask);
          for (int g = 0; g < md.n_mulin; ++g) {
            const uint32_t mk = (uint32_t)s_mlin[g].mask;
            dg += s_mc[g] * (R)(__popc(up & mk) + __popc(dn[m] & mk));
          }
          if (md.n_pairs) {
            int grp = s_pair[0].grp, cnt = 0;
            for (int p = 0; p < md.n_pairs; ++p) {
              const PairEntry pe = s_pair[p];
              if (pe.grp != grp) {
                dg += s_pcoef[grp] * (R)cnt;
                cnt = 0;
                grp = pe.grp;
              }
              const int ni = (int)((up >> pe.i) & 1u) + (int)((dn[m] >> pe.i) & 1u);
              const int nj = (int)((up >> pe.j) & 1u) + (int)((dn[m] >> pe.j) & 1u);
              cnt += ni * nj;
            }
            dg += s_pcoef[grp] * (R)cnt;
          }
          if (fold) dg *= (R)r_k;
        }
        if constexpr (!FIX) {
          const R hv = same_c ? dg * xq + c_up * (acc[m] + wv[m]) : dg * xq + c_up * acc[m] + c_dn * wv[m];
          epilogue<R, E, NQ>(idx, xq, (R)0, hv, (R)0, reinterpret_cast<R*>(w), fa, es, inv, red);
        } else if (fold) {
          const double xr = __ll2double_rn(xq);
          const long long S = acc[m] + wv[m];
          const double hvu = fma(dg, xr, __ll2double_rn(c_neg ? -S : S));  // hv = hvu 2^e2
          if constexpr (E == Epi::kStore) {
            reinterpret_cast<double*>(w)[idx] = hvu * s_e2;
          } else if constexpr (E == Epi::kLanczos1) {
            // P <- c1 hv - c2 P; partial <x, hv> in units of 2^(eoff + e2)
            const double pv = fma(es.c1 * s_e2, hvu, -(es.c2 * pin[m]));
            reinterpret_cast<double*>(fa.out)[idx] = pv;
            pmx = max(pmx, (int)((__double_as_longlong(pv) >> 52) & 0x7ff));
            red.add(0, xr, hvu);
            red.tick();
          } else if constexpr (E == Epi::kRefine) {
            refine_folded(hvu, xr, s_e2, idx, fa, red);
          } else if constexpr (E == Epi::kShift) {
            shift_folded(hvu, xr, es.c1 * r_k, s_e2, idx, fa, red);
          }
        } else {
          const double x = fix_to_double(xq, eoff);
          double hv;
          if (c_p2) hv = fma(dg, x, fix_to_double(c_neg ? -(acc[m] + wv[m]) : acc[m] + wv[m], eoff + c_l2));
          else if (same_c) hv = fma(dg, x, md.c_up * fix_to_double(acc[m] + wv[m], eoff));
          else hv = fma(dg, x, fma(md.c_up, fix_to_double(acc[m], eoff), md.c_dn * fix_to_double(wv[m], eoff)));
          if constexpr (E == Epi::kLanczos1) {  // the epilogue's Lanczos step, with the exponent kept
            const double pv = es.c1 * hv - es.c2 * pin[m];
            reinterpret_cast<double*>(fa.out)[idx] = pv;
            pmx = max(pmx, (int)((__double_as_longlong(pv) >> 52) & 0x7ff));
            red.add(0, x, hv);
            red.tick();
          } else {
            epilogue<double, E, NQ>(idx, x, 0.0, hv, 0.0, reinterpret_cast<double*>(w), fa, es, inv, red);
          }
        }
      }
    }
  }
  if constexpr (FIX && E == Epi::kLanczos1) {
    if (ic) red.add(0, i128_to_double(ia), 1.0);
    if (fa.pexp != nullptr) {
      pmx = (int)__reduce_max_sync(0xffffffffu, (unsigned)pmx);
      if ((tid & 31) == 0 && pmx > 0) atomicMax(fa.pexp, pmx);
    }
  }
  if constexpr (E != Epi::kStore) {
    // fixed-order reduction: warp shuffles, then the warps' sums in warp order
    constexpr int nq = n_red<E>();
    const int lane = tid & 31, wid = tid >> 5;
#pragma unroll
    for (int q = 0; q < nq; ++q) {
      double x = red.get(q);
      if (fold) x = folded_sum(x, q, s_eoff, s_e2);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
      if (lane == 0) s_red[wid * kMaxRedQ + q] = x;
    }
    __syncthreads();
    if (tid < nq) {
      double x = 0.0;
      for (int k = 0; k < NT / 32; ++k) x += s_red[k * kMaxRedQ + tid];
      fa.partials[(size_t)blockIdx.x * kMaxRedQ + tid] = x;
    }
  }
}

template <class R>
int pick_k(const HubDev& md) {
  const int64_t row = md.dim_up * (int64_t)sizeof(R);
  int k = 1;
  if (4 * row <= kSmemBudget) k = 4;
  else if (2 * row <= kSmemBudget) k = 2;
  if (md.up_k > 0 && md.up_k < k) k = (md.up_k >= 2) ? 2 : 1;
  return k;
}

int pick_kq(const HubDev& md) {
  int k = (2 * md.dim_up * 8 <= kSmemBudget) ? 2 : 1;
  if (md.up_k == 1) k = 1;
  return k;
}

// pass D launch with the tuned (or default) pieces per lane
template <class R>
Status launch_dn(const HubDev& md, const R* X, R* W, const int* done, unsigned long long* counter, cudaStream_t st) {
  auto items_of = [&](int pieces) -> int64_t {
    const int64_t sw = (int64_t)32 * pieces * 16 / (int64_t)sizeof(R);
    return ((md.dim_up + sw - 1) / sw) * md.dim_dn;
  };
  const int64_t warps = (int64_t)num_sms() * 32;
  int p = md.dn_ept;
  if (p != 1 && p != 2 && p != 4) p = items_of(kDnPieces) >= 2 * warps ? kDnPieces : 1;
  const int64_t items = items_of(p);
  const int gd = (int)std::min<int64_t>((items + 7) / 8, (int64_t)num_sms() * 8);
  // items per warp and claim: four, fewer while that would leave warps without one; 0: a warp for
  // every item, no counter
  const int claim = items <= (int64_t)gd * 8 ? 0 : (int)std::max<int64_t>(1, std::min<int64_t>(4, items / (2 * warps)));
  const bool vec = (md.dim_up * (int64_t)sizeof(R)) % 16 == 0 && ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(W)) & 15u) == 0;
  if (claim > 0) HPHI_CUDA_TRY(cudaMemsetAsync(counter, 0, sizeof(unsigned long long), st));
#define HPHI_DN(PP)                                                                    \
  if (vec) k_hub_dn<R, PP, true><<<gd, kThreads, 0, st>>>(md, X, W, done, counter, claim);    \
  else k_hub_dn<R, PP, false><<<gd, kThreads, 0, st>>>(md, X, W, done, counter, claim)
  if (p == 4) {
    HPHI_DN(4);
  } else if (p == 1) {
    HPHI_DN(1);
  } else {
    HPHI_DN(2);
  }
#undef HPHI_DN
  HPHI_CUDA_TRY(cudaGetLastError());
  return {};
}

// pass U threads: 1024 (one CTA per SM) for tiles above ~110 KB, else 512 so two CTAs per
// SM alternate between loading a tile and working on one
inline int up_threads(size_t tile_bytes) { return tile_bytes > 110000 ? 1024 : 512; }

template <class KernelT>
int occupancy_for(KernelT kern, int nt, size_t smem) {
  int n = 0;
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget + kZeroBytes);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, nt, smem) != cudaSuccess || n < 1) {
    cudaGetLastError();
    n = 1;
  }
  return n;
}

template <class T, int K>
size_t up_smem(const HubDev& md) {
  return (size_t)K * sizeof(T) * (size_t)(md.dim_up + gather_lanes(K * (int)sizeof(T)));
}

template <class T, int K, Epi E>
int up_occupancy(const HubDev& md) {
  const size_t smem = up_smem<T, K>(md);
  return up_threads(smem) == 1024 ? occupancy_for(k_hub_up<T, K, E, 1024>, 1024, smem)
                                  : occupancy_for(k_hub_up<T, K, E, 512>, 512, smem);
}

template <class T, int K, Epi E>
Status launch_up(const HubDev& md, const T* X, const T* W, const int* Ep, void* w, const FusedArgs& fa, int grid,
                 cudaStream_t st) {
  const size_t smem = up_smem<T, K>(md);
  const int most = kSmemBudget + kZeroBytes;
  if (up_threads(smem) == 1024) {
    HPHI_CUDA_TRY(cudaFuncSetAttribute(k_hub_up<T, K, E, 1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    k_hub_up<T, K, E, 1024><<<grid, 1024, smem, st>>>(md, X, W, Ep, w, fa);
  } else {
    HPHI_CUDA_TRY(cudaFuncSetAttribute(k_hub_up<T, K, E, 512>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    k_hub_up<T, K, E, 512><<<grid, 512, smem, st>>>(md, X, W, Ep, w, fa);
  }
  HPHI_CUDA_TRY(cudaGetLastError());
  return {};
}

// scratch layout of the quantised fp64 path: [Q: dim int64][WQ: dim int64][E: int]
size_t quant_scratch_bytes(const HubDev& md) { return (size_t)16 * md.dim + 256; }

template <Epi E>
Status launch_q(const HubDev& md, const void* v, void* w, void* scratch, const FusedArgs& fa, int grid_up,
                cudaStream_t st) {
  const double* X = reinterpret_cast<const double*>(v);
  long long* Q = reinterpret_cast<long long*>(scratch);
  long long* WQ = Q + md.dim;
  int* Ep = reinterpret_cast<int*>(WQ + md.dim);
  unsigned long long* counter = reinterpret_cast<unsigned long long*>(WQ + md.dim) + 1;
  if (fa.exp_ready != 2) {  // 2: the previous Lanczos pass 2 wrote Q and its exponent
    const Status s = launch_quant_vec(X, Q, md.dim, Ep, fa.done, fa.exp_ready != 0, 0, st);
    if (s.code) return s;
  }
  if (fa.pexp != nullptr) HPHI_CUDA_TRY(cudaMemsetAsync(fa.pexp, 0, sizeof(int), st));
  Status sd = launch_dn<long long>(md, Q, WQ, fa.done, counter, st);
  if (sd.code) return sd;
  return pick_kq(md) == 2 ? launch_up<long long, 2, E>(md, Q, WQ, Ep, w, fa, grid_up, st)
                          : launch_up<long long, 1, E>(md, Q, WQ, Ep, w, fa, grid_up, st);
}

int* hub_exponent_slot_impl(const HubDev& md, void* scratch) {
  return reinterpret_cast<int*>(reinterpret_cast<long long*>(scratch) + 2 * md.dim);
}

int upq_grid(const HubDev& md, Epi epi) {
  const int K = pick_kq(md);
  int occ = 1;
#define HPHI_OCCQ(KK)                                                          \
  switch (epi) {                                                               \
    case Epi::kStore: occ = up_occupancy<long long, KK, Epi::kStore>(md); break;         \
    case Epi::kLanczos1: occ = up_occupancy<long long, KK, Epi::kLanczos1>(md); break;   \
    case Epi::kTpq: occ = up_occupancy<long long, KK, Epi::kTpq>(md); break;             \
    case Epi::kRefine: occ = up_occupancy<long long, KK, Epi::kRefine>(md); break;       \
    case Epi::kShift: occ = up_occupancy<long long, KK, Epi::kShift>(md); break;         \
  }
  if (K == 2) { HPHI_OCCQ(2) } else { HPHI_OCCQ(1) }
#undef HPHI_OCCQ
  const int64_t tiles = (md.dim_dn + K - 1) / K;
  return (int)std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)num_sms() * occ));
}

template <class R, Epi E>
Status launch_r(const HubDev& md, const void* v, void* w, void* scratch, const FusedArgs& fa, int grid_up,
                cudaStream_t st) {
  const R* X = reinterpret_cast<const R*>(v);
  // kStore writes the down-spin sums into w and finishes them in place; the fused steps
  // use the scratch vector
  R* W = (E == Epi::kStore) ? reinterpret_cast<R*>(w) : reinterpret_cast<R*>(scratch);
  // the item counter of pass D sits after the fp32 scratch vector (first bytes of scratch
  // when the scratch holds no vector)
  const size_t voff = (E == Epi::kStore) ? 0 : (((size_t)md.dim * sizeof(R) + 255) / 256) * 256;
  unsigned long long* counter = reinterpret_cast<unsigned long long*>(static_cast<char*>(scratch) + voff);
  Status sd = launch_dn<R>(md, X, W, fa.done, counter, st);
  if (sd.code) return sd;
  switch (pick_k<R>(md)) {
    case 4: return launch_up<R, 4, E>(md, X, W, nullptr, w, fa, grid_up, st);
    case 2: return launch_up<R, 2, E>(md, X, W, nullptr, w, fa, grid_up, st);
    default: return launch_up<R, 1, E>(md, X, W, nullptr, w, fa, grid_up, st);
  }
}

template <class R>
int up_grid_r(const HubDev& md, Epi epi) {
  int occ = 1;
  const int k = pick_k<R>(md);
#define HPHI_OCC(KK)                                                         \
  switch (epi) {                                                             \
    case Epi::kStore: occ = up_occupancy<R, KK, Epi::kStore>(md); break;       \
    case Epi::kLanczos1: occ = up_occupancy<R, KK, Epi::kLanczos1>(md); break; \
    case Epi::kTpq: occ = up_occupancy<R, KK, Epi::kTpq>(md); break;           \
    case Epi::kRefine: occ = up_occupancy<R, KK, Epi::kRefine>(md); break;     \
    case Epi::kShift: break;                                                   \
  }
  if (k == 4) { HPHI_OCC(4) } else if (k == 2) { HPHI_OCC(2) } else { HPHI_OCC(1) }
#undef HPHI_OCC
  const int64_t tiles = (md.dim_dn + k - 1) / k;
  return (int)std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)num_sms() * occ));
}

// Device address of g_noalloc_scratch on the current device.  Looked up again on every call
// whose stream is not being captured (the lookup allocates nothing), so a device reset or
// another current context cannot leave a stale address behind; a capturing stream takes the
// address cached by the last such lookup on the device (a graph replays that address anyway).
std::mutex g_noalloc_mu;
void* g_noalloc_ptr[64] = {};

Status noalloc_scratch(void** out, cudaStream_t st) {
  int dev = 0;
  HPHI_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return {HPHI_ERR_UNSUPPORTED, "allocation-free path: device ordinal above 63"};
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  HPHI_CUDA_TRY(cudaStreamIsCapturing(st, &cs));
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (cs == cudaStreamCaptureStatusNone || g_noalloc_ptr[dev] == nullptr) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || p == nullptr) {
      cudaGetLastError();
      return {HPHI_ERR_CUDA, std::string("cudaGetSymbolAddress(allocation-free scratch): ") + cudaGetErrorString(e)};
    }
    g_noalloc_ptr[dev] = p;
  }
  *out = g_noalloc_ptr[dev];
  return {};
}

}  // namespace

HubDev with_shape(const HubDev& md, int prec);

Status launch_hub_store_noalloc(const HubDev& md0, const void* v, void* w, cudaStream_t st) {
  const HubDev md = with_shape(md0, HPHI_FP64);
  const size_t need = quant_scratch_bytes(md);
  if (need > kNoAllocScratchBytes)
    return {HPHI_ERR_INVALID_ARG, "hphi_apply_H_noalloc: the basis needs " + std::to_string(need) +
                                      " bytes of scratch, above the fixed " + std::to_string(kNoAllocScratchBytes) +
                                      " (at most " + std::to_string((kNoAllocScratchBytes - 256) / 16) + " rows)"};
  void* scratch = nullptr;
  Status s = noalloc_scratch(&scratch, st);
  if (s.code) return s;
  FusedArgs fa;  // plain H v: no reductions, no breakdown flag
  return launch_q<Epi::kStore>(md, v, w, scratch, fa, upq_grid(md, Epi::kStore), st);
}

int quant_kernels(int64_t n, int exp_ready) {
  return exp_ready == 2 ? 0 : (exp_ready != 0 || n <= kShortQuant ? 1 : 2);
}

Status launch_quant_vec(const double* X, long long* Q, int64_t n, int* Ep, const int* done, bool exp_ready, int extra,
                        cudaStream_t st) {
  if (!exp_ready && n <= kShortQuant) {
    k_quant_short<<<1, 1024, 0, st>>>(X, Q, (int)n, Ep, done, extra);
    HPHI_CUDA_TRY(cudaGetLastError());
    return {};
  }
  const int gv = (int)std::max<int64_t>(1, std::min<int64_t>((n + kThreads - 1) / kThreads, (int64_t)num_sms() * 8));
  if (!exp_ready) {
    HPHI_CUDA_TRY(cudaMemsetAsync(Ep, 0, sizeof(int), st));
    k_maxexp<<<gv, kThreads, 0, st>>>(X, n, Ep, done);
    HPHI_CUDA_TRY(cudaGetLastError());
  }
  k_quant<<<gv, kThreads, 0, st>>>(X, Q, n, Ep, done, extra);
  HPHI_CUDA_TRY(cudaGetLastError());
  return {};
}

Status build_hub_neighbours(const HubDev& md, int species, uint32_t* nbr, uint8_t* deg, uint8_t* npos,
                            cudaStream_t st) {
  const int64_t n = species ? md.dim_dn : md.dim_up;
  const int g = (int)std::max<int64_t>(1, std::min<int64_t>((n + kThreads - 1) / kThreads, (int64_t)num_sms() * 8));
  k_hub_nbr<<<g, kThreads, 0, st>>>(md, species, nbr, deg, npos);
  HPHI_CUDA_TRY(cudaGetLastError());
  return {};
}

bool hub_up_row_fits(const HubDev& md, int prec) {
  return md.dim_up * (int64_t)(prec == HPHI_FP64 ? 8 : 4) <= kSmemBudget;
}

bool hub_fast_ok(const HubDev& md, int prec, bool cplx, int nvec, Epi epi) {
  if (!md.fast || cplx || nvec != 1) return false;
  // fixed-point sums of at most 127 terms (|q| < 2^56) stay exact in 64 bits
  if (prec == HPHI_FP64 && md.maxdeg_up + md.maxdeg_dn > 126) return false;
  if ((epi == Epi::kRefine || epi == Epi::kShift) && prec != HPHI_FP64) return false;
  return hub_up_row_fits(md, prec);
}

// the launch shape of one precision: the autotuner's choice, else the built-in default
HubDev with_shape(const HubDev& md, int prec) {
  HubDev t = md;
  const int i = prec == HPHI_FP64 ? 0 : 1;
  t.dn_ept = md.tuned_ept[i];
  t.up_k = md.tuned_k[i];
  return t;
}

int hub_up_width(const HubDev& md0, int prec) {
  const HubDev md = with_shape(md0, prec);
  const int b = prec == HPHI_FP64 ? 8 * pick_kq(md) : 4 * pick_k<float>(md);
  return b >= 16 ? 2 : (b >= 8 ? 1 : 0);
}

int hub_up_grid(const HubDev& md0, int prec, Epi epi) {
  const HubDev md = with_shape(md0, prec);
  return prec == HPHI_FP64 ? upq_grid(md, epi) : up_grid_r<float>(md, epi);
}

int* hub_exponent_slot(const HubDev& md, void* scratch) { return hub_exponent_slot_impl(md, scratch); }

// Q at the start of the scratch; tail (after WQ) ints: exponent of Q at 0, work counter
// (u64) at 8, the exact exponents of the current / next vector at 16 and 20, pass-1's at 24
QSlots hub_qslots(const HubDev& md, void* scratch) {
  QSlots q;
  if (scratch == nullptr) return q;
  int* tail = hub_exponent_slot_impl(md, scratch);
  q.Q = reinterpret_cast<long long*>(scratch);
  q.eq = tail;
  q.ec[0] = tail + 4;
  q.ec[1] = tail + 5;
  q.ep = tail + 6;
  q.extra = 0;
  return q;
}

size_t hub_scratch_bytes(const HubDev& md, int prec, Epi epi) {
  if (prec == HPHI_FP64) return quant_scratch_bytes(md);
  return (epi == Epi::kStore ? 0 : (((size_t)4 * md.dim + 255) / 256) * 256) + 256;
}

Status launch_hub_fast(const HubDev& md0, int prec, const void* v, void* w, void* scratch, Epi epi,
                       const FusedArgs& fa, int grid_up, cudaStream_t st) {
  const HubDev md = with_shape(md0, prec);
  if (prec == HPHI_FP64) {
    switch (epi) {
      case Epi::kStore: return launch_q<Epi::kStore>(md, v, w, scratch, fa, grid_up, st);
      case Epi::kLanczos1: return launch_q<Epi::kLanczos1>(md, v, w, scratch, fa, grid_up, st);
      case Epi::kTpq: return launch_q<Epi::kTpq>(md, v, w, scratch, fa, grid_up, st);
      case Epi::kRefine: return launch_q<Epi::kRefine>(md, v, w, scratch, fa, grid_up, st);
      case Epi::kShift: return launch_q<Epi::kShift>(md, v, w, scratch, fa, grid_up, st);
    }
  } else {
    switch (epi) {
      case Epi::kStore: return launch_r<float, Epi::kStore>(md, v, w, scratch, fa, grid_up, st);
      case Epi::kLanczos1: return launch_r<float, Epi::kLanczos1>(md, v, w, scratch, fa, grid_up, st);
      case Epi::kTpq: return launch_r<float, Epi::kTpq>(md, v, w, scratch, fa, grid_up, st);
      case Epi::kRefine:
      case Epi::kShift: break;
    }
  }
  return {HPHI_ERR_INVALID_ARG, "two-pass Hubbard path: unsupported precision / epilogue"};
}

}  // namespace hphi

// Split-row H v for real spin models in a fixed-S^z sector (section 3.3's on-the-fly
// product over section 3.1's restricted basis), laid out for GB300's memory hierarchy.
//
// A sector configuration is s = (hi << L) | lo.  Ascending order sorts by hi first, so the
// rows of one high part are contiguous: row hi starts at hi_off[hi] and holds the C(L, q)
// low parts of popcount q = n_ones - popcount(hi) in ascending order.  In an S^z sector the
// only off-diagonal terms are exchange flips of two antiparallel spins, so
//   low-low bonds    act inside a row:        (hi, lo)  <- (hi, lo ^ m)
//   high-high bonds  combine whole rows:      row hi    <- row hi ^ m, same column
//   straddling bonds gather from one row:     (hi, lo)  <- (hi ^ 2^a, lo ^ 2^b)
// (section 4.3's point, terms acting on data that is already local, with the row as the
// local unit).  Two passes, each with its own split:
//   pass H  (k_sec_hi)  the row combinations of every bond above its split hL, stripe-major per
//           popcount class so one column stripe of every row of the class is the L2 working
//           set; the plain sums go to W (a scratch vector for Lanczos, else the output itself).
//   pass R  (k_sec_lo)  stages K rows of one class in shared memory, applies the bonds inside
//           the row that pass H left (those with a site below hL) from a gather table, gathers
//           the straddling ones from the partner rows (for one bond the column map
//           lo -> rank(lo ^ 2^b) is increasing, so a warp's gathers stay close together), adds
//           the diagonal from integer bond counts and a small table, adds W and runs the fused
//           Lanczos / mTPQ / refine epilogue.
// Pass H costs a third of pass R per active bond (coalesced, no tables), so hL is as small as
// rows of a few hundred entries allow: it takes the bonds of the sites hL .. L - 1 among
// themselves, which would be gathers of pass R, and those of these sites with the high part,
// which would straddle.
// fp64 vectors run on the 64-bit fixed-point copy (integer sums, one conversion per
// element); fp32 vectors sum in fp32.
#include <math.h>

#include <algorithm>
#include <map>
#include <memory>
#include <string>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "epilogue.cuh"
#include "gather.cuh"
#include "reduce.cuh"

namespace hphi {

// ====================================================================== host: analysis
namespace {

struct Bond {
  int i, j;    // i < j
  double c;    // element <s ^ m| H |s> for antiparallel bits i, j
};

struct Analysis {
  bool ok = false;
  std::string why;
  std::vector<Bond> bonds;
  std::vector<double> cls;        // distinct exchange coefficients
  std::vector<int> bond_cls;
  double unit = 0.0;              // fp64: cls[c] = mult[c] * unit
  std::vector<int> mult;
  bool int_ok = false;            // integer multiples found
  int qextra = 0;
  // the diagonal in units of `unit` is an integer everywhere (fp64 pass R then forms the whole
  // element as one exact int64 sum); maxdgi bounds its magnitude
  bool dint = false;
  double maxdgi = 0.0;
  // diagonal = c0 + sum_g gcoef[g] * count_g, count_g over pair bonds (both up) and sites (up)
  double c0 = 0.0;
  int n_dg = 0;
  double gcoef[2] = {0.0, 0.0};
  std::vector<std::pair<int, int>> gpairs[2];  // pair groups
  uint64_t gsites[2] = {0, 0};                 // site groups (linear terms)
  int gmax[2] = {0, 0};
};

uint64_t binom_u(int n, int k) {
  if (k < 0 || k > n || n < 0) return 0;
  if (k > n - k) k = n - k;
  unsigned __int128 r = 1;
  for (int i = 1; i <= k; ++i) r = r * (unsigned)(n - k + i) / (unsigned)i;
  return (uint64_t)r;
}

Analysis analyse(const SecTerms& t) {
  Analysis a;
  const int N = t.n_sites;
  if (N < 2 || N > kSecMaxL + kSecMaxH) {
    a.why = "split-row path: 2..42 sites";
    return a;
  }
  // exchange bonds: each entry flips two sites with a real element, the same both ways
  std::map<std::pair<int, int>, double> bond;
  for (const SpinEntry& e : t.ents) {
    if (e.i == e.j || __builtin_popcountll(e.mask) != 2) {
      a.why = "split-row path: only two-site exchange terms";
      return a;
    }
    const double2 c = t.cls[e.cls];
    if (c.y != 0.0) {
      a.why = "split-row path: real couplings only";
      return a;
    }
    const int code0 = e.phases & 7, code1 = (e.phases >> 3) & 7, code2 = (e.phases >> 6) & 7,
              code3 = (e.phases >> 9) & 7;
    auto val = [&](int code) -> double {
      return code == 1 ? c.x : (code == 3 ? -c.x : 0.0);
    };
    if (code0 || code3 || (code1 != 0 && code1 != 1 && code1 != 3) || (code2 != 0 && code2 != 1 && code2 != 3)) {
      a.why = "split-row path: exchange of antiparallel spins with real elements only";
      return a;
    }
    if (val(code1) != val(code2)) {
      a.why = "split-row path: non-symmetric exchange element";
      return a;
    }
    const int i = std::min<int>(e.i, e.j), j = std::max<int>(e.i, e.j);
    bond[std::make_pair(i, j)] += val(code1);
  }
  for (auto& kv : bond) {
    if (kv.second == 0.0) continue;
    a.bonds.push_back(Bond{kv.first.first, kv.first.second, kv.second});
  }
  for (const Bond& b : a.bonds) {
    int c = -1;
    for (size_t k = 0; k < a.cls.size(); ++k)
      if (a.cls[k] == b.c) c = (int)k;
    if (c < 0) {
      a.cls.push_back(b.c);
      c = (int)a.cls.size() - 1;
    }
    a.bond_cls.push_back(c);
  }
  if ((int)a.cls.size() > kSecMaxCls) {
    a.why = "split-row path: too many distinct exchange couplings";
    return a;
  }
  // fp64: integer multiples of one power of two (a single class is its own unit)
  if (a.cls.size() <= 1) {
    a.unit = a.cls.empty() ? 1.0 : a.cls[0];
    a.mult.assign(a.cls.size(), 1);
    a.int_ok = true;
  } else {
    int g = 1 << 20;
    for (double c : a.cls) {
      int e;
      const double f = frexp(fabs(c), &e);  // c = f 2^e, f in [0.5, 1)
      uint64_t M = (uint64_t)ldexp(f, 53);
      int z = 0;
      while (M && !(M & 1)) { M >>= 1; ++z; }
      g = std::min(g, e - 53 + z);
    }
    a.unit = ldexp(1.0, g);
    a.int_ok = true;
    for (double c : a.cls) {
      const double m = ldexp(c, -g);
      if (fabs(m) > 65536.0 || m != floor(m)) a.int_ok = false;
      a.mult.push_back((int)m);
    }
  }
  long long msum = 0;
  for (size_t k = 0; k < a.bonds.size(); ++k) msum += a.int_ok ? std::abs(a.mult[a.bond_cls[k]]) : 1;
  // integer sums of msum terms of magnitude < 2^(56 - qextra) must stay below 2^63
  while (a.qextra < 40 && (double)msum * ldexp(1.0, 56 - a.qextra) >= ldexp(1.0, 63)) ++a.qextra;
  // diagonal: c0 + linear site groups + pair groups; a linear coefficient common to every site
  // is constant in the sector (it multiplies n_ones)
  a.c0 = t.c0;
  std::vector<double> lin(N, 0.0);
  for (const LinGroup& g : t.lin)
    for (int i = 0; i < N; ++i)
      if ((g.mask >> i) & 1ull) lin[i] += g.coef;
  // the most frequent per-site coefficient l0 is part of the constant (sum_i l0 b_i = l0 n_ones);
  // sites with another coefficient form count groups of lin[i] - l0
  double l0 = lin[0];
  int best = 0;
  for (int i = 0; i < N; ++i) {
    const int c = (int)std::count(lin.begin(), lin.end(), lin[i]);
    if (c > best) {
      best = c;
      l0 = lin[i];
    }
  }
  a.c0 += l0 * t.n_ones;
  int ng = 0;
  std::vector<double> vals;
  for (int i = 0; i < N; ++i)
    if (lin[i] != l0 && std::find(vals.begin(), vals.end(), lin[i]) == vals.end()) vals.push_back(lin[i]);
  for (double v : vals) {
    if (ng >= 2) {
      a.why = "split-row path: the diagonal has more than two coefficient groups";
      return a;
    }
    a.gcoef[ng] = v - l0;
    for (int i = 0; i < N; ++i)
      if (lin[i] == v) a.gsites[ng] |= 1ull << i;
    ++ng;
  }
  for (size_t k = 0; k < t.pcoef.size(); ++k) {
    if (t.pcoef[k] == 0.0) continue;
    if (ng >= 2) {
      a.why = "split-row path: the diagonal has more than two coefficient groups";
      return a;
    }
    a.gcoef[ng] = t.pcoef[k];
    for (const PairEntry& p : t.pairs)
      if (p.grp == (uint16_t)k) a.gpairs[ng].push_back(std::make_pair((int)p.i, (int)p.j));
    ++ng;
  }
  a.n_dg = ng;
  for (int g = 0; g < ng; ++g) {
    a.gmax[g] = (int)a.gpairs[g].size() + __builtin_popcountll(a.gsites[g]);
    if (a.gmax[g] > 255) {
      a.why = "split-row path: more than 255 diagonal terms in one group";
      return a;
    }
  }
  if ((a.gmax[0] + 1) * (a.gmax[1] + 1) > kSecDtab) {
    a.why = "split-row path: diagonal table too large";
    return a;
  }
  if (a.int_ok && a.unit != 0.0) {
    bool all_int = true;
    double mx = 0.0;
    for (int x = 0; x <= a.gmax[0] && all_int; ++x)
      for (int y = 0; y <= a.gmax[1]; ++y) {
        const double v = (a.c0 + a.gcoef[0] * x + a.gcoef[1] * y) / a.unit;
        if (v != floor(v) || fabs(v) > 1048576.0) {
          all_int = false;
          break;
        }
        mx = std::max(mx, fabs(v));
      }
    if (all_int) {
      a.dint = true;
      a.maxdgi = mx;
      // the element d q + S sums msum + maxdgi terms of magnitude < 2^(56 - qextra)
      while (a.qextra < 40 && ((double)msum + mx) * ldexp(1.0, 56 - a.qextra) >= ldexp(1.0, 63)) ++a.qextra;
    }
  }
  a.ok = true;
  return a;
}

constexpr int kTileBudget = 200000;  // shared-memory bytes of one row tile (without its zero entries)
constexpr int kSecHighL = 12;        // pass H split where the number of high bits allows it

// longest row of a class present in the sector for low-part length L
uint64_t longest_row(int N, int n_ones, int L) {
  const int H = N - L;
  uint64_t mx = 0;
  for (int p = 0; p <= H; ++p) {
    const int q = n_ones - p;
    if (q < 0 || q > L) continue;
    mx = std::max(mx, binom_u(L, q));
  }
  return mx;
}

bool split_ok(int N, int L) { return L >= 1 && L <= kSecMaxL && N - L >= 1 && N - L <= kSecMaxH; }

}  // namespace

bool sec_applicable(const SecTerms& t, int prec, std::string* why) {
  Analysis a = analyse(t);
  if (!a.ok) {
    if (why) *why = a.why;
    return false;
  }
  if (prec == HPHI_FP64 && !a.int_ok) {
    if (why) *why = "split-row path (fp64): couplings are not small integer multiples of one power of two";
    return false;
  }
  if (sec_default_L(t, prec == HPHI_FP64 ? 8 : 4) == 0) {
    if (why) *why = "split-row path: no split whose rows fit shared memory";
    return false;
  }
  if (why) why->clear();
  return true;
}

namespace {

// largest low part whose longest row fits one tile of one row (0: none)
int largest_L(const SecTerms& t, int esz) {
  const int N = t.n_sites;
  for (int L = std::min(kSecMaxL, N - 1); L >= 1; --L) {
    if (!split_ok(N, L)) continue;
    const uint64_t r = longest_row(N, t.n_ones, L);
    if (r <= 65535 && r * (uint64_t)esz <= (uint64_t)kTileBudget) return L;
  }
  return 0;
}

// why split L cannot be built (empty: it can): the limits on bonds and pairs across it
std::string straddle_limits(const Analysis& a, int L) {
  int n_str = 0, n_sp = 0;
  uint64_t sites = 0;
  for (const Bond& b : a.bonds)
    if (b.i < L && b.j >= L) {
      ++n_str;
      sites |= 1ull << b.i;
    }
  if (n_str > kSecMaxStr) return "split-row path: too many straddling bonds";
  if (__builtin_popcountll(sites) > kSecMaxStrSites) return "split-row path: too many straddling sites";
  std::vector<std::pair<int, uint64_t>> layers;  // diagonal group, low sites used
  for (int g = 0; g < a.n_dg; ++g)
    for (const auto& pr : a.gpairs[g]) {
      if (!(pr.first < L && pr.second >= L)) continue;
      if (++n_sp > kSecMaxSp) return "split-row path: too many straddling S^z S^z pairs";
      const uint64_t bit = 1ull << pr.first;
      size_t l = 0;
      while (l < layers.size() && (layers[l].first != g || (layers[l].second & bit))) ++l;
      if (l == layers.size()) layers.emplace_back(g, 0);
      layers[l].second |= bit;
    }
  return layers.size() > (size_t)kSecMaxSl ? "split-row path: too many straddling pair layers" : "";
}

// Pass H's split.  Rows of C(12, 6) = 924 entries fill 128-column stripes to nine tenths; fp64
// Lanczos group (pass H + pass R) on GB300 at hL = 9 / 10 / 11 / 12 / 13, 6x5 torus, S^z = 0:
// 4.69 / 4.18 / 3.98 / 3.98 / 3.95 ms, and at 9 / 10 / 11 / 12, 28-site J1-J2 ring, 9 up:
// 0.50 / 0.40 / 0.36 / 0.33 ms (at 9 bits a row's part-filled stripes cost more than the bonds it
// takes over; 13 is within 1 % of 12).  Both sizes' stripes fit L2 (50 MB on 6x5).  On 36 sites the
// largest class's stripe is C(24, 12) KB = 2.8 GB and partner reads go to DRAM; a longer split for
// that size is not measured.
int high_L(int N, int L) { return std::min(L, std::max(kSecHighL, N - kSecMaxHH)); }

}  // namespace

// The low part used when nothing else is asked: rows of C(14, 7) = 3,432 entries in fp64, two a
// tile (55 KB), and C(15, 7) = 6,435 in fp32, four a tile (103 KB), so two CTAs share an SM;
// below 24 sites N - 10 bits (at least 12) keep enough tiles for every SM.  fp64 Lanczos group
// at (L, K) on GB300: 6x5 torus (13, 2) 4.68, (14, 2) 3.98, (15, 2) 4.06, (16, 1) 4.29,
// (17, 1) 4.43 ms; 28-site J1-J2 ring, S^z = 0 (13, 2) 1.31, (14, 2) 1.19, (15, 2) 1.24,
// (17, 1) 1.49 ms; 6x4 torus (12, 2) 0.108, (13, 2) 0.101, (14, 2) 0.099 ms.  A split that the
// limits above rule out gives way to the next larger.
int sec_default_L(const SecTerms& t, int esz) {
  const int most = largest_L(t, esz);
  if (most == 0) return 0;
  const Analysis a = analyse(t);
  if (!a.ok || !straddle_limits(a, most).empty()) return most;
  for (int L = std::min(most, std::min(esz >= 8 ? 14 : 15, std::max(12, t.n_sites - 10))); L < most; ++L)
    if (split_ok(t.n_sites, L) && straddle_limits(a, L).empty()) return L;
  return most;
}

bool sec_fits(const SecTerms& t, int L, int K, int esz) {
  if (!split_ok(t.n_sites, L) || K < 1) return false;
  const uint64_t r = longest_row(t.n_sites, t.n_ones, L);
  return r >= 1 && r <= 65535 && r * (uint64_t)esz * (uint64_t)K <= (uint64_t)kTileBudget;
}

// tallest tile that fits, up to kmax rows
static int tallest(const SecTerms& t, int L, int esz, int kmax) {
  const uint64_t r = std::max<uint64_t>(1, longest_row(t.n_sites, t.n_ones, L));
  int K = 1;
  while (K < kmax && r * esz * (uint64_t)(2 * K) <= (uint64_t)kTileBudget) K *= 2;
  return K;
}

// rows per tile: 16-byte tile entries (two int64 or four fp32 rows) take one shared-memory load
// a neighbour; taller tiles are left to the autotuner (8-byte elements stop at 4 rows: 8 int64
// rows run out of registers)
int sec_default_K(const SecTerms& t, int L, int esz) { return tallest(t, L, esz, 16 / esz); }

// ====================================================================== device tables
struct SecHigh {
  uint32_t* cls = nullptr;  // SecDev::h_cls
  uint64_t* off = nullptr;  // SecDev::h_off
  ~SecHigh() {
    if (cls) cudaFree(cls);
    if (off) cudaFree(off);
  }
};

struct SecTables {
  SecDev dev{};
  std::vector<void*> bufs;
  std::shared_ptr<SecHigh> high;
};

void sec_free(SecTables* t) {
  if (!t) return;
  for (void* p : t->bufs)
    if (p) cudaFree(p);
  delete t;
}

const SecDev& sec_dev(const SecTables* t) { return t->dev; }

namespace {

template <class X>
Status up(SecTables* T, const std::vector<X>& v, const X** out, cudaStream_t st) {
  void* p = nullptr;
  const size_t b = sizeof(X) * std::max<size_t>(1, v.size());
  cudaError_t e = cudaMalloc(&p, b);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return {e == cudaErrorMemoryAllocation ? HPHI_ERR_OUT_OF_MEMORY : HPHI_ERR_CUDA,
            std::string("split-row tables: cudaMalloc(") + std::to_string(b) + "): " + cudaGetErrorString(e)};
  }
  T->bufs.push_back(p);
  if (!v.empty()) HPHI_CUDA_TRY(cudaMemcpyAsync(p, v.data(), sizeof(X) * v.size(), cudaMemcpyHostToDevice, st));
  *out = reinterpret_cast<const X*>(p);
  return {};
}

// device room for n values, owned by T
template <class X>
Status room(SecTables* T, size_t n, X** out) {
  void* p = nullptr;
  const size_t b = sizeof(X) * std::max<size_t>(1, n);
  const cudaError_t e = cudaMalloc(&p, b);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return {e == cudaErrorMemoryAllocation ? HPHI_ERR_OUT_OF_MEMORY : HPHI_ERR_CUDA,
            std::string("split-row tables: cudaMalloc(") + std::to_string(b) + "): " + cudaGetErrorString(e)};
  }
  T->bufs.push_back(p);
  *out = reinterpret_cast<X*>(p);
  return {};
}

// neighbour lists of one low class: nbr[slot * n + u] = rank of lo ^ mask | class << 24
__global__ void k_sec_nbr(const uint32_t* __restrict__ list, int n, const uint32_t* __restrict__ rank,
                          const uint32_t* __restrict__ bonds, int n_bonds, uint32_t* __restrict__ nbr,
                          uint8_t* __restrict__ deg) {
  const int u = blockIdx.x * kThreads + threadIdx.x;
  if (u >= n) return;
  const uint32_t lo = list[u];
  int c = 0;
  for (int k = 0; k < n_bonds; ++k) {
    const uint32_t m = bonds[k] & 0xffffffu;
    if (__popc(lo & m) == 1) nbr[(int64_t)(c++) * n + u] = rank[lo ^ m] | (bonds[k] & 0xff000000u);
  }
  deg[u] = (uint8_t)c;
}

}  // namespace

Status sec_build(const SecTerms& t, int L, int K, int esz, SecHighCache& high, SecTables** out, cudaStream_t st) {
  *out = nullptr;
  Analysis a = analyse(t);
  if (!a.ok) return {HPHI_ERR_UNSUPPORTED, a.why};
  const int N = t.n_sites, n1 = t.n_ones;
  if (!split_ok(N, L)) return {HPHI_ERR_INVALID_ARG, "split-row path: low part of 1..20 bits, high part of 1..22"};
  if (K < 1 || K > 8 || (K & (K - 1))) return {HPHI_ERR_INVALID_ARG, "split-row path: tile rows K in {1, 2, 4, 8}"};
  const int H = N - L;
  const uint64_t nqmax = longest_row(N, n1, L);
  if (nqmax == 0) return {HPHI_ERR_INVALID_ARG, "split-row path: empty sector"};
  if (nqmax > 65535) return {HPHI_ERR_UNSUPPORTED, "split-row path: rows longer than 65,535 entries"};
  const uint32_t nL = 1u << L, nH = 1u << H;

  std::unique_ptr<SecTables, SecTablesDeleter> T(new SecTables());
  SecDev& d = T->dev;
  d.L = L;
  d.H = H;
  d.n_ones = n1;
  d.dim = (int64_t)binom_u(N, n1);
  d.K = K;
  d.nq_max = (int)nqmax;
  d.n_cls = (int)a.cls.size();
  d.one_cls = a.cls.size() <= 1 ? 1 : 0;
  for (size_t c = 0; c < a.cls.size(); ++c) {
    d.coef[c] = a.cls[c];
    d.mult[c] = a.int_ok ? a.mult[c] : 0;
  }
  d.unit = a.unit;
  d.qextra = a.qextra;
  d.dint = a.dint ? 1 : 0;

  {
    const std::string why = straddle_limits(a, L);
    if (!why.empty()) return {HPHI_ERR_UNSUPPORTED, why};
  }
  // low side: popcount-grouped list and ranks
  std::vector<uint32_t> lo_rank(nL), lo_list(nL);
  {
    std::vector<uint32_t> cnt(L + 2, 0);
    for (int q = 0; q <= L; ++q) cnt[q + 1] = cnt[q] + (uint32_t)binom_u(L, q);
    for (int q = 0; q <= L + 1; ++q) d.lo_off[q] = cnt[q];
    std::vector<uint32_t> fill(cnt.begin(), cnt.end() - 1);
    for (uint32_t lo = 0; lo < nL; ++lo) {  // ascending, so each class comes out ascending
      const int q = __builtin_popcount(lo);
      lo_rank[lo] = fill[q] - cnt[q];
      lo_list[fill[q]++] = lo;
    }
  }
  // the low-part tables cover the classes present, q in [n1 - H, n1] within [0, L]
  const int qmin = std::max(0, n1 - H), qmax = std::min(L, n1);
  d.lo_stride = 0;
  for (int q = qmin; q <= qmax; ++q) {
    d.lo_pad[q] = (uint32_t)d.lo_stride;
    d.lo_stride += (d.lo_off[q + 1] - d.lo_off[q] + 31) / 32 * 32;
  }
  // bonds by pass, class by class
  d.hL = high_L(N, L);
  d.hH = N - d.hL;
  std::vector<int> order(a.bonds.size());
  for (size_t k = 0; k < order.size(); ++k) order[k] = (int)k;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return a.bond_cls[x] < a.bond_cls[y]; });
  std::vector<uint32_t> ll, hh;  // ll: the two low bits | class << 24
  std::vector<int> stb;
  for (int c = 0; c <= kSecMaxCls; ++c) d.hh_c0[c] = 0;
  for (int k : order) {
    const Bond& b = a.bonds[k];
    const int c = a.bond_cls[k];
    if (b.i >= d.hL) {
      hh.push_back((1u << (b.i - d.hL)) | (1u << (b.j - d.hL)));
      for (int e = c + 1; e <= kSecMaxCls; ++e) ++d.hh_c0[e];
    } else if (b.j < L) {
      ll.push_back((1u << b.i) | (1u << b.j) | ((uint32_t)c << 24));
    } else {
      stb.push_back(k);
    }
  }
  d.n_str = (int)stb.size();
  for (int n = 0; n < d.n_str; ++n) {
    d.str_a[n] = (uint8_t)(a.bonds[stb[n]].j - L);
    d.str_cls[n] = (uint8_t)a.bond_cls[stb[n]];
  }
  // diagonal counts: field g of 8 bits
  auto counts = [&](uint64_t s, int side) -> uint16_t {  // side 0: low part only, 1: high part only
    uint32_t packed = 0;
    for (int g = 0; g < a.n_dg; ++g) {
      int c = 0;
      for (const auto& pr : a.gpairs[g]) {
        const bool lo_pair = pr.second < L, hi_pair = pr.first >= L;
        if ((side == 0 && lo_pair) || (side == 1 && hi_pair)) c += (int)((s >> pr.first) & (s >> pr.second) & 1ull);
      }
      const uint64_t sites = a.gsites[g] & (side == 0 ? ((1ull << L) - 1ull) : ~((1ull << L) - 1ull));
      c += __builtin_popcountll(s & sites);
      packed |= (uint32_t)c << (8 * g);
    }
    return (uint16_t)packed;
  };
  std::vector<uint2> lo_info((size_t)d.lo_stride, make_uint2(0u, 0u));
  const int n_sg = (d.n_str + 3) / 4;
  std::vector<uint16_t> str_rank((size_t)std::max(1, n_sg) * 4 * (size_t)d.lo_stride, 0);
  for (int q = qmin; q <= qmax; ++q)
    for (uint32_t u = 0; u < d.lo_off[q + 1] - d.lo_off[q]; ++u) {
      const uint32_t lo = lo_list[d.lo_off[q] + u];
      const size_t j = d.lo_pad[q] + u;
      const uint32_t dc = counts(lo, 0);
      uint32_t bits = 0;
      for (int n = 0; n < d.n_str; ++n) {
        const int b = a.bonds[stb[n]].i;
        bits |= ((lo >> b) & 1u) << n;
        // ranks in classes that never receive a straddling gather may exceed 16 bits; unused
        const uint32_t r = lo_rank[lo ^ (1u << b)];
        str_rank[((size_t)(n / 4) * (size_t)d.lo_stride + j) * 4 + (n % 4)] = (uint16_t)(r <= 65535 ? r : 0);
      }
      lo_info[j] = make_uint2(lo | ((dc & 0xffu) << 20), bits | ((dc >> 8) << 24));
    }
  // straddling S^z S^z pairs in layers: a pair joins the first layer of its group that has
  // no pair on the same low site yet (one low bit counts one pair per layer)
  d.n_sp = 0;
  d.n_sl = 0;
  std::vector<uint32_t> layer_bits;
  for (int g = 0; g < a.n_dg; ++g)
    for (const auto& pr : a.gpairs[g]) {
      if (pr.first < L && pr.second >= L) {
        const uint32_t bit = 1u << pr.first;
        int l = 0;
        while (l < d.n_sl && (d.sp_lg[l] != g || (layer_bits[l] & bit))) ++l;
        if (l == d.n_sl) {
          d.sp_lg[d.n_sl++] = (uint8_t)g;
          layer_bits.push_back(0u);
        }
        layer_bits[l] |= bit;
        d.sp_a[d.n_sp] = (uint8_t)(pr.second - L);
        d.sp_b[d.n_sp] = (uint8_t)pr.first;
        d.sp_l[d.n_sp] = (uint8_t)l;
        ++d.n_sp;
      }
    }
  d.n_dg = a.n_dg;
  d.dstride = a.gmax[0] + 1;
  std::vector<double> dtab((size_t)(a.gmax[0] + 1) * (a.gmax[1] + 1));
  for (int x = 0; x <= a.gmax[0]; ++x)
    for (int y = 0; y <= a.gmax[1]; ++y) dtab[(size_t)x + (size_t)d.dstride * y] = a.c0 + a.gcoef[0] * x + a.gcoef[1] * y;
  d.dtab_n = (int)dtab.size();
  // high side: row offsets, neighbour lists, diagonal counts
  std::vector<uint64_t> hi_off(nH);
  {
    uint64_t run = 0;
    for (uint32_t hi = 0; hi < nH; ++hi) {
      hi_off[hi] = run;
      run += binom_u(L, n1 - __builtin_popcount(hi));
    }
    if (run != (uint64_t)d.dim) return {HPHI_ERR_CUDA, "split-row path: row offsets do not add up to the dimension"};
  }
  std::vector<uint16_t> hi_diag(nH, 0);
  for (uint32_t hi = 0; hi < nH; ++hi) hi_diag[hi] = counts((uint64_t)hi << L, 1);
  // classes of pass H: high parts grouped by popcount
  d.n_pc = 0;
  {
    uint32_t row0 = 0;
    for (int p = 0; p <= d.hH; ++p) {
      const uint32_t rows = (uint32_t)binom_u(d.hH, p);
      const int q = n1 - p;
      if (q >= 0 && q <= d.hL) {
        d.pc_row0[d.n_pc] = row0;
        d.pc_rows[d.n_pc] = rows;
        d.pc_nq[d.n_pc] = (uint32_t)binom_u(d.hL, q);
        ++d.n_pc;
      }
      row0 += rows;
    }
  }
  // row-pass tiles.  A row is read three times: staged by its own tile, and gathered by the
  // tiles of its straddling partners hi ^ 2^a (a in S, the high bits of the straddling bonds),
  // which lie one class above or below.  Blocks of high parts that agree outside S are closed
  // under those flips; a block runs class by class, so a row's partners are read while its
  // neighbouring classes run and it stays in L2 between the three reads.  Up to K rows of one
  // class per tile.
  std::vector<uint32_t> hi_seq, tiles;
  {
    uint32_t S = 0;
    for (int n = 0; n < d.n_str; ++n) S |= 1u << d.str_a[n];
    // blocks of at least 2^8 high parts, so that the classes of a block fill tiles of K rows
    for (int b = 0; b < H && __builtin_popcount(S) < std::min(H, 8); ++b) S |= 1u << b;
    const uint32_t nonS = (uint32_t)(nH - 1) & ~S;
    std::vector<uint32_t> sv;  // the 2^|S| settings of the bits of S
    for (uint32_t x = S;; x = (x - 1) & S) {
      sv.push_back(x);
      if (x == 0) break;
    }
    std::sort(sv.begin(), sv.end());
    std::vector<uint32_t> in_cls;
    for (uint32_t o = 0;; o = ((o | S) + 1) & nonS) {  // the settings of the other bits, ascending
      for (int p = std::max(0, n1 - L); p <= std::min(H, n1); ++p) {
        in_cls.clear();
        for (uint32_t x : sv)
          if (__builtin_popcount(o | x) == p) in_cls.push_back(o | x);
        for (size_t r = 0; r < in_cls.size(); r += (size_t)K) {
          const size_t nk = std::min<size_t>((size_t)K, in_cls.size() - r);
          tiles.push_back((uint32_t)hi_seq.size() | ((uint32_t)(nk - 1) << 24));
          hi_seq.insert(hi_seq.end(), in_cls.begin() + (long)r, in_cls.begin() + (long)(r + nk));
        }
      }
      if (o == nonS) break;
    }
  }
  d.n_tiles = (int64_t)tiles.size();

  Status s;
  if ((s = up(T.get(), lo_info, &d.lo_info, st)).code) return s;
  {
    const uint16_t* p16 = nullptr;
    if ((s = up(T.get(), str_rank, &p16, st)).code) return s;
    d.str_rank4 = reinterpret_cast<const uint2*>(p16);
  }
  if ((s = up(T.get(), hh, &d.hh_mask, st)).code) return s;
  if ((s = up(T.get(), hi_off, &d.hi_off, st)).code) return s;
  if ((s = up(T.get(), hi_diag, &d.hi_diag, st)).code) return s;
  if ((s = up(T.get(), dtab, &d.dtab, st)).code) return s;
  if ((s = up(T.get(), hi_seq, &d.hi_seq, st)).code) return s;
  if ((s = up(T.get(), tiles, &d.tiles, st)).code) return s;
  // the gather table (per class, in its padded place) and pass H's row offsets and class lists
  // are built on the device; what only the builders read is freed with `tmp`
  SecTables tmp;
  struct Free {
    SecTables& t;
    ~Free() {
      for (void* p : t.bufs) cudaFree(p);
    }
  } free_tmp{tmp};
  const uint32_t *g_rank = nullptr, *g_list = nullptr, *g_ll = nullptr, *g_off = nullptr;
  if ((s = up(&tmp, lo_rank, &g_rank, st)).code) return s;
  if ((s = up(&tmp, lo_list, &g_list, st)).code) return s;
  if ((s = up(&tmp, ll, &g_ll, st)).code) return s;
  const int n_ll = (int)ll.size();
  const int slots = std::max(1, (n_ll + 4 * kGatherChunk - 1) / (4 * kGatherChunk)) * 4 * kGatherChunk;
  uint32_t* g_nbr = nullptr;
  uint8_t* g_deg = nullptr;
  uint2* rec = nullptr;
  uint4* hdr = nullptr;
  if ((s = room(&tmp, (size_t)std::max(1, n_ll) * nqmax, &g_nbr)).code) return s;
  if ((s = room(&tmp, nqmax, &g_deg)).code) return s;
  if ((s = room(T.get(), (size_t)(slots / 4) * (size_t)d.lo_stride, &rec)).code) return s;
  if ((s = room(T.get(), (size_t)d.lo_stride / 32, &hdr)).code) return s;
  const int entry = (int)(K * esz);
  for (int q = qmin; q <= qmax; ++q) {
    const int n = (int)(d.lo_off[q + 1] - d.lo_off[q]);
    k_sec_nbr<<<(n + kThreads - 1) / kThreads, kThreads, 0, st>>>(g_list + d.lo_off[q], n, g_rank, g_ll, n_ll, g_nbr, g_deg);
    HPHI_CUDA_TRY(cudaGetLastError());
    if ((s = build_gather_table(g_nbr, n, g_deg, n_ll, n, 24, std::max(1, d.n_cls), d.nq_max, entry, rec, d.lo_stride,
                                d.lo_pad[q], slots, hdr, st)).code)
      return s;
  }
  T->high = high[d.hL].lock();
  if (!T->high) {
    T->high = std::make_shared<SecHigh>();
    const size_t n_h = (size_t)1 << d.hH;
    SecTables own;  // (its buffers pass to T->high)
    uint32_t* h_rank = nullptr;
    if ((s = room(&tmp, n_h, &h_rank)).code) return s;
    if ((s = room(&own, n_h, &T->high->cls)).code) return s;
    if ((s = room(&own, n_h, &T->high->off)).code) return s;
    std::vector<uint32_t> off(d.hH + 2, 0);
    for (int p = 0; p <= d.hH; ++p) off[p + 1] = off[p] + (uint32_t)binom_u(d.hH, p);
    if ((s = up(&tmp, off, &g_off, st)).code) return s;
    HPHI_CUDA_TRY(cudaStreamSynchronize(st));  // `off` dies here
    if ((s = build_popcount_tables(d.hH, h_rank, T->high->cls, g_off, st)).code) return s;
    if ((s = build_hi_offsets(d.hL, d.hH, n1, T->high->off, st)).code) return s;
    high[d.hL] = T->high;
  }
  d.lo_rec = rec;
  d.lo_hdr = hdr;
  d.h_cls = T->high->cls;
  d.h_off = T->high->off;
  HPHI_CUDA_TRY(cudaStreamSynchronize(st));  // host vectors die here
  *out = T.release();
  return {};
}

// ====================================================================== kernels
namespace {

constexpr int kHiWarps = kThreads / 32;
constexpr int kHiClaim = 4;  // items per warp per counter claim

// weight of exchange class c: fp32 the coefficient, fixed point the integer multiple
template <class T>
__device__ __forceinline__ T sec_w(const SecDev& d, int c);
template <>
__device__ __forceinline__ float sec_w<float>(const SecDev& d, int c) { return (float)d.coef[c]; }
template <>
__device__ __forceinline__ long long sec_w<long long>(const SecDev& d, int c) { return (long long)d.mult[c]; }

// pass H: W[row hi][col] = sum over active bonds above the split hL of w X[row hi'][col].  Warp
// items (class, stripe of 32 * EPT columns, row) run class by class and stripe by stripe,
// claimed in order from a counter, so the stripe of all rows of the class stays in L2 while it
// is used.  Lane k of the warp tests bond k and fetches its partner row's offset; the active
// ones are compacted into shared memory and read back as broadcasts.  Bonds of one coefficient
// class are summed plainly and weighted once.  6x5 torus, S^z = 0 (155,117,520 rows), int64, 30
// bonds at hL = 12 (25 lie above pass R's L = 14): 1.09 ms, bound by the loads' L1
// wavefronts (84 %), the integer pipe (65 %) and L2 (69 %).
template <class T, int EPT, bool ONE>
__global__ void __launch_bounds__(kThreads) k_sec_hi(const SecDev d, const T* __restrict__ X, T* W,
                                                     const int* __restrict__ done,
                                                     unsigned long long* __restrict__ counter) {
  if (done != nullptr && *done) return;
  constexpr int SW = 32 * EPT;
  __shared__ long long s_item0[kSecMaxHH + 2];
  __shared__ uint32_t s_nrow[kSecMaxHH + 1], s_nq[kSecMaxHH + 1], s_row0[kSecMaxHH + 1];
  __shared__ int s_c0[kSecMaxCls + 1];
  __shared__ T s_w[kSecMaxCls];
  __shared__ unsigned long long s_claim;
  __shared__ uint64_t s_src[kHiWarps][32];  // per warp: first element of each active partner row
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    long long acc = 0;
    for (int i = 0; i < d.n_pc; ++i) {
      s_item0[i] = acc;
      s_nrow[i] = d.pc_rows[i];
      s_nq[i] = d.pc_nq[i];
      s_row0[i] = d.pc_row0[i];
      acc += (long long)d.pc_rows[i] * ((d.pc_nq[i] + SW - 1) / SW);
    }
    s_item0[d.n_pc] = acc;
  }
  if (tid < kSecMaxCls) s_w[tid] = tid < d.n_cls ? sec_w<T>(d, tid) : (T)0;
  if (tid <= kSecMaxCls) s_c0[tid] = d.hh_c0[tid];
  __syncthreads();
  const long long total = s_item0[d.n_pc];
  const int n_cls = ONE ? 1 : d.n_cls;
  for (;;) {
    if (tid == 0) s_claim = atomicAdd(counter, (unsigned long long)(kHiWarps * kHiClaim));
    __syncthreads();
    const long long base = (long long)s_claim;
    __syncthreads();
    if (base >= total) break;
    for (int it = 0; it < kHiClaim; ++it) {
      const long long item = base + (long long)it * kHiWarps + warp;  // the CTA's warps on neighbouring rows
      if (item >= total) break;
      int pc = 0;
      while (item >= s_item0[pc + 1]) ++pc;
      const long long k = item - s_item0[pc];
      const uint32_t nrow = s_nrow[pc];
      const uint32_t sidx = (uint32_t)k / nrow;  // fewer than 2^32 items a class
      const uint32_t r = (uint32_t)k - sidx * nrow;
      const int nq = (int)s_nq[pc];
      const uint32_t hi = __ldg(d.h_cls + s_row0[pc] + r);
      const uint64_t o = __ldg(d.h_off + hi);
      const int col0 = (int)sidx * SW + lane;
      const bool full = (int)sidx * SW + SW <= nq;  // the whole stripe lies inside the row
      T tot[EPT];
#pragma unroll
      for (int j = 0; j < EPT; ++j) tot[j] = (T)0;
      for (int c = 0; c < n_cls; ++c) {
        T acc[EPT];
#pragma unroll
        for (int j = 0; j < EPT; ++j) acc[j] = (T)0;
        const int b1 = s_c0[c + 1];
        for (int qb = s_c0[c]; qb < b1; qb += 32) {
          const uint32_t m = qb + lane < b1 ? __ldg(d.hh_mask + qb + lane) : 0u;
          const bool on = __popc(hi & m) == 1;
          const unsigned bal = __ballot_sync(0xffffffffu, on);  // the previous batch has been read
          if (on) s_src[warp][__popc(bal & ((1u << lane) - 1u))] = __ldg(d.h_off + (hi ^ m));
          const int nn = __popc(bal);
          __syncwarp();
          for (int q0 = 0; q0 < nn; q0 += 4) {
            T x[4][EPT];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
              const bool live = q0 + t < nn;
              const T* p = X + s_src[warp][(q0 + t) & 31] + col0;
#pragma unroll
              for (int j = 0; j < EPT; ++j) x[t][j] = (live && (full || col0 + j * 32 < nq)) ? __ldg(p + j * 32) : (T)0;
            }
#pragma unroll
            for (int t = 0; t < 4; ++t)
#pragma unroll
              for (int j = 0; j < EPT; ++j) acc[j] += x[t][j];
          }
          __syncwarp();
        }
        if constexpr (ONE) {
#pragma unroll
          for (int j = 0; j < EPT; ++j) tot[j] = acc[j];
        } else {
          const T wt = s_w[c];
#pragma unroll
          for (int j = 0; j < EPT; ++j) tot[j] += wt * acc[j];
        }
      }
#pragma unroll
      for (int j = 0; j < EPT; ++j) {
        const int col = col0 + j * 32;
        if (col < nq) W[o + col] = tot[j];
      }
    }
  }
}

// K consecutive values of an interleaved shared-memory tile with the widest aligned loads
template <class T, int K>
__device__ __forceinline__ void tile_load(const T* p, T* out) {
  if constexpr (sizeof(T) * K == 16 && sizeof(T) == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    out[0] = t.x; out[1] = t.y; out[2] = t.z; out[3] = t.w;
  } else if constexpr (sizeof(T) * K == 16 && sizeof(T) == 8) {
    const longlong2 t = *reinterpret_cast<const longlong2*>(p);
    out[0] = t.x; out[1] = t.y;
  } else if constexpr (sizeof(T) * K == 8 && sizeof(T) == 4) {
    const float2 t = *reinterpret_cast<const float2*>(p);
    out[0] = t.x; out[1] = t.y;
  } else {
#pragma unroll
    for (int m = 0; m < K; ++m) out[m] = p[m];
  }
}

// a tile's rows as pass R keeps them in shared memory
template <int K>
struct __align__(8) LoRows {
  uint64_t roff[K];
  uint32_t hrow[K], hdiag[K];
  uint32_t hb[K];                // bit n: the high bit of straddling bond n
  uint32_t spm[K][kSecMaxSl];
  int nk;                        // 0: no tile left
};

// pass R: K rows of one class in shared memory; the bonds inside the row from the gather table,
// straddling exchange gathered from the partner rows, diagonal from packed counts, plus the
// pass-H sums Wh, then the fused epilogue.  X is the input (fp32) or its fixed-point copy.  A
// thread owns one column of the K rows at a time: the table's records are streamed a chunk
// ahead across columns, W and the previous Lanczos vector are requested before the straddling
// gathers, which run four bonds (4 K loads) at a time.
//
// 6x5 torus, S^z = 0 (155,117,520 rows), Lanczos step on GB300: fp64 2.58 ms (L = 14, two rows a
// tile), fp32 1.62 ms (L = 15, four rows).  Instruction issue (65 %) and shared-memory wavefronts
// (59 %) share it with the latencies of a tile's start and of the straddling gathers: with the
// gathers in the tile left out it takes 0.2 ms less, with the straddling ones left out 0.75 ms.
// Reading a bond's row pointers in 16-byte pieces and shifting the activity bits instead of testing
// bond numbers gave 0.16 and 0.23 ms, knowing the next tile's rows ahead 0.14 ms in fp64.
// One row a tile at L = 17, every bond below L in state order and all bonds across L gathered
// here, took 5.82 and 5.29 ms (pass H then 0.78 and 0.49 ms instead of 1.09 and 0.76 ms).
template <class T, int K, Epi E, int NT, bool ONE>
__global__ void __launch_bounds__(NT, (NT >= 1024) ? 1 : 2) k_sec_lo(const SecDev d, const T* __restrict__ X,
                                                                    const T* Wh, void* w, FusedArgs fa,
                                                                    const int* __restrict__ Ep,
                                                                    unsigned long long* __restrict__ claim) {
  using R = std::conditional_t<sizeof(T) == 4, float, double>;
  constexpr bool FIX = sizeof(T) == 8;
  constexpr int kZero = gather_lanes(K * (int)sizeof(T));
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* tile = reinterpret_cast<T*>(smem_raw);
  R* s_dtab = reinterpret_cast<R*>(smem_raw + (((size_t)(d.nq_max + kZero) * K * sizeof(T) + 15) / 16) * 16);
  int* s_dti = reinterpret_cast<int*>(s_dtab + d.dtab_n);  // fp64 with d.dint: the table in units
  __shared__ LoRows<K> s_cur, s_nxt;         // the rows of this tile and of the next
  __shared__ __align__(16) const T* s_ptr[kSecMaxStr][K];  // partner row of row m through the bond
  __shared__ T s_w[kSecMaxCls];
  __shared__ T s_sw[kSecMaxStr];             // weight of each straddling bond
  __shared__ double s_red[(NT / 32) * kMaxRedQ];

  if (fa.done != nullptr && *fa.done) return;
  const int tid = threadIdx.x;
  // fixed point: element = q 2^eoff; a power-of-two unit 2^k folds into the scales (see
  // k_hub_up): hv = (dg 2^-k xr + (+-S)) 2^(eoff + k)
  const int eoff = FIX ? (*Ep + d.qextra - 1078) : 0;
  const long long ubits = __double_as_longlong(d.unit);
  const int uexp = (int)((ubits >> 52) & 0x7ff);
  const bool u_p2 = FIX && (ubits & 0xfffffffffffffll) == 0 && uexp > 0 && uexp < 0x7ff;
  const bool u_neg = ubits < 0;
  const int u_l2 = uexp - 1023;
  const int e2 = eoff + u_l2;
  const bool fold = u_p2 && eoff >= -1022 && eoff <= 1023 && e2 >= -1022 && e2 <= 1023 &&
                    E != Epi::kTpq;
  const double s_eoff = fold ? __longlong_as_double((long long)(eoff + 1023) << 52) : 1.0;
  const double s_e2 = fold ? __longlong_as_double((long long)(e2 + 1023) << 52) : 1.0;
  const double r_k = fold ? __longlong_as_double((long long)(1023 - u_l2) << 52) : 1.0;
  for (int k = tid; k < d.dtab_n; k += NT) s_dtab[k] = (R)(d.dtab[k] * r_k);
  // integral diagonal (in units of `unit`): in the folded fp64 product and Lanczos step the
  // element is one exact int64 sum d q + (+-S), so its conversion is the only rounding, and
  // <x, H x> adds the exact products q (d q +- S) in 128 bits, moved to fp64 every 64 elements
  const bool dint = fold && d.dint;
  if (dint)
    for (int k = tid; k < d.dtab_n; k += NT) s_dti[k] = (int)__double2ll_rn(d.dtab[k] * r_k);
  __int128 ia = 0;
  int ic = 0;
  if (tid < kSecMaxCls) s_w[tid] = tid < d.n_cls ? sec_w<T>(d, tid) : (T)0;
  if (tid < d.n_str) s_sw[tid] = sec_w<T>(d, d.str_cls[tid]);
  for (int k = tid; k < kZero * K; k += NT) tile[(size_t)d.nq_max * K + k] = (T)0;  // entries unused slots read
  const EpiScalars<R> es = epi_scalars<R, E>(fa);
  const R inv = E == Epi::kTpq ? opaque((R)fa.scal[0]) : (R)0;
  const double c1e = FIX ? (double)es.c1 * (E == Epi::kShift ? r_k : s_e2) : 0.0;  // c1 in folded units
  const R coef0 = opaque((R)d.coef[0]);
  const int n_str = d.n_str, n_cls = d.n_cls;
  const uint32_t str_mask = n_str < 32 ? (1u << n_str) - 1u : 0xffffffffu;
  const int64_t stride = d.lo_stride;
  constexpr int NQ = n_red<E>() > 0 ? n_red<E>() : 1;  // reduced quantities of the epilogue
  Red<FIX, NQ> red;
  red.zero();
  int pmx = 0;  // fp64 Lanczos: largest exponent field of the P values written (fa.pexp)

  // tiles are claimed in order from a counter, so the tiles in flight stay a narrow window of
  // the processing order (a fixed stride would let CTAs drift apart over thousands of tiles);
  // with a CTA for every tile each takes its own, so the partial sums keep their places
  const bool own = d.n_tiles <= (int64_t)gridDim.x;
  // The last warp claims the next tile and reads its rows' table entries, four dependent reads
  // from memory, while the others gather: its share of a row is the shortest of a partial round.
  auto fetch = [&](int l) {
    __syncwarp();
    int64_t t = s_nxt.nk < 0 ? (int64_t)blockIdx.x : d.n_tiles;  // own: the first time round only
    __syncwarp();
    if (!own) {
      unsigned long long c = 0;
      if (l == 0) c = atomicAdd(claim, 1ull);
      t = (int64_t)__shfl_sync(0xffffffffu, c, 0);
    }
    if (t >= d.n_tiles) {
      if (l == 0) s_nxt.nk = 0;
      return;
    }
    if (l >= K) return;
    const uint32_t tw = __ldg(d.tiles + t);
    const uint32_t start = tw & 0xffffffu;
    const int nk = (int)(tw >> 24) + 1;
    uint64_t roff = 0;
    uint32_t hd = 0, hi = 0, hb = 0;
    for (int n = 0; n < kSecMaxSl; ++n) s_nxt.spm[l][n] = 0u;
    if (l < nk) {
      hi = __ldg(d.hi_seq + start + l);
      roff = __ldg(d.hi_off + hi);
      hd = __ldg(d.hi_diag + hi);
      for (int n = 0; n < d.n_sp; ++n)
        if ((hi >> d.sp_a[n]) & 1u) s_nxt.spm[l][d.sp_l[n]] |= 1u << d.sp_b[n];
      for (int n = 0; n < n_str; ++n) hb |= ((hi >> d.str_a[n]) & 1u) << n;
    }
    if (l == 0) s_nxt.nk = nk;
    s_nxt.roff[l] = roff;
    s_nxt.hrow[l] = hi;
    s_nxt.hdiag[l] = hd;
    s_nxt.hb[l] = hb;
  };
  if (tid == NT - 32) s_nxt.nk = -1;
  for (;;) {
    if (tid >= NT - 32) fetch(tid - (NT - 32));
    __syncthreads();  // the previous tile's rows are no longer read, this tile's are known
    const int nk = s_nxt.nk;
    if (nk == 0) break;
    for (int k = tid; k < (int)(sizeof(s_cur) / 8); k += NT)
      reinterpret_cast<uint2*>(&s_cur)[k] = reinterpret_cast<const uint2*>(&s_nxt)[k];
    const int q = d.n_ones - __popc(s_nxt.hrow[0]);
    const uint32_t lpad = d.lo_pad[q];
    const int nq = (int)(d.lo_off[q + 1] - d.lo_off[q]);
    const int nqp = (nq + 31) & ~31;
    if (tid < n_str) {  // partner rows, one bond per thread (read after the staging barrier)
      const uint32_t a = d.str_a[tid];
#pragma unroll
      for (int m = 0; m < K; ++m) s_ptr[tid][m] = X + (m < nk ? __ldg(d.hi_off + (s_nxt.hrow[m] ^ (1u << a))) : 0ull);
    }
    // stage the rows, tile[u * K + m] = X[row m][u]
    for (int u = tid; u < nq; u += NT) {
#pragma unroll
      for (int m = 0; m < K; ++m) {
        if (m < nk) copy_async<(int)sizeof(T)>(tile + u * K + m, X + s_nxt.roff[m] + u);
        else tile[u * K + m] = (T)0;
      }
    }
    // whole warps run to the padded row length: the table's padding reads zero entries
    const uint2* rec = d.lo_rec + lpad;
    const uint4* hdr = d.lo_hdr + (lpad >> 5);
    uint2 cur[kGatherChunk];
    uint4 hd = make_uint4(0u, 0u, 0u, 0u);
    if (tid < nqp) {
      if constexpr (ONE) hd.x = __ldg(&hdr[tid >> 5].x);
      else hd = __ldg(hdr + (tid >> 5));
#pragma unroll
      for (int j = 0; j < kGatherChunk; ++j) cur[j] = __ldg(rec + tid + j * stride);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    for (int u = tid; u < nqp; u += NT) {
      const bool on = u < nq;
      const uint4 h = hd;
      const int ng = ((int)(ONE ? h.x & 0xffffu : h.w >> 16) + 3) >> 2;
      const int un = u + NT < nqp ? u + NT : u;
      if constexpr (ONE) hd.x = __ldg(&hdr[un >> 5].x);
      else hd = __ldg(hdr + (un >> 5));
      const uint2 info = __ldg(d.lo_info + lpad + u);
      uint2 rk = n_str > 0 ? __ldg(d.str_rank4 + lpad + u) : make_uint2(0u, 0u);
      T acc[K];
#pragma unroll
      for (int m = 0; m < K; ++m) acc[m] = (T)0;
      int f = 0, fe = ONE ? 0 : gather_end(h, 0);  // class of the current slots and its end
      int c0 = 0;
      do {
        const uint2* src = c0 + kGatherChunk < ng ? rec + u + (int64_t)(c0 + kGatherChunk) * stride : rec + un;
        uint2 nxt[kGatherChunk];
#pragma unroll
        for (int j = 0; j < kGatherChunk; ++j) nxt[j] = __ldg(src + j * stride);
#pragma unroll
        for (int j = 0; j < kGatherChunk; ++j) {
          if (c0 + j < ng) {
            const uint2 r = cur[j];
            T v[4][K];
            tile_load<T, K>(tile + (r.x & 0xffffu) * K, v[0]);
            tile_load<T, K>(tile + (r.x >> 16) * K, v[1]);
            tile_load<T, K>(tile + (r.y & 0xffffu) * K, v[2]);
            tile_load<T, K>(tile + (r.y >> 16) * K, v[3]);
            if constexpr (ONE) {
#pragma unroll
              for (int m = 0; m < K; ++m) acc[m] += (v[0][m] + v[1][m]) + (v[2][m] + v[3][m]);
            } else {
              const int s0 = 4 * (c0 + j);
              while (f + 1 < n_cls && s0 >= fe) fe = gather_end(h, ++f);
              if (s0 + 4 <= fe || f + 1 == n_cls) {  // one class, or padding after the last
                const T wf = s_w[f];
#pragma unroll
                for (int m = 0; m < K; ++m) acc[m] += wf * ((v[0][m] + v[1][m]) + (v[2][m] + v[3][m]));
              } else {
                int ff = f, ffe = fe;
#pragma unroll
                for (int t4 = 0; t4 < 4; ++t4) {
                  while (ff + 1 < n_cls && s0 + t4 >= ffe) ffe = gather_end(h, ++ff);
                  const T wf = s_w[ff];
#pragma unroll
                  for (int m = 0; m < K; ++m) acc[m] += wf * v[t4][m];
                }
              }
            }
          }
        }
#pragma unroll
        for (int j = 0; j < kGatherChunk; ++j) cur[j] = nxt[j];
        c0 += kGatherChunk;
      } while (c0 < ng);
      // this column's W and (Lanczos) previous vector, then the straddling gathers
      T wv[K];
      R pin[K];
#pragma unroll
      for (int m = 0; m < K; ++m) {
        const int64_t idx = (int64_t)s_cur.roff[m] + u;
        wv[m] = (on && m < nk) ? Wh[idx] : (T)0;
        if constexpr (E == Epi::kLanczos1)
          pin[m] = (on && m < nk) ? reinterpret_cast<const R*>(fa.in ? fa.in : fa.out)[idx] : (R)0;
      }
      uint32_t act[K];  // bond n acts on row m: its low bit differs from its high bit
#pragma unroll
      for (int m = 0; m < K; ++m) act[m] = (on && m < nk) ? (info.y ^ s_cur.hb[m]) & str_mask : 0u;
      for (int n0 = 0; n0 < n_str; n0 += 4) {
        const uint2 r = rk;
        if (n0 + 4 < n_str) rk = __ldg(d.str_rank4 + (int64_t)(n0 / 4 + 1) * stride + lpad + u);
        T x[4][K];
#pragma unroll
        for (int t4 = 0; t4 < 4; ++t4) {
          const uint32_t word = t4 < 2 ? r.x : r.y;
          const uint32_t col = (t4 & 1) ? word >> 16 : word & 0xffffu;
          const T* pr[K];  // the rows' pointers in 16-byte reads
          if constexpr (K >= 2) {
#pragma unroll
            for (int m = 0; m < K; m += 2) {
              const ulonglong2 two = *reinterpret_cast<const ulonglong2*>(&s_ptr[n0 + t4][m]);
              pr[m] = reinterpret_cast<const T*>(two.x);
              pr[m + 1] = reinterpret_cast<const T*>(two.y);
            }
          } else {
            pr[0] = s_ptr[n0 + t4][0];
          }
#pragma unroll
          for (int m = 0; m < K; ++m) {
            x[t4][m] = (T)0;
            if (act[m] & (1u << t4)) x[t4][m] = __ldg(pr[m] + col);
          }
        }
#pragma unroll
        for (int m = 0; m < K; ++m) act[m] >>= 4;
        if constexpr (ONE) {
#pragma unroll
          for (int m = 0; m < K; ++m) acc[m] += (x[0][m] + x[1][m]) + (x[2][m] + x[3][m]);
        } else {
#pragma unroll
          for (int t4 = 0; t4 < 4; ++t4) {
            const T wn = n0 + t4 < n_str ? s_sw[n0 + t4] : (T)0;
#pragma unroll
            for (int m = 0; m < K; ++m) acc[m] += wn * x[t4][m];
          }
        }
      }
      if (!on) continue;
      // diagonal and the epilogue
      const uint32_t lo = info.x & 0xfffffu;
      const uint32_t ldc = (info.x >> 20) | ((info.y >> 24) << 8);
#pragma unroll
      for (int m = 0; m < K; ++m) {
        if (m >= nk) break;
        uint32_t c = ldc + s_cur.hdiag[m];
        for (int l = 0; l < d.n_sl; ++l) c += (uint32_t)__popc(lo & s_cur.spm[m][l]) << (8 * d.sp_lg[l]);
        const int ci = (int)(c & 0xffu) + d.dstride * (int)(c >> 8);
        const int64_t idx = (int64_t)s_cur.roff[m] + u;
        const T xq = tile[u * K + m];
        const T S = acc[m] + wv[m];
        if constexpr (!FIX) {
          const R dg = s_dtab[ci];
          const float hv = ONE ? dg * xq + coef0 * S : dg * xq + S;
          if constexpr (E == Epi::kLanczos1) {
            reinterpret_cast<float*>(fa.out)[idx] = es.c1 * hv - es.c2 * pin[m];
            red.add(0, xq, hv);
            red.tick();
          } else {
            epilogue<float, E, NQ>(idx, xq, 0.f, hv, 0.f, reinterpret_cast<float*>(w), fa, es, inv, red);
          }
        } else {
          if (dint) {
            const long long hq = (long long)s_dti[ci] * xq + (u_neg ? -S : S);  // hv = hq 2^e2
            const double hvu = __ll2double_rn(hq);
            if constexpr (E == Epi::kStore) {
              reinterpret_cast<double*>(w)[idx] = hvu * s_e2;
            } else if constexpr (E == Epi::kLanczos1) {
              const double pv = fma(c1e, hvu, -(es.c2 * pin[m]));
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
              shift_folded(hvu, __ll2double_rn(xq), c1e, s_e2, idx, fa, red);
            }
            continue;
          }
          const R dg = s_dtab[ci];
          const double xr = __ll2double_rn(xq);
          if (fold) {
            const double hvu = fma(dg, xr, __ll2double_rn(u_neg ? -S : S));  // hv = hvu 2^e2
            if constexpr (E == Epi::kStore) {
              reinterpret_cast<double*>(w)[idx] = hvu * s_e2;
            } else if constexpr (E == Epi::kLanczos1) {
              const double pv = fma(c1e, hvu, -(es.c2 * pin[m]));
              reinterpret_cast<double*>(fa.out)[idx] = pv;
              pmx = max(pmx, (int)((__double_as_longlong(pv) >> 52) & 0x7ff));
              red.add(0, xr, hvu);
              red.tick();
            } else if constexpr (E == Epi::kRefine) {
              refine_folded(hvu, xr, s_e2, idx, fa, red);
            } else if constexpr (E == Epi::kShift) {
              shift_folded(hvu, xr, c1e, s_e2, idx, fa, red);
            }
          } else {
            const double x = fix_to_double(xq, eoff);
            const double hv = fma((double)dg, x, d.unit * fix_to_double(S, eoff));
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
  }
  if constexpr (FIX && E == Epi::kLanczos1) {
    if (ic) red.add(0, i128_to_double(ia), 1.0);
    if (fa.pexp != nullptr) {
      pmx = (int)__reduce_max_sync(0xffffffffu, (unsigned)pmx);
      if ((tid & 31) == 0 && pmx > 0) atomicMax(fa.pexp, pmx);
    }
  }
  if constexpr (E != Epi::kStore) {
    constexpr int nq = n_red<E>();
    const int lane = tid & 31, wid = tid >> 5;
#pragma unroll
    for (int qq = 0; qq < nq; ++qq) {
      double x = red.get(qq);
      if (fold) x = folded_sum(x, qq, s_eoff, s_e2);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
      if (lane == 0) s_red[wid * kMaxRedQ + qq] = x;
    }
    __syncthreads();
    if (tid < nq) {
      double x = 0.0;
      for (int k = 0; k < NT / 32; ++k) x += s_red[k * kMaxRedQ + tid];
      fa.partials[(size_t)blockIdx.x * kMaxRedQ + tid] = x;
    }
  }
}

// ---------------------------------------------------------------- launch helpers
size_t lo_smem(const SecDev& d, int esz) {  // the rows, their zero entries, the diagonal table(s)
  return (((size_t)(d.nq_max + gather_lanes(d.K * esz)) * d.K * esz + 15) / 16) * 16 + (size_t)d.dtab_n * esz +
         (esz == 8 && d.dint ? (size_t)d.dtab_n * 4 : 0);
}

// row-pass threads: 1024 (one CTA per SM) for tiles above ~110 KB, else 512
int lo_threads(const SecDev& d, int esz) { return lo_smem(d, esz) > 110000 ? 1024 : 512; }

template <class KernelT>
int occupancy_of(KernelT kern, int nt, size_t smem) {
  int n = 0;
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, nt, smem) != cudaSuccess || n < 1) {
    cudaGetLastError();
    n = 1;
  }
  return n;
}

template <class T, int K, Epi E, bool ONE>
Status launch_lo_t(const SecDev& d, const T* X, const T* Wh, void* w, const FusedArgs& fa, const int* Ep, int grid,
                   unsigned long long* claim, cudaStream_t st) {
  const size_t smem = lo_smem(d, (int)sizeof(T));
  if (d.n_tiles > grid) HPHI_CUDA_TRY(cudaMemsetAsync(claim, 0, sizeof(unsigned long long), st));
#define HPHI_SECLO(NN)                                                                                        \
  HPHI_CUDA_TRY(cudaFuncSetAttribute(k_sec_lo<T, K, E, NN, ONE>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                     (int)smem));                                                             \
  k_sec_lo<T, K, E, NN, ONE><<<grid, NN, smem, st>>>(d, X, Wh, w, fa, Ep, claim);
  if (lo_threads(d, (int)sizeof(T)) == 1024) {
    HPHI_SECLO(1024)
  } else {
    HPHI_SECLO(512)
  }
#undef HPHI_SECLO
  HPHI_CUDA_TRY(cudaGetLastError());
  return {};
}

template <class T, int K, Epi E, bool ONE>
int lo_occupancy_t(const SecDev& d) {
  const size_t smem = lo_smem(d, (int)sizeof(T));
  return lo_threads(d, (int)sizeof(T)) == 1024 ? occupancy_of(k_sec_lo<T, K, E, 1024, ONE>, 1024, smem)
                                               : occupancy_of(k_sec_lo<T, K, E, 512, ONE>, 512, smem);
}

template <class T, Epi E>
Status launch_lo_k(const SecDev& d, const T* X, const T* Wh, void* w, const FusedArgs& fa, const int* Ep, int grid,
                   unsigned long long* claim, cudaStream_t st) {
  const bool one = d.one_cls != 0;
#define HPHI_SECK(KK)                                                                 \
  return one ? launch_lo_t<T, KK, E, true>(d, X, Wh, w, fa, Ep, grid, claim, st)      \
             : launch_lo_t<T, KK, E, false>(d, X, Wh, w, fa, Ep, grid, claim, st);
  switch (d.K) {
    case 8: HPHI_SECK(8)
    case 4: HPHI_SECK(4)
    case 2: HPHI_SECK(2)
    default: HPHI_SECK(1)
  }
#undef HPHI_SECK
}

template <class T, Epi E>
int lo_occupancy_k(const SecDev& d) {
  const bool one = d.one_cls != 0;
  switch (d.K) {
    case 8: return one ? lo_occupancy_t<T, 8, E, true>(d) : lo_occupancy_t<T, 8, E, false>(d);
    case 4: return one ? lo_occupancy_t<T, 4, E, true>(d) : lo_occupancy_t<T, 4, E, false>(d);
    case 2: return one ? lo_occupancy_t<T, 2, E, true>(d) : lo_occupancy_t<T, 2, E, false>(d);
    default: return one ? lo_occupancy_t<T, 1, E, true>(d) : lo_occupancy_t<T, 1, E, false>(d);
  }
}

template <class T>
Status launch_hi(const SecDev& d, const T* X, T* W, const int* done, unsigned long long* counter, cudaStream_t st) {
  HPHI_CUDA_TRY(cudaMemsetAsync(counter, 0, sizeof(unsigned long long), st));
  const int grid = num_sms() * 8;
  const bool one = d.one_cls != 0;
  // 1 KB row stripes per warp item (4 int64 / 8 fp32 columns per lane): wide stripes spread each
  // partner's address arithmetic and offset read over more columns.  The autotuner may halve them
  // (d.hi_cols), which halves the stripe of a class that should stay in L2.
  constexpr int EPT = sizeof(T) == 8 ? 4 : 8;
  if (d.hi_cols == EPT / 2) {
    if (one) k_sec_hi<T, EPT / 2, true><<<grid, kThreads, 0, st>>>(d, X, W, done, counter);
    else k_sec_hi<T, EPT / 2, false><<<grid, kThreads, 0, st>>>(d, X, W, done, counter);
  } else {
    if (one) k_sec_hi<T, EPT, true><<<grid, kThreads, 0, st>>>(d, X, W, done, counter);
    else k_sec_hi<T, EPT, false><<<grid, kThreads, 0, st>>>(d, X, W, done, counter);
  }
  HPHI_CUDA_TRY(cudaGetLastError());
  return {};
}

// scratch layout: fp64 [Q: dim int64][W: dim int64, Lanczos only][tail]; fp32 [W: dim float,
// Lanczos only][tail]; tail = 256 bytes: exponent (int) at 0 (and the QSlots ints at 4, 8,
// 192), pass-H counter (u64) at 64, pass-R tile counter (u64) at 128
size_t vec_bytes(const SecDev& d, int esz) { return (((size_t)d.dim * esz + 255) / 256) * 256; }

}  // namespace

size_t sec_scratch_bytes(const SecDev& d, int prec, Epi epi) {
  const int esz = prec == HPHI_FP64 ? 8 : 4;
  size_t b = 256;
  if (prec == HPHI_FP64) b += vec_bytes(d, 8);
  if (epi == Epi::kLanczos1) b += vec_bytes(d, esz);
  return b;
}

int* sec_exponent_slot(const SecDev& d, int prec, Epi epi, void* scratch) {
  return reinterpret_cast<int*>(static_cast<char*>(scratch) + sec_scratch_bytes(d, prec, epi) - 256);
}

// fp64: Q at the start of the scratch; tail ints: exponent of Q at 0, the exact exponents of
// the current / next vector at 4 and 8, the pass-1 exponent at 192
QSlots sec_qslots(const SecDev& d, int prec, Epi epi, void* scratch) {
  QSlots q;
  if (prec != HPHI_FP64 || scratch == nullptr) return q;
  char* tail = static_cast<char*>(scratch) + sec_scratch_bytes(d, prec, epi) - 256;
  q.Q = reinterpret_cast<long long*>(scratch);
  q.eq = reinterpret_cast<int*>(tail);
  q.ec[0] = reinterpret_cast<int*>(tail + 4);
  q.ec[1] = reinterpret_cast<int*>(tail + 8);
  q.ep = reinterpret_cast<int*>(tail + 192);
  q.extra = d.qextra;
  return q;
}

int sec_grid(const SecDev& d, int prec, Epi epi) {
  int occ = 1;
#define HPHI_SECOCC(TT)                                                      \
  switch (epi) {                                                             \
    case Epi::kStore: occ = lo_occupancy_k<TT, Epi::kStore>(d); break;       \
    case Epi::kLanczos1: occ = lo_occupancy_k<TT, Epi::kLanczos1>(d); break; \
    case Epi::kTpq: occ = lo_occupancy_k<TT, Epi::kTpq>(d); break;           \
    case Epi::kRefine: occ = lo_occupancy_k<TT, Epi::kRefine>(d); break;     \
    case Epi::kShift: occ = lo_occupancy_k<long long, Epi::kShift>(d); break; \
  }
  if (prec == HPHI_FP64) { HPHI_SECOCC(long long) } else { HPHI_SECOCC(float) }
#undef HPHI_SECOCC
  return (int)std::max<int64_t>(1, std::min<int64_t>(d.n_tiles, (int64_t)num_sms() * occ));
}

Status launch_sec(const SecDev& d, int prec, const void* v, void* w, void* scratch, Epi epi, const FusedArgs& fa,
                  int grid, cudaStream_t st) {
  if ((epi == Epi::kRefine || epi == Epi::kShift) && prec != HPHI_FP64)
    return {HPHI_ERR_INVALID_ARG, "refinement runs in fp64"};
  char* sc = static_cast<char*>(scratch);
  char* tail = sc + sec_scratch_bytes(d, prec, epi) - 256;
  int* Ep = reinterpret_cast<int*>(tail);
  unsigned long long* counter = reinterpret_cast<unsigned long long*>(tail + 64);
  unsigned long long* claim = reinterpret_cast<unsigned long long*>(tail + 128);
  // the output buffer receives the pass-H sums and is finished in place, except in Lanczos
  // steps, whose output (P) is also an input: their sums go to the scratch vector
  void* out = (epi == Epi::kStore) ? w : fa.out;
  if (prec == HPHI_FP64) {
    long long* Q = reinterpret_cast<long long*>(sc);
    long long* W = (epi == Epi::kLanczos1) ? reinterpret_cast<long long*>(sc + vec_bytes(d, 8))
                                           : reinterpret_cast<long long*>(out);
    Status s;
    if (fa.exp_ready != 2) {  // 2: the previous Lanczos pass 2 wrote Q and its exponent
      s = launch_quant_vec(reinterpret_cast<const double*>(v), Q, d.dim, Ep, fa.done, fa.exp_ready != 0, d.qextra, st);
      if (s.code) return s;
    }
    if (fa.pexp != nullptr) HPHI_CUDA_TRY(cudaMemsetAsync(fa.pexp, 0, sizeof(int), st));
    if ((s = launch_hi<long long>(d, Q, W, fa.done, counter, st)).code) return s;
    switch (epi) {
      case Epi::kStore: return launch_lo_k<long long, Epi::kStore>(d, Q, W, w, fa, Ep, grid, claim, st);
      case Epi::kLanczos1: return launch_lo_k<long long, Epi::kLanczos1>(d, Q, W, w, fa, Ep, grid, claim, st);
      case Epi::kTpq: return launch_lo_k<long long, Epi::kTpq>(d, Q, W, w, fa, Ep, grid, claim, st);
      case Epi::kRefine: return launch_lo_k<long long, Epi::kRefine>(d, Q, W, w, fa, Ep, grid, claim, st);
      case Epi::kShift: return launch_lo_k<long long, Epi::kShift>(d, Q, W, w, fa, Ep, grid, claim, st);
    }
  } else {
    const float* X = reinterpret_cast<const float*>(v);
    float* W = (epi == Epi::kLanczos1) ? reinterpret_cast<float*>(sc) : reinterpret_cast<float*>(out);
    Status s = launch_hi<float>(d, X, W, fa.done, counter, st);
    if (s.code) return s;
    switch (epi) {
      case Epi::kStore: return launch_lo_k<float, Epi::kStore>(d, X, W, w, fa, Ep, grid, claim, st);
      case Epi::kLanczos1: return launch_lo_k<float, Epi::kLanczos1>(d, X, W, w, fa, Ep, grid, claim, st);
      case Epi::kTpq: return launch_lo_k<float, Epi::kTpq>(d, X, W, w, fa, Ep, grid, claim, st);
      case Epi::kRefine:
      case Epi::kShift: break;
    }
  }
  return {HPHI_ERR_INVALID_ARG, "split-row path: unsupported precision / epilogue"};
}

}  // namespace hphi

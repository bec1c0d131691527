// Inverse iteration by conjugate gradients (section 3.4.1): y_{k+1} solves
// (H - E + delta) y_{k+1} = y_k, the shift delta > 0 keeping the operator positive definite
// when E lies at or just above the lowest eigenvalue, and the CG solve starting from y_k
// itself.  fp64 throughout; complex vectors run as real vectors of twice the length (H is
// Hermitian, so Re <u, A v> is the inner product CG needs).  Besides the caller's vector the
// solve keeps four: the iterate y, the residual r, the direction p and q = A p.
//
// A p = H p + c p (c = delta - E) is never stored: H p comes with <p, (H + c) p>, summed element
// by element, from the product's shift epilogue, and the residual update adds c p where it reads p
// anyway.  On the fixed-point paths the direction kernel also finds the new direction's largest
// exponent, so the next product quantises it on its own scale without a scan.
// 32 iterations on 24 sites (2.7 million rows) on GB300: 5.5 ms; 6.3 ms with a scan and a separate
// shift pass per product (9 kernels an iteration instead of 7).
//
// Every kernel streams its vectors once with four elements per thread one grid stride apart
// and leaves one fp64 partial sum per CTA; a one-CTA finaliser turns the partials into the
// CG scalars on the device, so a whole solve is a fixed launch sequence.
#include "common.cuh"

namespace hphi {
namespace {

__device__ double cg_block_sum(double x, double* sm) {
  const int tid = threadIdx.x;
  __syncthreads();  // an earlier sum's result has been read by every thread
  sm[tid] = x;
  __syncthreads();
  for (int off = kThreads / 2; off > 0; off >>= 1) {
    if (tid < off) sm[tid] += sm[tid + off];
    __syncthreads();
  }
  return sm[0];
}

__device__ __forceinline__ void cg_partial(double acc, double* partials, int q) {
  __shared__ double sm[kThreads];
  const double t = cg_block_sum(acc, sm);
  if (threadIdx.x == 0) partials[(size_t)blockIdx.x * kMaxRedQ + q] = t;
}

// mode 0: start of a solve: y <- b, r <- b - A b (q = H b), p <- r; partials |r|^2, |b|^2
// mode 1: y += alpha p, r -= alpha A p (q = H p); partial |r|^2
__global__ void __launch_bounds__(kThreads) k_cg_update(CgDev cg, int mode, const double* __restrict__ b,
                                                         double* __restrict__ y, double* __restrict__ r,
                                                         double* __restrict__ p, const double* __restrict__ q,
                                                         int64_t n, double* __restrict__ partials) {
  if (*cg.done) return;
  const double al = cg.s[1], c = cg.s[4];
  const int64_t stride = (int64_t)gridDim.x * kThreads;
  double rr = 0.0, bb = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < n; i += 4 * stride) {
    double a[4], qv[4], yv[4], rv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t k = i + u * stride;
      const bool on = k < n;
      a[u] = on ? (mode == 0 ? b[k] : p[k]) : 0.0;
      qv[u] = on ? q[k] : 0.0;
      yv[u] = on && mode != 0 ? y[k] : 0.0;
      rv[u] = on && mode != 0 ? r[k] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t k = i + u * stride;
      if (k >= n) break;
      const double ap = fma(c, a[u], qv[u]);
      double t;
      if (mode == 0) {
        t = a[u] - ap;
        y[k] = a[u];
        p[k] = t;
        bb = fma(a[u], a[u], bb);
      } else {
        y[k] = fma(al, a[u], yv[u]);
        t = fma(-al, ap, rv[u]);
      }
      r[k] = t;
      rr = fma(t, t, rr);
    }
  }
  cg_partial(rr, partials, 0);
  if (mode == 0) cg_partial(bb, partials, 1);
}

// p <- r + beta p; emax (may be null): the largest exponent field of the new p
__global__ void __launch_bounds__(kThreads) k_cg_dir(CgDev cg, const double* __restrict__ r, double* __restrict__ p,
                                                      int64_t n, int* emax) {
  if (*cg.done) return;
  const double be = cg.s[2];
  int mx = 0;
  const int64_t stride = (int64_t)gridDim.x * kThreads;
  for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < n; i += 4 * stride) {
    double rv[4], pv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t k = i + u * stride;
      rv[u] = k < n ? r[k] : 0.0;
      pv[u] = k < n ? p[k] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t k = i + u * stride;
      if (k >= n) break;
      const double t = fma(be, pv[u], rv[u]);
      p[k] = t;
      mx = max(mx, (__double2hiint(t) >> 20) & 0x7ff);
    }
  }
  if (emax != nullptr) {
    mx = (int)__reduce_max_sync(0xffffffffu, (unsigned)mx);
    if ((threadIdx.x & 31) == 0 && mx > 0) atomicMax(emax, mx);
  }
}

// x <- y / |y| (mode 0: partial |y|^2 first; mode 1: scale, the norm in s[9])
__global__ void __launch_bounds__(kThreads) k_cg_norm(CgDev cg, int mode, const double* __restrict__ y,
                                                       double* __restrict__ x, int64_t n,
                                                       double* __restrict__ partials) {
  const int64_t stride = (int64_t)gridDim.x * kThreads;
  if (mode == 0) {
    double acc = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < n; i += stride) acc = fma(y[i], y[i], acc);
    cg_partial(acc, partials, 0);
    return;
  }
  const double sc = cg.s[9];
  for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < n; i += stride) x[i] = y[i] * sc;
}

// Rayleigh quotient of x (unit) with hx = H x: partials <x, hx>, <hx, hx>; then |hx - e x|^2
__global__ void __launch_bounds__(kThreads) k_cg_rq(CgDev cg, int mode, const double* __restrict__ x,
                                                     const double* __restrict__ hx, int64_t n,
                                                     double* __restrict__ partials) {
  const int64_t stride = (int64_t)gridDim.x * kThreads;
  if (mode == 0) {
    double xh = 0.0, hh = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < n; i += stride) {
      xh = fma(x[i], hx[i], xh);
      hh = fma(hx[i], hx[i], hh);
    }
    cg_partial(xh, partials, 0);
    cg_partial(hh, partials, 1);
    return;
  }
  const double e = cg.s[6];
  double rr = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x; i < n; i += stride) {
    const double d = fma(-e, x[i], hx[i]);
    rr = fma(d, d, rr);
  }
  cg_partial(rr, partials, 0);
}

__device__ double cg_sum(const double* __restrict__ partials, int grid, int q, double* sm) {
  double s = 0.0;
  for (int b = threadIdx.x; b < grid; b += kThreads) s += partials[(size_t)b * kMaxRedQ + q];
  return cg_block_sum(s, sm);
}

// scalar steps of the solve, one CTA:
// 0 start (rr, |b|^2, done if r = 0)  1 alpha = rr / <p, A p>  2 beta = rr' / rr, test
// 3 the norm of y  4 e and the variance  5 the residual
// clear (may be null): an exponent slot the next kernel raises
__global__ void __launch_bounds__(kThreads) k_cg_fin(CgDev cg, int mode, const double* __restrict__ partials,
                                                      int grid, int* clear) {
  __shared__ double sm[kThreads];
  if ((mode == 1 || mode == 2) && *cg.done) return;
  const double s0 = cg_sum(partials, grid, 0, sm);
  const double s1 = (mode == 0 || mode == 4) ? cg_sum(partials, grid, 1, sm) : 0.0;
  if (threadIdx.x != 0) return;
  if (clear != nullptr) *clear = 0;
  if (mode == 0) {
    cg.s[0] = s0;
    cg.s[3] = s1;
    *cg.done = (s0 <= cg.s[5] * s1) ? 1 : 0;
  } else if (mode == 1) {
    if (!(s0 > 0.0)) {  // A is positive definite on a non-zero p: only p = 0 gives this
      *cg.done = 1;
      return;
    }
    cg.s[1] = cg.s[0] / s0;
  } else if (mode == 2) {
    cg.s[2] = s0 / cg.s[0];
    cg.s[0] = s0;
    *cg.steps += 1;
    if (s0 <= cg.s[5] * cg.s[3]) *cg.done = 1;
  } else if (mode == 3) {
    cg.s[9] = s0 > 0.0 ? 1.0 / sqrt(s0) : 0.0;
  } else if (mode == 4) {
    cg.s[6] = s0;          // <x|H|x>, x a unit vector
    cg.s[8] = s1 - s0 * s0;  // <H^2> - <H>^2
  } else {
    cg.s[7] = sqrt(s0);    // |H x - e x|
  }
}

}  // namespace

Status launch_cg_update(const CgDev& cg, int mode, const double* b, double* y, double* r, double* p, const double* q,
                        int64_t n, double* partials, int grid, cudaStream_t st) {
  k_cg_update<<<grid, kThreads, 0, st>>>(cg, mode, b, y, r, p, q, n, partials);
  HPHI_CUDA_TRY(cudaGetLastError());
  return {};
}

Status launch_cg_dir(const CgDev& cg, const double* r, double* p, int64_t n, int grid, int* emax, cudaStream_t st) {
  k_cg_dir<<<grid, kThreads, 0, st>>>(cg, r, p, n, emax);
  HPHI_CUDA_TRY(cudaGetLastError());
  return {};
}

Status launch_cg_norm(const CgDev& cg, int mode, const double* y, double* x, int64_t n, double* partials, int grid,
                      cudaStream_t st) {
  k_cg_norm<<<grid, kThreads, 0, st>>>(cg, mode, y, x, n, partials);
  HPHI_CUDA_TRY(cudaGetLastError());
  return {};
}

Status launch_cg_rq(const CgDev& cg, int mode, const double* x, const double* hx, int64_t n, double* partials,
                    int grid, cudaStream_t st) {
  k_cg_rq<<<grid, kThreads, 0, st>>>(cg, mode, x, hx, n, partials);
  HPHI_CUDA_TRY(cudaGetLastError());
  return {};
}

Status launch_cg_fin(const CgDev& cg, int mode, const double* partials, int grid, int* clear, cudaStream_t st) {
  k_cg_fin<<<1, kThreads, 0, st>>>(cg, mode, partials, grid, clear);
  HPHI_CUDA_TRY(cudaGetLastError());
  return {};
}

}  // namespace hphi

// Lanczos exponential on flat FP64 vectors (Supplement, "Lanczos-based
// exponential method"), in three launches per Krylov step beside the apply:
//
//   lanczos_dots   h = Q^T w                                  (w = H q_k)
//   lanczos_orth   w <- w - Q h, then h2 = Q^T w and |w|^2    (second pass)
//   lanczos_next   q_{k+1} = (w - Q h2) / beta_k
//
// that is classical Gram-Schmidt, twice, against the whole basis; alpha_k is
// the component of the first pass along q_k, and beta_k^2 = |w|^2 - |h2|^2
// (Pythagoras: h2 is a rounding-size correction, and where it is not small
// beside |w| the breakdown test has fired).  The two-stage reductions end in
// the last CTA to arrive (an atomic ticket that wraps to zero), which sums the
// partials in a fixed order and does the scalar work: no finalising launches,
// same bits on every run.  After the last step that CTA also computes
// c = exp(t T) e_1 and normalises it: Q is orthonormal, so |sum_j c_j q_j| =
// |c|, and what rounding leaves of it the next exponential's |x| picks up.
//
// What bounds it: launches (a step was 12 of them, 30 us, most in one-warp
// finalising kernels) and the FP64 pipe, 2 multiply-adds per clock and SM:
// ~4 n (k + 1) of them per step, spread over all SMs.  A warp-wide FP64
// addition takes 64 clocks of a sub-partition, so the in-warp sums of V values
// exchange halves (V + 1 additions or fewer, not 5 V).
//
// Measured (beta-step, against 12 launches per Krylov step): 2x2 cluster
// D = 64 FP64 5.4 -> 3.1 ms, CL4x8 D = 256 FP64 162 -> 140 ms, D = 300 exact
// 217 -> 192 ms.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "tt_kernels.h"

namespace tt {

namespace {

constexpr int LT = 256;
constexpr int LW = LT / 32;
constexpr int LMAX = VEC_SUMS;  // values per partial record

// sums of a[0..V-1] over the warp: value i ends in every lane with
// lane >> (5 - log2 V) == i
template <int V>
__device__ __forceinline__ double warp_sums(double* a) {
  const int lane = threadIdx.x & 31;
  int off = 16;
#pragma unroll
  for (int half = V / 2; half >= 1; half >>= 1, off >>= 1) {
    const bool up = lane & off;
#pragma unroll
    for (int i = 0; i < V / 2; ++i)
      if (i < half) {
        const double send = up ? a[i] : a[i + half], keep = up ? a[i + half] : a[i];
        a[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
      }
  }
  double s = a[0];
  for (; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  return s;
}

__device__ __forceinline__ double warp_sum1(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <int V>
struct Log2 {
  static constexpr int v = 1 + Log2<V / 2>::v;
};
template <>
struct Log2<1> {
  static constexpr int v = 0;
};

// This CTA's sums of acc[0..V-1] (and of extra as value V when EXTRA) to
// partial[blockIdx.x * LMAX + .]; true in every thread of the last CTA.
template <int V, bool EXTRA>
__device__ __forceinline__ bool publish(double* acc, double extra, double* __restrict__ partial,
                                        unsigned* __restrict__ ticket) {
  __shared__ double red[LW][LMAX];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  constexpr int L = Log2<V>::v;
  const double s = warp_sums<V>(acc);
  if ((lane & ((32 >> L) - 1)) == 0) red[wp][lane >> (5 - L)] = s;
  if (EXTRA) {
    const double x = warp_sum1(extra);
    if (lane == 0) red[wp][V] = x;
  }
  __syncthreads();
  {  // the warps' sums: LW lanes per value
    constexpr int NV = V + (EXTRA ? 1 : 0);
    const int j = threadIdx.x / LW, q = threadIdx.x % LW;
    double t = j < NV ? red[q][j] : 0.0;
#pragma unroll
    for (int o = LW / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (j < NV && q == 0) {
      partial[blockIdx.x * LMAX + j] = t;
      __threadfence();
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// out[j] (shared, j < nv <= LMAX) = sum over the CTAs of partial[. * LMAX + j]
// in a fixed order: a warp per value
__device__ __forceinline__ void total(const double* __restrict__ partial, int nblk, int nv, double* out) {
  const int wp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int j = wp; j < nv; j += LW) {
    double s = 0.0;
    for (int b = lane; b < nblk; b += 32) s += __ldcg(&partial[b * LMAX + j]);
    s = warp_sum1(s);
    if (lane == 0) out[j] = s;
  }
  __syncthreads();
}

// x -> |x| (last CTA: a fresh KrylovState)
__global__ void __launch_bounds__(LT) lanczos_begin(const double* __restrict__ x, long long n,
                                                    double* __restrict__ partial, KrylovState* __restrict__ ks) {
  double acc[1] = {0.0};
  for (long long i = blockIdx.x * (long long)LT + threadIdx.x; i < n; i += (long long)gridDim.x * LT)
    acc[0] = fma(x[i], x[i], acc[0]);
  if (!publish<1, false>(acc, 0.0, partial, &ks->ticket)) return;
  __shared__ double s[1];
  total(partial, gridDim.x, 1, s);
  if (threadIdx.x < 17) {
    const int j = threadIdx.x;
    ks->alpha[j] = 0;
    ks->beta[j] = 0;
    ks->h[j] = 0;
    ks->h2[j] = 0;
    ks->c[j] = 0;
  }
  if (threadIdx.x == 0) {
    const double nb = sqrt(s[0]);
    ks->nb = nb;
    ks->hscale = 0.0;
    ks->resid = 0.0;
    ks->kdim = 0;
    ks->broken = 0;
    ks->bad = !isfinite(nb) ? 1 : 0;
  }
}

__global__ void __launch_bounds__(LT) lanczos_first(const double* __restrict__ x, long long n,
                                                    const KrylovState* __restrict__ ks, double* __restrict__ q0) {
  const double d = ks->nb;
  const double inv = d == 0.0 ? 0.0 : 1.0 / d;
  for (long long i = blockIdx.x * (long long)LT + threadIdx.x; i < n; i += (long long)gridDim.x * LT) q0[i] = x[i] * inv;
}

template <int V>
__global__ void __launch_bounds__(LT) lanczos_dots(const double* __restrict__ Q, long long ldq, int nv,
                                                   const double* __restrict__ w, long long n,
                                                   double* __restrict__ partial, KrylovState* __restrict__ ks) {
  double acc[V];
#pragma unroll
  for (int j = 0; j < V; ++j) acc[j] = 0.0;
  for (long long i = blockIdx.x * (long long)LT + threadIdx.x; i < n; i += (long long)gridDim.x * LT) {
    const double wi = w[i];
#pragma unroll
    for (int j = 0; j < V; ++j)
      if (j < nv) acc[j] = fma(Q[j * ldq + i], wi, acc[j]);
  }
  if (!publish<V, false>(acc, 0.0, partial, &ks->ticket)) return;
  __shared__ double s[LMAX];
  total(partial, gridDim.x, nv, s);
  if (threadIdx.x < nv) ks->h[threadIdx.x] = s[threadIdx.x];
}

// c = exp(t T) e_1 for the m x m tridiagonal T (m <= 16), by one CTA.  With
// nrm = ||t T||_1 <= 8: ceil(nrm) steps of the Taylor series of exp(M) v, M =
// t T / steps, one lane per entry (degree 18: remainder 1 / 19! < 2^-56); above
// that scaling and squaring of the matrix polynomial (Moler & Van Loan,
// "Nineteen dubious ways", method 3), whose cost grows with log nrm only.  The
// vector series takes ~4 us where the matrix form took 25.
__device__ void krylov_exp(const KrylovState* ks, double t, int m, double* c) {
  __shared__ double M[16][16], E[16][16], P[16][16];
  __shared__ double nrm_s;
  const int tid = threadIdx.x;
  if (tid < 32) {
    double col = 0.0;
    if (tid < m) {
      col = fabs(ks->alpha[tid]);
      if (tid > 0) col += fabs(ks->beta[tid - 1]);
      if (tid + 1 < m) col += fabs(ks->beta[tid]);
      col *= fabs(t);
    }
    for (int o = 16; o > 0; o >>= 1) col = fmax(col, __shfl_xor_sync(0xffffffffu, col, o));
    if (tid == 0) nrm_s = col;
  }
  __syncthreads();
  double nrm = nrm_s;
  if (nrm <= 8.0) {
    if (tid < 32) {
      const int steps = nrm > 1.0 ? (int)ceil(nrm) : 1;
      const double f = t / steps;
      const double a = tid < m ? f * ks->alpha[tid] : 0.0;
      const double bl = (tid > 0 && tid < m) ? f * ks->beta[tid - 1] : 0.0;
      const double bu = tid + 1 < m ? f * ks->beta[tid] : 0.0;
      double v = tid == 0 ? 1.0 : 0.0;
      for (int s = 0; s < steps; ++s) {
        double term = v;
#pragma unroll
        for (int p = 1; p <= 18; ++p) {
          const double lo = __shfl_up_sync(0xffffffffu, term, 1), hi = __shfl_down_sync(0xffffffffu, term, 1);
          const double x = fma(bl, lo, fma(bu, hi, a * term));
          term = x * (1.0 / p);
          v += term;
        }
      }
      if (tid < 17) c[tid] = tid < m ? v : 0.0;
    }
    __syncthreads();
    return;
  }
  const int i = tid / 16, j = tid % 16;
  int sq = 0;
  while (nrm > 0.25 && sq < 60) {
    nrm *= 0.5;
    ++sq;
  }
  double mij = 0.0;
  if (i < m && j < m) {
    if (i == j) mij = ks->alpha[i];
    else if (j == i + 1) mij = ks->beta[i];
    else if (i == j + 1) mij = ks->beta[j];
    mij *= ldexp(t, -sq);
  }
  M[i][j] = mij;
  E[i][j] = (i == j && i < m) ? 1.0 : 0.0;  // Horner: E = I + M/18, then E = I + M E / k
  __syncthreads();
  for (int k = 18; k >= 1; --k) {
    double acc = 0.0;
    for (int q = 0; q < m; ++q) acc = fma(M[i][q], E[q][j], acc);
    __syncthreads();
    E[i][j] = (i < m && j < m) ? ((i == j ? 1.0 : 0.0) + acc / (double)k) : 0.0;
    __syncthreads();
  }
  for (int r = 0; r < sq; ++r) {
    double acc = 0.0;
    for (int q = 0; q < m; ++q) acc = fma(E[i][q], E[q][j], acc);
    P[i][j] = acc;
    __syncthreads();
    E[i][j] = P[i][j];
    __syncthreads();
  }
  if (tid < 17) c[tid] = (tid < m) ? E[tid][0] : 0.0;
  __syncthreads();
}

// w <- w - Q h; h2 = Q^T w; beta_k and the breakdown test; after the last step
// (k = K - 1, beta_k is the residual norm) the coefficients of the result
template <int V>
__global__ void __launch_bounds__(LT) lanczos_orth(const double* __restrict__ Q, long long ldq, int k, int K,
                                                   double* __restrict__ w, long long n, double* __restrict__ partial,
                                                   KrylovState* __restrict__ ks, RhoScalars* __restrict__ rs, double tol,
                                                   double t) {
  const int nv = k + 1;
  __shared__ double h[LMAX];
  if (threadIdx.x < V) h[threadIdx.x] = threadIdx.x < nv ? ks->h[threadIdx.x] : 0.0;
  __syncthreads();
  double acc[V], ww = 0.0;
#pragma unroll
  for (int j = 0; j < V; ++j) acc[j] = 0.0;
  for (long long i = blockIdx.x * (long long)LT + threadIdx.x; i < n; i += (long long)gridDim.x * LT) {
    double q[V], v = w[i];
#pragma unroll
    for (int j = 0; j < V; ++j) q[j] = j < nv ? Q[j * ldq + i] : 0.0;
#pragma unroll
    for (int j = 0; j < V; ++j)
      if (j < nv) v = fma(-h[j], q[j], v);
    w[i] = v;
#pragma unroll
    for (int j = 0; j < V; ++j)
      if (j < nv) acc[j] = fma(q[j], v, acc[j]);
    ww = fma(v, v, ww);
  }
  if (!publish<V, true>(acc, ww, partial, &ks->ticket)) return;
  __shared__ double s[LMAX];
  total(partial, gridDim.x, V + 1, s);
  if (threadIdx.x < nv) ks->h2[threadIdx.x] = s[threadIdx.x];
  if (threadIdx.x == 0) {
    double b2 = s[V];
    for (int j = 0; j < nv; ++j) b2 = fma(-s[j], s[j], b2);
    if (ks->broken) {
      ks->beta[k] = 0.0;
    } else {
      const double a = ks->h[k], b = sqrt(b2 > 0.0 || !(b2 == b2) ? b2 : 0.0);
      ks->alpha[k] = a;
      if (!isfinite(b) || !isfinite(a)) ks->bad = 1;
      const double hs = fmax(ks->hscale, fabs(a) + b);
      ks->hscale = hs;
      ks->kdim = k + 1;
      // the residual norm (k = K - 1) is not part of T
      if (k < K - 1 && b <= tol * hs) {
        ks->broken = 1;
        ks->beta[k] = 0.0;
      } else {
        ks->beta[k] = b;
      }
    }
  }
  if (k < K - 1) return;
  __syncthreads();
  __shared__ double c[LMAX];
  const int m = ks->kdim;
  krylov_exp(ks, t, m, c);
  if (threadIdx.x == 0) {
    double c2 = 0.0;
    for (int j = 0; j < m; ++j) c2 = fma(c[j], c[j], c2);
    const double cn = sqrt(c2), nrm = ks->nb * cn;
    ks->nrm = nrm;
    const double resid = (!ks->broken && m == K) ? ks->nb * ks->beta[K - 1] * fabs(c[K - 1]) : 0.0;
    ks->resid = resid;
    const double inv = cn == 0.0 ? 0.0 : 1.0 / cn;
    for (int j = 0; j < m; ++j) ks->c[j] = c[j] * inv;
    if (!isfinite(nrm) || nrm == 0.0 || ks->bad) {
      rs->bad = 1;
    } else {
      rs->logscale += log(nrm);
      rs->resid_max = fmax(rs->resid_max, resid);
    }
  }
}

// q_{k+1} = (w - Q h2) / beta_k (zero after a breakdown)
template <int V>
__global__ void __launch_bounds__(LT) lanczos_next(const double* __restrict__ Q, long long ldq, int k,
                                                   const double* __restrict__ w, long long n,
                                                   const KrylovState* __restrict__ ks, double* __restrict__ qn) {
  const int nv = k + 1;
  __shared__ double h[LMAX];
  if (threadIdx.x < V) h[threadIdx.x] = threadIdx.x < nv ? ks->h2[threadIdx.x] : 0.0;
  const double d = ks->beta[k];
  const double inv = (ks->broken || d == 0.0) ? 0.0 : 1.0 / d;
  __syncthreads();
  for (long long i = blockIdx.x * (long long)LT + threadIdx.x; i < n; i += (long long)gridDim.x * LT) {
    double q[V], v = w[i];
#pragma unroll
    for (int j = 0; j < V; ++j) q[j] = j < nv ? Q[j * ldq + i] : 0.0;
#pragma unroll
    for (int j = 0; j < V; ++j)
      if (j < nv) v = fma(-h[j], q[j], v);
    qn[i] = v * inv;
  }
}

// y = sum_j c_j q_j (c normalised)
__global__ void __launch_bounds__(LT) lanczos_combine(const double* __restrict__ Q, long long ldq,
                                                      const KrylovState* __restrict__ ks, double* __restrict__ y,
                                                      long long n) {
  __shared__ double c[LMAX];
  __shared__ int m;
  if (threadIdx.x < LMAX) c[threadIdx.x] = ks->c[threadIdx.x];
  if (threadIdx.x == 0) m = ks->kdim;
  __syncthreads();
  for (long long i = blockIdx.x * (long long)LT + threadIdx.x; i < n; i += (long long)gridDim.x * LT) {
    double v = 0.0;
#pragma unroll 8
    for (int j = 0; j < m; ++j) v = fma(c[j], Q[(long long)j * ldq + i], v);
    y[i] = v;
  }
}

int lgrid(int64_t n) {
  const int64_t g = (n + LT - 1) / LT;
  return (int)(g > VEC_CTAS ? VEC_CTAS : (g < 1 ? 1 : g));
}

}  // namespace

cudaError_t k_lanczos_begin(const double* x, int64_t n, double* partial, KrylovState* ks, double* q0, cudaStream_t s) {
  lanczos_begin<<<lgrid(n), LT, 0, s>>>(x, n, partial, ks);
  lanczos_first<<<lgrid(n), LT, 0, s>>>(x, n, ks, q0);
  return cudaGetLastError();
}

cudaError_t k_lanczos_step(double* Q, int64_t ldq, int k, int K, double* w, int64_t n, double* partial, KrylovState* ks,
                           RhoScalars* rs, double tol, double t, cudaStream_t s) {
  if (k < 0 || k >= K || K > 16) return cudaErrorInvalidValue;
  const int g = lgrid(n), nv = k + 1;
  double* qn = k + 1 < K ? Q + (int64_t)(k + 1) * ldq : nullptr;
  auto run = [&](auto v) {
    constexpr int V = decltype(v)::value;
    lanczos_dots<V><<<g, LT, 0, s>>>(Q, ldq, nv, w, n, partial, ks);
    lanczos_orth<V><<<g, LT, 0, s>>>(Q, ldq, k, K, w, n, partial, ks, rs, tol, t);
    if (qn) lanczos_next<V><<<g, LT, 0, s>>>(Q, ldq, k, w, n, ks, qn);
  };
  if (nv <= 1) run(std::integral_constant<int, 1>{});
  else if (nv <= 2) run(std::integral_constant<int, 2>{});
  else if (nv <= 4) run(std::integral_constant<int, 4>{});
  else if (nv <= 8) run(std::integral_constant<int, 8>{});
  else run(std::integral_constant<int, 16>{});
  return cudaGetLastError();
}

cudaError_t k_lanczos_end(const double* Q, int64_t ldq, const KrylovState* ks, double* y, int64_t n, cudaStream_t s) {
  lanczos_combine<<<lgrid(n), LT, 0, s>>>(Q, ldq, ks, y, n);
  return cudaGetLastError();
}

}  // namespace tt

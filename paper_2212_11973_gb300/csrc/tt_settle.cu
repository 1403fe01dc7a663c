// The arithmetic in which a padded state settles: Lanczos steps, Cholesky factors
// and the digit gather of the first beta-step after a padding.
//
// tt_rho_pad adds directions of weight zero.  The first beta-step gives them
// weight, but far fewer at a time than a bond gains: on the way through the chain
// the columns of a sector span 1 down to 1e-120, and from some 1e-16 of each
// other on they are linearly dependent, so that the directions completing the
// basis are what the rounding of all earlier operations left there.  1-TDVP keeps
// that basis, and the energies of the following steps depend on it by up to 5e-6
// (2x8 ladders of D = 64 to 128): as much as on a change of precision, and any
// change of the order of an FP64 sum makes another choice.  After the step no
// sector is deficient (sigma_min / sigma_max above 1e-10), and another order of
// the sums no longer matters (1e-15 in FP64, 3e-8 in split-BF16 x6 over five
// steps).
//
// So up to the end of that step every operation keeps one order of its sums, which
// does not change with the kernels of the later steps:
//   FP64 GEMM      one accumulator per output, ascending K (the one-warp tiles of
//                  tt_gemm64.cu: m8n8k4 is four fused multiply-adds in order)
//   Lanczos        three-term step, two Gram-Schmidt passes (here)
//   CholeskyQR     double-float products in the mixed modes, factor and inverse
//                  row by row (here)
//   split-BF16     level by level over 64 of K, no shared tiles (tt_tcgen05p.cu)
//   digits         rounded from the top level down (tt_fixed.h), no shared tiles,
//                  the gather's two-float sums as compiled here
//   hi + lo        rounded as an FP64 addition
// A state that is padded as tt_rho_create made it is made again in this order
// (45 ms a 2x8 ladder).  Growth keeps the later steps' kernels: two-site steps
// choose their bonds anew.
//
// It runs once per padding and is not captured; launches and idle SMs are not what
// these kernels were written against.  First step of six 2x8 ladders, D = 64 to
// 128, with plans and allocations: FP64 235 ms without it, 350 with it; split-BF16
// x6 390 and 460; exact split 410 and 470.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "tt_df.h"
#include "tt_fixed.h"
#include "tt_kernels.h"

namespace tt {

namespace {

constexpr int VT = 256;

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// this CTA's sum of acc to partial[blockIdx.x * VEC_SUMS]
__device__ __forceinline__ void publish(double acc, double* __restrict__ partial) {
  __shared__ double red[VT / 32];
  const double s = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < VT / 32; ++q) t += red[q];
    partial[blockIdx.x * VEC_SUMS] = t;
  }
}

// out[j] = sum_b partial[b * VEC_SUMS + j], by one warp
__device__ void finalize_sums(const double* partial, int nblk, int nv, double* out) {
  const int lane = threadIdx.x & 31;
  for (int j = 0; j < nv; ++j) {
    double s = 0.0;
    for (int b = lane; b < nblk; b += 32) s += partial[b * VEC_SUMS + j];
    s = warp_sum(s);
    if (lane == 0) out[j] = s;
  }
}

__global__ void sumsq_kernel(const double* __restrict__ v, long long n, double* __restrict__ partial) {
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)VT + threadIdx.x; i < n; i += (long long)gridDim.x * VT)
    acc = fma(v[i], v[i], acc);
  publish(acc, partial);
}

__global__ void norm_init_finalize(const double* partial, int nblk, KrylovState* ks) {
  __shared__ double s;
  finalize_sums(partial, nblk, 1, &s);
  __syncwarp();
  if (threadIdx.x == 0) {
    double nb = sqrt(s);
    ks->nb = nb;
    ks->hscale = 0.0;
    ks->resid = 0.0;
    ks->kdim = 0;
    ks->broken = 0;
    ks->bad = !isfinite(nb) ? 1 : 0;
    for (int j = 0; j < 17; ++j) { ks->alpha[j] = 0; ks->beta[j] = 0; ks->h[j] = 0; ks->c[j] = 0; }
  }
}

__global__ void scale_kernel(const double* __restrict__ v, long long n, const double* __restrict__ denom,
                             const int* __restrict__ dead, double* __restrict__ out) {
  const double d = *denom;
  const bool z = (dead && *dead) || d == 0.0;
  const double inv = z ? 0.0 : 1.0 / d;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[i] = v[i] * inv;
}

template <int MAXV>
__global__ void __launch_bounds__(VT) multidot_kernel(const double* __restrict__ Q, long long ldq, int j0, int nv,
                                                      const double* __restrict__ w, long long n,
                                                      double* __restrict__ partial) {
  double acc[MAXV];
#pragma unroll
  for (int j = 0; j < MAXV; ++j) acc[j] = 0.0;
  for (long long i = blockIdx.x * (long long)VT + threadIdx.x; i < n; i += (long long)gridDim.x * VT) {
    double wi = w[i];
#pragma unroll
    for (int j = 0; j < MAXV; ++j)
      if (j < nv) acc[j] = fma(Q[(long long)(j0 + j) * ldq + i], wi, acc[j]);
  }
  __shared__ double red[VT / 32][MAXV];
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
#pragma unroll
  for (int j = 0; j < MAXV; ++j) {
    double v = warp_sum(acc[j]);
    if (lane == 0) red[wp][j] = v;
  }
  __syncthreads();
  if (threadIdx.x < nv) {
    double s = 0.0;
    for (int q = 0; q < VT / 32; ++q) s += red[q][threadIdx.x];
    partial[blockIdx.x * VEC_SUMS + threadIdx.x] = s;
  }
}

__global__ void alpha_finalize(const double* partial, int nblk, int k, KrylovState* ks) {
  __shared__ double s;
  finalize_sums(partial, nblk, 1, &s);
  __syncwarp();
  if (threadIdx.x == 0 && !ks->broken) ks->alpha[k] = s;
}

__global__ void three_term_kernel(const double* __restrict__ Q, long long ldq, int k, double* __restrict__ w,
                                  long long n, const KrylovState* __restrict__ ks) {
  const double a = ks->alpha[k];
  const double b = (k > 0) ? ks->beta[k - 1] : 0.0;
  const double* qk = Q + (long long)k * ldq;
  const double* qp = Q + (long long)(k > 0 ? k - 1 : 0) * ldq;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    double v = w[i] - a * qk[i];
    if (k > 0) v -= b * qp[i];
    w[i] = v;
  }
}

__global__ void h_finalize(const double* partial, int nblk, int nv, KrylovState* ks) {
  finalize_sums(partial, nblk, nv, ks->h);
}

// w -= sum_j h_j Q_j ; optional partial ||w||^2
__global__ void __launch_bounds__(VT) axpy_multi_kernel(const double* __restrict__ Q, long long ldq, int nv,
                                                        const KrylovState* __restrict__ ks, double* __restrict__ w,
                                                        long long n, double* __restrict__ partial) {
  __shared__ double h[17];
  if (threadIdx.x < 17) h[threadIdx.x] = ks->h[threadIdx.x];
  __syncthreads();
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)VT + threadIdx.x; i < n; i += (long long)gridDim.x * VT) {
    double v = w[i];
    for (int j = 0; j < nv; ++j) v -= h[j] * Q[(long long)j * ldq + i];
    w[i] = v;
    acc = fma(v, v, acc);
  }
  if (partial) publish(acc, partial);
}

// beta_k = ||w||; breakdown test; stores beta (or 0 if broken)
__global__ void beta_finalize(const double* partial, int nblk, int k, int K, double tol, KrylovState* ks) {
  __shared__ double s;
  finalize_sums(partial, nblk, 1, &s);
  __syncwarp();
  if (threadIdx.x != 0) return;
  if (ks->broken) {
    ks->beta[k] = 0.0;
    return;
  }
  double b = sqrt(s);
  if (!isfinite(b) || !isfinite(ks->alpha[k])) ks->bad = 1;
  double hs = fmax(ks->hscale, fabs(ks->alpha[k]) + b);
  ks->hscale = hs;
  ks->kdim = k + 1;
  if (k == K - 1) {
    ks->beta[k] = b;  // residual norm, not part of T
    return;
  }
  if (b <= tol * hs) {
    ks->broken = 1;
    ks->beta[k] = 0.0;
    return;
  }
  ks->beta[k] = b;
}

// c = exp(t T) e_1 for the kdim x kdim tridiagonal T, by scaling and squaring
// with a degree-18 Taylor polynomial (Moler & Van Loan, "Nineteen dubious
// ways", method 3): M = t T / 2^s with ||M||_1 <= 1/4, E = sum_k M^k / k!
// (Horner), then E <- E^2 s times.  One thread per matrix entry (kdim <= 16).
__global__ void __launch_bounds__(256) krylov_exp_kernel(KrylovState* ks, double t, int K) {
  __shared__ double M[16][16], E[16][16], P[16][16];
  __shared__ int m_s, s_s;
  const int tid = threadIdx.x, i = tid / 16, j = tid % 16;
  if (tid == 0) {
    const int m = ks->kdim;
    double nrm = 0.0;  // ||t T||_1 (T symmetric tridiagonal)
    for (int c = 0; c < m; ++c) {
      double col = fabs(ks->alpha[c]);
      if (c > 0) col += fabs(ks->beta[c - 1]);
      if (c + 1 < m) col += fabs(ks->beta[c]);
      nrm = fmax(nrm, fabs(t) * col);
    }
    int sq = 0;
    while (nrm > 0.25 && sq < 60) { nrm *= 0.5; ++sq; }
    m_s = m;
    s_s = sq;
  }
  __syncthreads();
  const int m = m_s, sq = s_s;
  const double scale = ldexp(t, -sq);
  double mij = 0.0;
  if (i < m && j < m) {
    if (i == j) mij = ks->alpha[i];
    else if (j == i + 1) mij = ks->beta[i];
    else if (i == j + 1) mij = ks->beta[j];
    mij *= scale;
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
  if (tid < 17) ks->c[tid] = (tid < m) ? E[tid][0] : 0.0;
  if (tid == 0) ks->resid = (!ks->broken && m == K) ? ks->nb * ks->beta[K - 1] * fabs(E[K - 1][0]) : 0.0;
}

__global__ void __launch_bounds__(VT) combine_kernel(const double* __restrict__ Q, long long ldq,
                                                     const KrylovState* __restrict__ ks, double* __restrict__ y,
                                                     long long n, double* __restrict__ partial) {
  __shared__ double c[17];
  __shared__ int m;
  if (threadIdx.x < 17) c[threadIdx.x] = ks->c[threadIdx.x] * ks->nb;
  if (threadIdx.x == 0) m = ks->kdim;
  __syncthreads();
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)VT + threadIdx.x; i < n; i += (long long)gridDim.x * VT) {
    double v = 0.0;
    for (int j = 0; j < m; ++j) v = fma(c[j], Q[(long long)j * ldq + i], v);
    y[i] = v;
    acc = fma(v, v, acc);
  }
  publish(acc, partial);
}

__global__ void nrm_finalize(const double* partial, int nblk, KrylovState* ks, RhoScalars* rs) {
  __shared__ double s;
  finalize_sums(partial, nblk, 1, &s);
  __syncwarp();
  if (threadIdx.x != 0) return;
  double nrm = sqrt(s);
  ks->nrm = nrm;
  if (!isfinite(nrm) || nrm == 0.0 || ks->bad) {
    rs->bad = 1;
    return;
  }
  rs->logscale += log(nrm);
  rs->resid_max = fmax(rs->resid_max, ks->resid);
}

// ---------------------------------------------------------------------------
// Cholesky G = R^T R (G the sum of the job's partial Gram matrices) and R^-1, one
// CTA per job, right-looking row by row; CholJob::shift as in tt_chol.cu.  The
// upper triangle is packed row by row in shared memory, or for n > ROWS_SMEM_MAXN
// in the job's workspace scratch.
// ---------------------------------------------------------------------------
constexpr int ROWS_SMEM_MAXN = 230;
constexpr int ROWS_T = 512;

__device__ __forceinline__ int pk(int i, int j, int n) { return i * n - (i * (i - 1)) / 2 + (j - i); }

struct RowsF64 {
  using T = double;
  static constexpr double u = 1.1102230246251565e-16;  // unit roundoff 2^-53
  static __device__ __forceinline__ T of(double x) { return x; }
  static __device__ __forceinline__ double dbl(T a) { return a; }
  static __device__ __forceinline__ T zero() { return 0.0; }
  static __device__ __forceinline__ T add(T a, double v) { return a + v; }
  // |a - target| (a test against a threshold)
  static __device__ __forceinline__ double dev(T a, double target) { return fabs(a - target); }
  // a - b c
  static __device__ __forceinline__ T fnms(T a, T b, T c) { return fma(-b, c, a); }
  static __device__ __forceinline__ T mul(T a, T b) { return a * b; }
};

struct RowsDF {
  using T = float2;  // value x + y, |y| <= ulp(x) / 2
  static constexpr double u = 1.4210854715202004e-14;  // 2^-46
  static __device__ __forceinline__ T of(double v) { return df_split(v); }
  static __device__ __forceinline__ double dbl(T a) { return dbl_of_float(a.x) + dbl_of_float(a.y); }
  static __device__ __forceinline__ T zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ T two_sum(float s, float t) {
    const float h = s + t;
    const float bp = h - s;
    return make_float2(h, (s - (h - bp)) + (t - bp));
  }
  static __device__ __forceinline__ T add(T a, double v) {
    const float2 b = df_split(v);
    const float s = a.x + b.x;
    const float bp = s - a.x;
    const float t = ((a.x - (s - bp)) + (b.x - bp)) + (a.y + b.y);
    return two_sum(s, t);
  }
  static __device__ __forceinline__ double dev(T a, double target) {
    return (double)fabsf((a.x - (float)target) + a.y);
  }
  static __device__ __forceinline__ T fnms(T a, T b, T c) {
    const float p = b.x * c.x;
    float e = fmaf(b.x, c.x, -p);  // b.x c.x = p + e exactly
    e = fmaf(b.x, c.y, e);
    e = fmaf(b.y, c.x, e);
    const float s = a.x - p;       // a.x - p = s + t exactly
    const float bp = s - a.x;
    float t = (a.x - (s - bp)) + (-p - bp);
    t += a.y - e;
    return two_sum(s, t);
  }
  static __device__ __forceinline__ T mul(T a, T b) {
    const float p = a.x * b.x;
    float e = fmaf(a.x, b.x, -p);
    e = fmaf(a.x, b.y, e);
    e = fmaf(a.y, b.x, e);
    return two_sum(p, e);
  }
};

template <class A>
__global__ void __launch_bounds__(ROWS_T, 1) chol_rows_kernel(const CholJob* __restrict__ jobs, double* __restrict__ ws,
                                                              int* __restrict__ fail) {
  using T = typename A::T;
  extern __shared__ __align__(16) unsigned char rows_raw[];
  const CholJob J = jobs[blockIdx.x];
  const int n = J.n;
  T* sm = n <= ROWS_SMEM_MAXN ? reinterpret_cast<T*>(rows_raw) : reinterpret_cast<T*>(ws + J.pk);
  if (J.shift == 3) {
    if (threadIdx.x == 0) fail[J.sec] = 1;
    return;
  }
  if (fail[J.sec]) return;
  double* G = ws + J.g;
  double* R = ws + J.r;
  double* Ri = ws + J.ri;
  const long long nn = (long long)n * n;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = blockDim.x >> 5;
  __shared__ double red[ROWS_T / 32];
  __shared__ T piv_t, ipiv_t;  // the current pivot and its reciprocal
  __shared__ int bad;
  for (int i = warp; i < n; i += nw)
    for (int j = i + lane; j < n; j += 32) {
      const long long e = (long long)i * n + j;
      T acc = A::of(G[e]);
      for (int s = 1; s < J.parts; ++s) acc = A::add(acc, G[s * nn + e]);
      sm[pk(i, j, n)] = acc;
    }
  __syncthreads();
  if (J.shift == 2) {
    double mx = 0.0;
    for (int i = warp; i < n; i += nw)
      for (int j = i + lane; j < n; j += 32) {
        const double dev = A::dev(sm[pk(i, j, n)], i == j ? 1.0 : 0.0);
        mx = (dev <= mx) ? mx : (dev == dev ? dev : 1e300);
      }
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) red[warp] = mx;
    __syncthreads();
    double all = 0.0;
    for (int q = 0; q < nw; ++q) all = fmax(all, red[q]);
    if (!(all <= 1e-3)) {
      if (tid == 0) fail[J.sec] = 1;
      return;
    }
    if ((double)n * all <= 1e-8) {
      for (int i = warp; i < n; i += nw)
        for (int j = lane; j < n; j += 32) {
          const long long e = (long long)i * n + j;
          if (j < i) {
            R[e] = 0.0;
            Ri[e] = 0.0;
          } else if (j == i) {
            const double h = 0.5 * (A::dbl(sm[pk(i, i, n)]) - 1.0);
            R[e] = 1.0 + h;
            Ri[e] = 1.0 - h;
          } else {
            const double g = A::dbl(sm[pk(i, j, n)]);
            R[e] = g;
            Ri[e] = -g;
          }
        }
      return;
    }
  }
  if (tid == 0) {
    bad = 0;
    if (J.shift == 1) {
      double tr = 0.0;
      for (int i = 0; i < n; ++i) tr += A::dbl(sm[pk(i, i, n)]);
      const double sft = 11.0 * ((double)J.m * n + (double)n * (n + 1)) * A::u * tr;
      for (int i = 0; i < n; ++i) sm[pk(i, i, n)] = A::of(A::dbl(sm[pk(i, i, n)]) + sft);
    }
  }
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    if (tid == 0) {
      const double d = A::dbl(sm[pk(k, k, n)]);
      if (!(d > 0.0) || !isfinite(d)) {
        bad = 1;
        fail[J.sec] = 1;
      }
      const double p = bad ? 1.0 : sqrt(d);
      piv_t = A::of(p);
      ipiv_t = A::of(1.0 / p);
    }
    __syncthreads();
    if (bad) return;
    for (int j = k + tid; j < n; j += blockDim.x) sm[pk(k, j, n)] = j == k ? piv_t : A::mul(sm[pk(k, j, n)], ipiv_t);
    __syncthreads();
    for (int i = k + 1 + warp; i < n; i += nw) {
      const T rki = sm[pk(k, i, n)];
      for (int j = i + lane; j < n; j += 32) sm[pk(i, j, n)] = A::fnms(sm[pk(i, j, n)], rki, sm[pk(k, j, n)]);
    }
    __syncthreads();
  }
  for (int i = warp; i < n; i += nw)
    for (int j = lane; j < n; j += 32) R[(long long)i * n + j] = (j >= i) ? A::dbl(sm[pk(i, j, n)]) : 0.0;
  // in-place inverse, rows from the bottom
  for (int k = n - 1; k >= 0; --k) {
    __syncthreads();
    if (tid == 0) ipiv_t = A::of(1.0 / A::dbl(sm[pk(k, k, n)]));
    __syncthreads();
    for (int c = k + tid; c < n; c += blockDim.x) sm[pk(k, c, n)] = c == k ? ipiv_t : A::mul(sm[pk(k, c, n)], ipiv_t);
    __syncthreads();
    for (int i = warp; i < k; i += nw) {
      const T rik = sm[pk(i, k, n)];
      __syncwarp();
      for (int c = k + lane; c < n; c += 32)
        sm[pk(i, c, n)] = A::fnms(c == k ? A::zero() : sm[pk(i, c, n)], rik, sm[pk(k, c, n)]);
    }
  }
  __syncthreads();
  for (int i = warp; i < n; i += nw)
    for (int j = lane; j < n; j += 32) Ri[(long long)i * n + j] = (j >= i) ? A::dbl(sm[pk(i, j, n)]) : 0.0;
}

// ---------------------------------------------------------------------------
// W-gather of the exact path (gather_digits_kernel of tt_digits.cu), one row of a
// warp and one term at a time.  The compiler's choice of fused multiply-adds in the
// two-float sums is part of the fixed arithmetic, and it goes with this text.
// ---------------------------------------------------------------------------
constexpr int ROWS_MAXC = 256, ROWS_MAXK = 64;

__device__ __forceinline__ int slot_of(Ref r) { return (int)(r >> 56); }
__device__ __forceinline__ long long off_of(Ref r) { return (long long)(r & 0x00FFFFFFFFFFFFFFull); }

__global__ void __launch_bounds__(VT) gather_digits_rows_kernel(const GItem* __restrict__ items,
                                                           const GContrib* __restrict__ cs, Bases bs) {
  const GItem it = items[blockIdx.x];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int lg = 0;
  while ((1 << lg) < 32 && 2 * (1 << lg) < it.cols) ++lg;
  const int G = 1 << lg, rpw = 32 >> lg;
  const int sub = lane >> lg, gl = lane & (G - 1);
  uint32_t* dst = reinterpret_cast<uint32_t*>(reinterpret_cast<__nv_bfloat16*>(sel_base(bs, slot_of(it.dst))) +
                                              off_of(it.dst));
  short* ex = reinterpret_cast<short*>(sel_base(bs, slot_of(it.e))) + off_of(it.e);
  const long long lo2 = sel_lo(bs, slot_of(it.dst)) / 2;  // level stride in BF16 pairs
  constexpr int PP = ROWS_MAXC / 64;                      // column pairs per lane at G = 32
  // the item's MPO coefficients as float pairs, split once per CTA (FP64
  // arithmetic runs at ~1/64 of FP32 on GB300)
  __shared__ float2 cf[ROWS_MAXK];
  // the host rejects items with more terms; the clamp keeps the table in bounds
  const int nk = min(it.c1 - it.c0, ROWS_MAXK);
  for (int k = threadIdx.x; k < nk; k += VT) {
    const double v = cs[it.c0 + k].coef;
    const float ch = (float)v;
    cf[k] = make_float2(ch, (float)(v - (double)ch));
  }
  __syncthreads();
  for (int r0 = it.r0 + warp * rpw; r0 < it.rows; r0 += (VT / 32) * rpw) {
    const int r = r0 + sub;
    const bool rin = r < it.rows;
    float h[2 * PP], l[2 * PP];
#pragma unroll
    for (int i = 0; i < 2 * PP; ++i) { h[i] = 0.f; l[i] = 0.f; }
    for (int k = it.c0; k < it.c0 + nk; ++k) {
      const GContrib cb = cs[k];
      const float ch = cf[k - it.c0].x, cl = cf[k - it.c0].y;
      const float2* s = reinterpret_cast<const float2*>(sel_base(bs, slot_of(cb.src))) + off_of(cb.src) +
                        (long long)r * cb.src_rs;
      const bool al16 = (reinterpret_cast<uintptr_t>(s) & 15) == 0;
#pragma unroll
      for (int i = 0; i < PP; ++i) {
        const int c = 2 * (gl + G * i);
        if (rin && c < it.cols) {
          float4 v;
          if (al16 && c + 1 < it.cols) {
            v = *reinterpret_cast<const float4*>(s + c);
          } else {
            const float2 v0 = s[c];
            const float2 v1 = c + 1 < it.cols ? s[c + 1] : make_float2(0.f, 0.f);
            v = make_float4(v0.x, v0.y, v1.x, v1.y);
          }
          df_fma(h[2 * i], l[2 * i], ch, cl, v.x, v.y);
          df_fma(h[2 * i + 1], l[2 * i + 1], ch, cl, v.z, v.w);
        }
      }
    }
    // renormalise every pair (TwoSum of h and l): after cancellation l may be
    // as large as h, and the digits below are taken from h and l separately
#pragma unroll
    for (int i = 0; i < 2 * PP; ++i) {
      const float sv = h[i] + l[i];
      const float bp = sv - h[i];
      l[i] = (h[i] - (sv - bp)) + (l[i] - bp);
      h[i] = sv;
    }
    int m = 0;
#pragma unroll
    for (int i = 0; i < PP; ++i) {
      const int c = 2 * (gl + G * i);
      if (c < it.cols) m = max(m, fexp(h[2 * i]));
      if (c + 1 < it.cols) m = max(m, fexp(h[2 * i + 1]));
    }
    for (int o = G >> 1; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    // one exponent above the largest: |h + l| < 2^(m - 1023), so the scaled
    // values stay below 2^31 also after rounding
    if (m) m = m + 1;
    // scale 2^(1054 - m) as two exact power-of-two factors in the FP32 range
    const int sh = m ? 1054 - m : 0, sa = sh / 2, sb = sh - sa;
    const float fa = p2f(sa), fb = p2f(sb);
    if (rin) {
      uint32_t* drow = dst + ((long long)r * it.dst_rs >> 1);
#pragma unroll
      for (int i = 0; i < PP; ++i) {
        const int c = 2 * (gl + G * i);
        if (c < it.cols) {
          uint32_t d0[4], d1[4] = {0u, 0u, 0u, 0u};
          digits_of_pair((h[2 * i] * fa) * fb, (l[2 * i] * fa) * fb, d0);
          if (c + 1 < it.cols) digits_of_pair((h[2 * i + 1] * fa) * fb, (l[2 * i + 1] * fa) * fb, d1);
#pragma unroll
          for (int lv = 0; lv < 4; ++lv) drow[lv * lo2 + (c >> 1)] = __byte_perm(d0[lv], d1[lv], 0x7632);
        }
      }
      if (gl == 0) ex[(long long)r * it.e_rs] = (short)m;
    }
  }
}

int grid_for(long long n) {
  const long long g = (n + VT - 1) / VT;
  return (int)(g > VEC_CTAS ? VEC_CTAS : (g < 1 ? 1 : g));
}

}  // namespace

cudaError_t k_settle_begin(const double* x, int64_t n, double* partial, KrylovState* ks, double* q0, cudaStream_t s) {
  const int g = grid_for(n);
  sumsq_kernel<<<g, VT, 0, s>>>(x, n, partial);
  norm_init_finalize<<<1, 32, 0, s>>>(partial, g, ks);
  scale_kernel<<<g, VT, 0, s>>>(x, n, &ks->nb, nullptr, q0);
  return cudaGetLastError();
}

cudaError_t k_settle_step(double* Q, int64_t ldq, int k, int K, double* w, int64_t n, double* partial, KrylovState* ks,
                          double tol, cudaStream_t s) {
  if (k < 0 || k >= K || K > 16) return cudaErrorInvalidValue;
  const int g = grid_for(n), nv = k + 1;
  multidot_kernel<1><<<g, VT, 0, s>>>(Q, ldq, k, 1, w, n, partial);
  alpha_finalize<<<1, 32, 0, s>>>(partial, g, k, ks);
  three_term_kernel<<<g, VT, 0, s>>>(Q, ldq, k, w, n, ks);
  for (int pass = 0; pass < 2; ++pass) {
    if (nv <= 4) multidot_kernel<4><<<g, VT, 0, s>>>(Q, ldq, 0, nv, w, n, partial);
    else if (nv <= 8) multidot_kernel<8><<<g, VT, 0, s>>>(Q, ldq, 0, nv, w, n, partial);
    else multidot_kernel<17><<<g, VT, 0, s>>>(Q, ldq, 0, nv, w, n, partial);
    h_finalize<<<1, 32, 0, s>>>(partial, g, nv, ks);
    axpy_multi_kernel<<<g, VT, 0, s>>>(Q, ldq, nv, ks, w, n, pass ? partial : nullptr);
  }
  beta_finalize<<<1, 32, 0, s>>>(partial, g, k, K, tol, ks);
  if (k + 1 < K) scale_kernel<<<g, VT, 0, s>>>(w, n, &ks->beta[k], &ks->broken, Q + (int64_t)(k + 1) * ldq);
  return cudaGetLastError();
}

cudaError_t k_settle_end(const double* Q, int64_t ldq, KrylovState* ks, double t, int K, double* y, int64_t n,
                         double* partial, RhoScalars* rs, cudaStream_t s) {
  const int g = grid_for(n);
  krylov_exp_kernel<<<1, 256, 0, s>>>(ks, t, K);
  combine_kernel<<<g, VT, 0, s>>>(Q, ldq, ks, y, n, partial);
  nrm_finalize<<<1, 32, 0, s>>>(partial, g, ks, rs);
  scale_kernel<<<g, VT, 0, s>>>(y, n, &ks->nrm, nullptr, y);
  return cudaGetLastError();
}

cudaError_t launch_gather_digits_rows(const DevGather& g, const Bases& b, cudaStream_t s) {
  if (g.nitems == 0) return cudaSuccess;
  gather_digits_rows_kernel<<<g.nitems, VT, 0, s>>>(g.items, g.contribs, b);
  return cudaGetLastError();
}

cudaError_t launch_chol_rows(const CholJob* jobs, int njobs, double* ws, int* fail, cudaStream_t s, int maxn, bool df) {
  if (njobs == 0) return cudaSuccess;
  const int ns = maxn < ROWS_SMEM_MAXN ? maxn : ROWS_SMEM_MAXN;
  const size_t smem = ((size_t)ns * (ns + 1) / 2) * 8;
  auto run = [&](auto kernel) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<njobs, ROWS_T, smem, s>>>(jobs, ws, fail);
    return cudaGetLastError();
  };
  return df ? run(chol_rows_kernel<RowsDF>) : run(chol_rows_kernel<RowsF64>);
}

}  // namespace tt

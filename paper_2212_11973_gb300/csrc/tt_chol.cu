// Cholesky factor and triangular inverse of the CholeskyQR gauge, one CTA per
// sector.
//
// G = R^T R (R upper; G the sum of the job's partial Gram matrices, row-major
// n x n at ws + g) and R^-1.  Optional diagonal shift s = 11 (m n + n (n + 1)) u
// tr(G) (shifted CholeskyQR, Fukaya, Kannan, Nakatsukasa, Yamamoto, Yanagisawa
// 2020).  A non-positive or non-finite pivot marks fail[sec] and leaves the job
// to the Householder fallback.
//
// The upper triangle is packed row by row (row i holds columns i..n-1) in shared
// memory, or for sectors too large for it in the job's workspace scratch, and
// factorised and then inverted in place in blocks of NB = 8 rows:
//   factor, from the top:    one warp factorises the diagonal block in registers
//     (two columns of a row per lane) and inverts it; a thread per column solves the
//     block row; every warp updates trailing rows with all 8 pivot rows at once;
//   inverse, from the bottom (S holds - sum R X): block row X = D S with the
//     diagonal block's inverse D, then every row above takes its rank-8 update,
//     with the block's columns of R copied aside first.
//
// Element arithmetic: FP64, or double-float (~2^-46 relative) on the FP32 pipe.
//
// What bounds it: the chain of n pivots on one CTA.  Row by row (one pivot with
// a square root and a division in FP64, three barriers and a pass over the
// trailing triangle each) a step took ~2.8 us; in blocks of 8 a pivot's scalar
// is a float rsqrt and one third-order correction (~1000 clocks with the exchange
// of its row), there are 4 barriers per 8 rows, the next diagonal block is factorised
// while the trailing triangle is updated, and a trailing element is loaded and
// stored once per 8 multiply-adds whose other operands sit in registers or are
// one broadcast load.  Measured, double-float, one sector with its partial
// matrices: n = 180 1018 -> 448 us, n = 53 154 -> 70 us; n = 53 in FP64 117 us.
// Normalising the pairs after each of a block's 8 terms (df_tidy) costs 6 % of that:
// 113 -> 119 ms of a width-6 x 12 beta-step at D = 1024.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "tt_df.h"
#include "tt_kernels.h"

namespace tt {

namespace {

constexpr int CHOL_T = 512, CHOL_W = CHOL_T / 32, NB = 8;
constexpr size_t CHOL_SMEM = 226 * 1024;

// elements of a job's packed triangle, to a 16-byte boundary, and the largest n whose
// triangle and n x 8 copies fit shared memory together (232)
__host__ __device__ constexpr int tri_elems(int n) { return (n * (n + 1) / 2 + 1) & ~1; }
constexpr size_t chol_bytes(int n) { return ((size_t)tri_elems(n) + (size_t)NB * n) * 8; }
constexpr int chol_max_n() {
  int n = 0;
  while (chol_bytes(n + 1) <= CHOL_SMEM) ++n;
  return n;
}
constexpr int CHOL_MAXN = chol_max_n();

__device__ __forceinline__ int pk(int i, int j, int n) { return i * n - (i * (i - 1)) / 2 + (j - i); }

struct CholF64 {
  using T = double;
  using D = double;  // |a - target|
  using Acc = double;
  static constexpr double u = 1.1102230246251565e-16;  // unit roundoff 2^-53
  static __device__ __forceinline__ T of(double x) { return x; }
  static __device__ __forceinline__ double dbl(T a) { return a; }
  static __device__ __forceinline__ T zero() { return 0.0; }
  static __device__ __forceinline__ T neg(T a) { return -a; }
  static __device__ __forceinline__ T add(T a, double v) { return a + v; }
  static __device__ __forceinline__ D dev(T a, double target) { return fabs(a - target); }
  static __device__ __forceinline__ T mul(T a, T b) { return a * b; }
  static __device__ __forceinline__ bool positive(T a) { return a > 0.0 && isfinite(a); }
  static __device__ __forceinline__ T shfl(T a, int l) { return __shfl_sync(0xffffffffu, a, l); }
  // a - b c, accumulated
  static __device__ __forceinline__ Acc open(T a) { return a; }
  static __device__ __forceinline__ void fnms(Acc& a, T b, T c) { a = fma(-b, c, a); }
  static __device__ __forceinline__ void tidy(Acc&) {}
  static __device__ __forceinline__ T close(Acc a) { return a; }
  // 1 / sqrt(d): float seed y of the mantissa's (1 - d y^2 = e below 2^-21),
  // y (1 + e/2 + 3 e^2 / 8) leaves ~e^3
  static __device__ __forceinline__ T rsqrt(T d) {
    const int ex = ((__double2hiint(d) >> 20) & 0x7FF) - 1023;
    if (ex == -1023) return 1.0 / sqrt(d);  // subnormal
    const int h = ex >> 1;
    const double dn = __hiloint2double(__double2hiint(d) - 2 * h * (1 << 20), __double2loint(d));  // in [1, 4)
    const double y = (double)rsqrtf((float)dn);
    const double e = fma(-(dn * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y) * __hiloint2double((1023 - h) << 20, 0);
  }
  static __device__ __forceinline__ T sqrt_of(T d, T) { return sqrt(d); }
};

struct CholDF {
  using T = float2;  // value x + y, |y| <= ulp(x) / 2
  using D = float;
  using Acc = float2;  // not normalised between fnms and tidy or close
  static constexpr double u = 1.4210854715202004e-14;  // 2^-46
  static __device__ __forceinline__ T of(double v) { return df_split(v); }
  // one FP64 addition (the conversions are integer operations)
  static __device__ __forceinline__ double dbl(T a) { return dbl_of_float(a.x) + dbl_of_float(a.y); }
  static __device__ __forceinline__ T zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ T neg(T a) { return make_float2(-a.x, -a.y); }
  static __device__ __forceinline__ T add(T a, double v) {
    const float2 b = df_split(v);
    const float s = a.x + b.x;
    const float bp = s - a.x;
    const float t = ((a.x - (s - bp)) + (b.x - bp)) + (a.y + b.y);
    return df_two_sum(s, t);
  }
  static __device__ __forceinline__ D dev(T a, double target) { return fabsf((a.x - (float)target) + a.y); }
  static __device__ __forceinline__ T mul(T a, T b) { return df_mul(a, b); }
  static __device__ __forceinline__ bool positive(T a) { return a.x >= 1.17549435e-38f && isfinite(a.x); }
  static __device__ __forceinline__ T shfl(T a, int l) {
    return make_float2(__shfl_sync(0xffffffffu, a.x, l), __shfl_sync(0xffffffffu, a.y, l));
  }
  static __device__ __forceinline__ Acc open(T a) { return a; }
  static __device__ __forceinline__ void fnms(Acc& a, T b, T c) { df_fnms(a, b, c); }
  static __device__ __forceinline__ void tidy(Acc& a) { df_tidy(a); }
  static __device__ __forceinline__ T close(Acc a) { return df_two_sum(a.x, a.y); }
  static __device__ __forceinline__ T rsqrt(T d) { return df_rsqrt(d); }
  static __device__ __forceinline__ T sqrt_of(T d, T ip) { return df_sqrt(d, ip); }
};

// t[e1] -= sum_s p1[s] x[s] and the same at e2 (skipped below zero; fresh: from
// zero instead of t): two rows at once, so that their chains overlap
template <class A, class T = typename A::T>
__device__ __forceinline__ void rank8(T* t, int e1, int e2, const T* p1, const T* p2, const T* x, bool fresh) {
  if (e1 < 0 && e2 < 0) return;
  __align__(16) T q1[NB], q2[NB];
#pragma unroll
  for (int s = 0; s < NB; s += 2) {
    *reinterpret_cast<int4*>(q1 + s) = *reinterpret_cast<const int4*>(p1 + s);
    *reinterpret_cast<int4*>(q2 + s) = *reinterpret_cast<const int4*>(p2 + s);
  }
  typename A::Acc c1 = A::open(fresh || e1 < 0 ? A::zero() : t[e1]), c2 = A::open(fresh || e2 < 0 ? A::zero() : t[e2]);
#pragma unroll
  for (int s = 0; s < NB; ++s) {
    A::fnms(c1, q1[s], x[s]);
    A::fnms(c2, q2[s], x[s]);
    A::tidy(c1);
    A::tidy(c2);
  }
  if (e1 >= 0) t[e1] = A::close(c1);
  if (e2 >= 0) t[e2] = A::close(c2);
}

template <class A>
__global__ void __launch_bounds__(CHOL_T, 1) chol_inv_kernel(const CholJob* __restrict__ jobs, double* __restrict__ ws,
                                                             int* __restrict__ fail) {
  using T = typename A::T;
  using D = typename A::D;
  extern __shared__ __align__(16) unsigned char chol_raw[];
  const CholJob J = jobs[blockIdx.x];
  const int n = J.n;
  if (J.shift == 3) {
    if (threadIdx.x == 0) fail[J.sec] = 1;
    return;
  }
  if (fail[J.sec]) return;
  // the packed triangle: shared memory, or the job's workspace scratch (L2
  // resident) for the sectors too large for it; then n x 8: a block's columns or rows
  // of R, for broadcast loads
  const bool in_smem = n <= CHOL_MAXN;
  T* sm = in_smem ? reinterpret_cast<T*>(chol_raw) : reinterpret_cast<T*>(ws + J.pk);
  T* P = reinterpret_cast<T*>(chol_raw) + (in_smem ? tri_elems(n) : 0);
  const double* G = ws + J.g;
  double* R = ws + J.r;
  double* Ri = ws + J.ri;
  const long long nn = (long long)n * n;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  __shared__ D red[CHOL_W];
  __shared__ T dg[NB][NB];    // diagonal block (rows of R)
  __shared__ T dip[NB];       // reciprocals of its pivots
  __shared__ int bad;
  // G: the partial matrices of one element all in flight (one load at a time, a
  // sector of 180 with 6 of them spent 70 us here)
  for (int i = warp; i < n; i += CHOL_W)
    for (int j = i + lane; j < n; j += 32) {
      const double* ge = G + (long long)i * n + j;
      double g[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) g[q] = q < J.parts ? ge[q * nn] : 0.0;
      T acc = A::of(g[0]);
#pragma unroll
      for (int q = 1; q < 8; ++q)
        if (q < J.parts) acc = A::add(acc, g[q]);
      for (int q = 8; q < J.parts; ++q) acc = A::add(acc, ge[q * nn]);
      sm[pk(i, j, n)] = acc;
    }
  if (tid == 0) bad = 0;
  __syncthreads();
  if (J.shift == 2) {
    // last pass: G = I + E; first-order factor when n max|E| <= 1e-8, else a
    // full factorisation; far from I (> 1e-3): Householder fallback
    const D big = (D)1e30;
    D mx = 0;
    for (int i = warp; i < n; i += CHOL_W)
      for (int j = i + lane; j < n; j += 32) {
        const D dev = A::dev(sm[pk(i, j, n)], i == j ? 1.0 : 0.0);
        mx = (dev <= mx) ? mx : (dev == dev ? dev : big);
      }
    for (int o = 16; o > 0; o >>= 1) {
      const D other = __shfl_xor_sync(0xffffffffu, mx, o);
      mx = other > mx ? other : mx;
    }
    if (lane == 0) red[warp] = mx;
    __syncthreads();
    D all = 0;
    for (int q = 0; q < CHOL_W; ++q) all = red[q] > all ? red[q] : all;
    if (!(all <= (D)1e-3)) {
      if (tid == 0) fail[J.sec] = 1;
      return;
    }
    if ((double)n * (double)all <= 1e-8) {
      for (int i = warp; i < n; i += CHOL_W)
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
  if (J.shift == 1) {
    // shift s = 11 (m n + n (n + 1)) u ||X||^2 with ||X||^2 <= tr(G), u the unit
    // roundoff of the arithmetic that factorises G
    if (warp == 0) {
      double tr = 0.0;
      for (int i = lane; i < n; i += 32) tr += A::dbl(sm[pk(i, i, n)]);
      for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
      const double sft = 11.0 * ((double)J.m * n + (double)n * (n + 1)) * A::u * tr;
      for (int i = lane; i < n; i += 32) sm[pk(i, i, n)] = A::of(A::dbl(sm[pk(i, i, n)]) + sft);
    }
    __syncthreads();
  }
  // ---- factor.  Warp 0 factorises and inverts the diagonal block at k0, after
  // taking the update by the block before it, while the other warps update the
  // rest of the trailing triangle.  Lane l holds columns 2 (l % 4), + 1 of row
  // l / 4 of the block and of the identity beside it: the row operations that
  // turn the block into R turn the identity into R^-T.
  auto diagonal = [&](int k0) {
    const int kb = min(NB, n - k0);
    const int i = lane >> 2, j0 = 2 * (lane & 3);
    T a[2], w[2];
    {
      typename A::Acc c[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int j = j0 + q;
        w[q] = A::of(i == j ? 1.0 : 0.0);
        c[q] = A::open((i <= j && j < kb) ? sm[pk(k0 + i, k0 + j, n)] : w[q]);
      }
      if (k0 > 0) {
#pragma unroll 2
        for (int t = 0; t < NB; ++t) {
          const T ri = P[(k0 + min(i, kb - 1)) * NB + t];
#pragma unroll
          for (int q = 0; q < 2; ++q)
            if (i <= j0 + q && j0 + q < kb) {
              A::fnms(c[q], ri, P[(k0 + j0 + q) * NB + t]);
              A::tidy(c[q]);
            }
        }
      }
      a[0] = A::close(c[0]);
      a[1] = A::close(c[1]);
    }
    bool ok = true;
    T own = A::of(1.0);  // reciprocal of row i's pivot
#pragma unroll 1
    for (int s = 0; s < kb; ++s) {
      const T d = A::shfl((s & 1) ? a[1] : a[0], 4 * s + (s >> 1));
      ok = ok && A::positive(d);
      const T ip = A::rsqrt(d);
      if (i == s) {  // (the pivot itself after the loop, off the chain)
        own = ip;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          if (j0 + q != s) a[q] = A::mul(a[q], ip);
          w[q] = A::mul(w[q], ip);
        }
      }
      __syncwarp();
      // row s at this lane's columns, and R(s, i)
      const T r0 = A::shfl(a[0], 4 * s + (lane & 3)), r1 = A::shfl(a[1], 4 * s + (lane & 3));
      const T v0 = A::shfl(w[0], 4 * s + (lane & 3)), v1 = A::shfl(w[1], 4 * s + (lane & 3));
      const T e0 = A::shfl(a[0], 4 * s + (i >> 1)), e1 = A::shfl(a[1], 4 * s + (i >> 1));
      const T rsi = (i & 1) ? e1 : e0;
      if (i > s) {
        typename A::Acc c0 = A::open(a[0]), c1 = A::open(a[1]), u0 = A::open(w[0]), u1 = A::open(w[1]);
        A::fnms(c0, rsi, r0);
        A::fnms(c1, rsi, r1);
        A::fnms(u0, rsi, v0);
        A::fnms(u1, rsi, v1);
        a[0] = A::close(c0);
        a[1] = A::close(c1);
        w[0] = A::close(u0);
        w[1] = A::close(u1);
      }
      if (lane == 0) dip[s] = ip;
    }
    if (!ok && lane == 0) {
      bad = 1;
      fail[J.sec] = 1;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int j = j0 + q;
      if (i == j && i < kb) a[q] = A::sqrt_of(a[q], own);
      dg[i][j] = i <= j ? a[q] : A::zero();
      if (i <= j && j < kb) sm[pk(k0 + i, k0 + j, n)] = a[q];
      if (j <= i && i < kb) Ri[(long long)(k0 + j) * n + k0 + i] = A::dbl(w[q]);  // R^-1 = (R^-T)^T
    }
  };
  if (warp == 0) diagonal(0);
  __syncthreads();
  for (int k0 = 0; !bad && k0 + NB < n; k0 += NB) {
    const int c0 = k0 + NB;  // first trailing column
    for (int j = c0 + tid; j < n; j += CHOL_T) {
      typename A::Acc v[NB];
      T r[NB];
#pragma unroll
      for (int s = 0; s < NB; ++s) v[s] = A::open(sm[pk(k0 + s, j, n)]);
#pragma unroll
      for (int s = 0; s < NB; ++s) {
        r[s] = A::mul(A::close(v[s]), dip[s]);
#pragma unroll
        for (int t = s + 1; t < NB; ++t) A::fnms(v[t], dg[s][t], r[s]);
      }
#pragma unroll
      for (int s = 0; s < NB; ++s) {
        sm[pk(k0 + s, j, n)] = r[s];
        P[j * NB + s] = r[s];
      }
    }
    __syncthreads();
    if (warp == 0) {
      diagonal(c0);
    } else if ((warp & 3) || n - c0 > 96) {
      // while the diagonal block takes longer than the rest, warp 0 keeps its SM
      // sub-partition to itself
      const bool all = n - c0 > 96;
      const int tw = all ? warp - 1 : warp - 1 - (warp >> 2), TRAIL_W = all ? CHOL_W - 1 : CHOL_W - CHOL_W / 4;
      for (int j0 = c0; j0 < n; j0 += 32) {
        const int j = j0 + lane;
        T r[NB];
#pragma unroll
        for (int s = 0; s < NB; ++s) r[s] = j < n ? sm[pk(k0 + s, j, n)] : A::zero();
        const int iend = min(j0 + 32, n);
        for (int i = c0 + tw; i < iend; i += 2 * TRAIL_W) {
          const int i2 = i + TRAIL_W;
          const bool in1 = j < n && j >= i && j >= c0 + NB, in2 = i2 < iend && j < n && j >= i2 && j >= c0 + NB;
          rank8<A>(sm, in1 ? pk(i, j, n) : -1, in2 ? pk(i2, j, n) : -1, P + i * NB, P + (i2 < n ? i2 : i) * NB, r, false);
        }
      }
    }
    __syncthreads();
  }
  if (bad) return;
  for (int i = warp; i < n; i += CHOL_W)
    for (int j = lane; j < n; j += 32) R[(long long)i * n + j] = (j >= i) ? A::dbl(sm[pk(i, j, n)]) : 0.0;
  __syncthreads();
  // ---- inverse: the diagonal blocks' inverses (written above) take their place
  for (int e = tid; e < (n + NB - 1) / NB * (NB * NB); e += CHOL_T) {
    const int k0 = e / (NB * NB) * NB, i = k0 + (e / NB) % NB, j = k0 + e % NB;
    if (i <= j && j < n) sm[pk(i, j, n)] = A::of(Ri[(long long)i * n + j]);
  }
  __syncthreads();
  for (int k0 = (n - 1) / NB * NB; k0 >= 0; k0 -= NB) {
    const int kb = min(NB, n - k0);
    if (tid < CHOL_T / 2) {
      // block row: X(K, c) = D S(K, c)
      for (int c = k0 + kb + tid; c < n; c += CHOL_T / 2) {
        T sv[NB];
#pragma unroll
        for (int s = 0; s < NB; ++s) {
          const T v = s < kb ? sm[pk(k0 + s, c, n)] : A::zero();
          sv[s] = v;
        }
#pragma unroll
        for (int s = 0; s < NB; ++s) {
          if (s < kb) {
            typename A::Acc a = A::open(A::zero());
#pragma unroll
            for (int t = s; t < NB; ++t)
              if (t < kb) A::fnms(a, sm[pk(k0 + s, k0 + t, n)], sv[t]);
            sm[pk(k0 + s, c, n)] = A::neg(A::close(a));
          }
        }
      }
    } else {
      // the block's columns of R above it
      for (int e = tid - CHOL_T / 2; e < k0 * NB; e += CHOL_T / 2) {
        const int i = e / NB, s = e % NB;
        P[i * NB + s] = s < kb ? sm[pk(i, k0 + s, n)] : A::zero();
      }
    }
    __syncthreads();
    for (int j0 = k0; j0 < n; j0 += 32) {
      const int c = j0 + lane;
      T x[NB];
#pragma unroll
      for (int s = 0; s < NB; ++s) x[s] = (s < kb && c < n && c >= k0 + s) ? sm[pk(k0 + s, c, n)] : A::zero();
      const bool fresh = c < k0 + kb;
      for (int i = warp; i < k0; i += 2 * CHOL_W) {
        const int i2 = i + CHOL_W;
        rank8<A>(sm, c < n ? pk(i, c, n) : -1, c < n && i2 < k0 ? pk(i2, c, n) : -1, P + i * NB,
                 P + (i2 < k0 ? i2 : i) * NB, x, fresh);
      }
    }
    __syncthreads();
  }
  for (int i = warp; i < n; i += CHOL_W)
    for (int j = lane; j < n; j += 32) Ri[(long long)i * n + j] = (j >= i) ? A::dbl(sm[pk(i, j, n)]) : 0.0;
}

}  // namespace

cudaError_t launch_chol_inv(const CholJob* jobs, int njobs, double* ws, int* fail, cudaStream_t s, int maxn, bool df) {
  if (njobs == 0) return cudaSuccess;
  // every job's own triangle and copies (of a sector too large for it the copies)
  const size_t copy = (size_t)NB * maxn * 8, small = chol_bytes(maxn < CHOL_MAXN ? maxn : CHOL_MAXN);
  if (copy > CHOL_SMEM) return cudaErrorInvalidValue;
  const size_t smem = copy > small ? copy : small;
  // once per process (thread-safe static initialisation): the largest size
  static const cudaError_t e1 =
      cudaFuncSetAttribute(chol_inv_kernel<CholF64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CHOL_SMEM);
  static const cudaError_t e2 =
      cudaFuncSetAttribute(chol_inv_kernel<CholDF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CHOL_SMEM);
  if (e1 != cudaSuccess) return e1;
  if (e2 != cudaSuccess) return e2;
  if (df) chol_inv_kernel<CholDF><<<njobs, CHOL_T, smem, s>>>(jobs, ws, fail);
  else chol_inv_kernel<CholF64><<<njobs, CHOL_T, smem, s>>>(jobs, ws, fail);
  return cudaGetLastError();
}

}  // namespace tt

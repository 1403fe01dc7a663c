// Householder QR of one matrix over the whole GPU (tt_qr_device): the columns
// dealt to the CTAs of one cooperative launch, one or a few per CTA, each kept
// in that CTA's shared memory.
//
// Step k needs column k after k reflections.  Its owner publishes it (global
// memory, then a flag); every CTA with later columns reads it, forms its norm
// and its products with the CTA's own columns in one pass and one reduction,
// computes the reflector's scalars itself and updates its columns, the owner
// of column k + 1 that one first.  A column of Q is H_0 .. H_j e_j: no CTA
// needs another for it.  Waits are bounded (the cooperative launch makes every
// CTA resident, so they end; a budget that runs out sets an error flag and the
// kernel returns, and the caller takes the one-CTA kernel).
//
// What bounds it: GB300 does 2 FP64 multiply-adds per clock and SM, so one CTA
// needs 40 ms for the 1.6e8 of a 2100 x 200 matrix; over the columns they take
// 0.3 ms and the chain of n steps bounds the rest: publish and read through
// L2, the reduction, a square root and a division, 3 to 4 us a step.
// Measured (whole call): 2100 x 200 110 -> 1.9 ms, 333 x 37 0.65 -> 0.26 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "tt_kernels.h"

namespace tt {

namespace {

constexpr int GT = 256, GW = GT / 32;
constexpr int GE = 16;                   // column elements per thread: m <= GT * GE
constexpr size_t GSMEM = 160 * 1024;     // shared memory for columns and scalars

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// sums of a and b over the CTA, in every thread
__device__ __forceinline__ double2 cta_sum2(double a, double b, double (*red)[2]) {
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const bool up = lane & 16;  // halves exchange: one value per half-warp
  double s = (up ? b : a) + __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((lane & 15) == 0) red[wp][lane >> 4] = s;
  __syncthreads();
  s = red[lane & 7][(lane >> 3) & 1];
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return make_double2(__shfl_sync(0xffffffffu, s, 0), __shfl_sync(0xffffffffu, s, 8));
}

// E: column elements per thread (m <= 256 E)
template <int E>
__global__ void __launch_bounds__(GT, 1) qr_grid_kernel(const double* __restrict__ A, int m, int n, double* V,
                                                        int* flag, int* err, double* __restrict__ Q,
                                                        double* __restrict__ R, long long wait_ns) {
  extern __shared__ __align__(16) double sm[];
  __shared__ double red[2][GW][2];
  __shared__ double ws_s;
  __shared__ int stop;
  const int c = blockIdx.x, G = gridDim.x, tid = threadIdx.x;
  const int ncol = (n - c + G - 1) / G;  // own columns c, c + G, ...
  double* sc = sm;                       // scale and tau of the reflectors, tau >= 0
                                         // with the sign bit of R(k, k)
  double* ta = sm + n;
  double* col = sm + 2 * n;
  if (tid == 0) stop = 0;
  for (int q = 0; q < ncol; ++q)
    for (int i = tid; i < m; i += GT) col[(size_t)q * m + i] = A[(size_t)(c + q * G) * m + i];
  __syncthreads();
  auto publish = [&](int j, const double* x) {
    for (int i = tid; i < m; i += GT) __stcg(&V[(size_t)j * m + i], x[i]);
    __threadfence();
    __syncthreads();
    if (tid == 0) st_release(&flag[j], 1);
  };
  if (c == 0) publish(0, col);
  const int jlast = c + (ncol - 1) * G;
  int par = 0;
  for (int k = 0; k <= jlast; ++k) {
    // ---- column k of the reduced matrix
    double x[E];
    const bool own = k % G == c;
    if (!own && tid == 0 && ld_acquire(&flag[k]) == 0) {
      const unsigned long long t0 = now_ns();
      while (ld_acquire(&flag[k]) == 0)
        if ((long long)(now_ns() - t0) > wait_ns || ld_acquire(err) != 0) {
          st_release(err, 1);
          stop = 1;
          break;
        }
    }
    __syncthreads();
    if (stop) return;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int i = tid + e * GT;
      x[e] = i > k && i < m ? __ldcg(&V[(size_t)k * m + i]) : 0.0;
    }
    const double alpha = __ldcg(&V[(size_t)k * m + k]);
    const int q0 = k < c ? 0 : (k - c) / G + 1;  // first own column after k
    double s = 0.0;
#pragma unroll
    for (int e = 0; e < E; ++e) s = fma(x[e], x[e], s);
    for (int q = q0; q == q0 || q < ncol; ++q) {
      double* cj = col + (size_t)q * m;
      double d = 0.0;
      if (q < ncol) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int i = tid + e * GT;
          if (i > k && i < m) d = fma(x[e], cj[i], d);
        }
      }
      const double2 sd = cta_sum2(s, d, red[par]);
      par ^= 1;
      if (tid < 32) {
        double scale, tau;
        if (q == q0) {
          // lanes 0 and 1: 1 / (alpha - beta) and 1 / beta in one division
          const double beta = sd.x > 0.0 ? -copysign(sqrt(fma(alpha, alpha, sd.x)), alpha) : 1.0;
          const double inv = 1.0 / ((tid & 1) ? beta : (sd.x > 0.0 ? alpha - beta : 1.0));
          scale = sd.x > 0.0 ? __shfl_sync(0xffffffffu, inv, 0) : 0.0;
          tau = sd.x > 0.0 ? (beta - alpha) * __shfl_sync(0xffffffffu, inv, 1) : 0.0;
          if (tid == 0) {
            const double rkk = sd.x > 0.0 ? beta : alpha;
            sc[k] = scale;
            ta[k] = rkk < 0.0 ? -tau : tau;
            if (own) col[(size_t)(k / G) * m + k] = rkk;
          }
        } else {
          scale = sc[k];
          tau = fabs(ta[k]);
        }
        if (tid == 0) {
          const double w = q < ncol ? tau * fma(scale, sd.y, cj[k]) : 0.0;
          ws_s = w * scale;
          if (q < ncol) cj[k] -= w;
        }
      }
      __syncthreads();
      if (q < ncol) {
        const double ws = ws_s;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int i = tid + e * GT;
          if (i > k && i < m) cj[i] = fma(-ws, x[e], cj[i]);
        }
        if (c + q * G == k + 1) {
          __syncthreads();
          publish(k + 1, cj);
        }
      }
    }
  }
  __syncthreads();
  // ---- R (diag >= 0: row i negated where R(i, i) < 0) and Q, column by column
  for (int q = 0; q < ncol; ++q) {
    const int j = c + q * G;
    double* cj = col + (size_t)q * m;
    for (int i = tid; i < n; i += GT) {
      const double v = i <= j ? cj[i] : 0.0;
      R[(size_t)j * n + i] = i <= j && signbit(ta[i]) ? -v : v;
    }
    const bool neg = signbit(ta[j]);
    double y[E];
#pragma unroll
    for (int e = 0; e < E; ++e) y[e] = tid + e * GT == j ? 1.0 : 0.0;
    double x[E], xn[E];
    auto load = [&](int k, double* to) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int i = tid + e * GT;
        to[e] = i > k && i < m ? __ldcg(&V[(size_t)k * m + i]) : 0.0;
      }
    };
    load(j, x);
    for (int k = j; k >= 0; --k) {
      if (k > 0) load(k - 1, xn);
      const double scale = sc[k], tau = fabs(ta[k]);
      double d = 0.0, yk = 0.0;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        d = fma(x[e], y[e], d);
        if (tid + e * GT == k) yk = y[e];
      }
      const double2 sd = cta_sum2(d, yk, red[par]);
      par ^= 1;
      const double w = tau * fma(scale, sd.x, sd.y), ws = w * scale;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        y[e] = fma(-ws, x[e], y[e]);
        if (tid + e * GT == k) y[e] -= w;
        x[e] = xn[e];
      }
    }
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int i = tid + e * GT;
      if (i < m) Q[(size_t)j * m + i] = neg ? -y[e] : y[e];
    }
  }
}

}  // namespace

// CTAs for an m x n matrix, or 0 where the kernel does not apply (a column
// longer than its register tile, or more of them per CTA than shared memory
// holds: the one-CTA kernel's case)
static int ctas_of(int m, int n, int sms) {
  if (m > GT * GE) return 0;
  const int G = std::min(n, sms), cp = (n + G - 1) / G;
  return ((size_t)cp * m + 2 * (size_t)n) * sizeof(double) <= GSMEM ? G : 0;
}

cudaError_t qr_grid_ctas(int m, int n, int* ctas) {
  *ctas = 0;
  int dev = 0, sms = 0, coop = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (e == cudaSuccess && coop) *ctas = ctas_of(m, n, sms);
  return e;
}

size_t qr_grid_scratch(int m, int n) { return (size_t)m * n * sizeof(double) + ((size_t)n + 1) * sizeof(int); }

cudaError_t launch_qr_grid(const double* A, int m, int n, int ctas, double* Q, double* R, void* scratch,
                           long long wait_ns, cudaStream_t s, int** err, bool* done) {
  *done = false;
  *err = nullptr;
  const int G = ctas;
  double* V = (double*)scratch;
  int* flag = (int*)(V + (size_t)m * n);
  int* er = flag + n;
  cudaError_t e = cudaMemsetAsync(flag, 0, ((size_t)n + 1) * sizeof(int), s);
  if (e != cudaSuccess) return e;
  const size_t smem = ((size_t)((n + G - 1) / G) * m + 2 * (size_t)n) * sizeof(double);
  const int el = (m + GT - 1) / GT;
  const void* k = el <= 2 ? (const void*)qr_grid_kernel<2>
                          : el <= 4 ? (const void*)qr_grid_kernel<4>
                                    : el <= 9 ? (const void*)qr_grid_kernel<9> : (const void*)qr_grid_kernel<GE>;
  e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GSMEM);
  if (e != cudaSuccess) return e;
  void* args[] = {(void*)&A, &m, &n, &V, &flag, &er, &Q, &R, &wait_ns};
  e = cudaLaunchCooperativeKernel(k, dim3(G), dim3(GT), args, smem, s);
  if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {  // (a share of the GPU only)
    cudaGetLastError();
    return cudaSuccess;
  }
  if (e != cudaSuccess) return e;
  *err = er;
  *done = true;
  return cudaSuccess;
}

}  // namespace tt

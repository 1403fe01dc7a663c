// Device kernels of the tanTRG hot path (sm_103a).
//
//  * grouped, segmented GEMM (split-BF16 on the tensor cores; FP64 in
//    tt_gemm64.cu, double-float in tt_gemmdf.cu):
//    every contraction of the H_eff apply (Supplement, Fig. "Lanczos": L_i A_i,
//    then H_i, then R_i), the bond apply (Fig. "optimalB"(d)), the environment
//    updates and the absorb step is a list of groups C_g = sum_seg A_seg B_seg;
//  * W gather: applies the sparse MPO tensor between the two GEMM stages;
//  * norms and dot products with deterministic two-stage reductions;
//  * Householder QR (FP64) of the per-sector gauge matrices.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <type_traits>

#include "tt_kernels.h"

namespace tt {

namespace {

__device__ __forceinline__ int slot_of(Ref r) { return (int)(r >> 56); }
__device__ __forceinline__ long long off_of(Ref r) { return (long long)(r & 0x00FFFFFFFFFFFFFFull); }

template <typename T>
__device__ __forceinline__ T* rptr(const Bases& b, Ref r) {
  return reinterpret_cast<T*>(sel_base(b, slot_of(r))) + off_of(r);
}

constexpr int VT = 256;

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------------------
// Split-BF16 grouped GEMM on the tensor cores (mma.sync m16n8k16, FP32
// accumulation).  Operands are stored as NS bf16 levels x = x0 + x1 (+ x2),
// level l at element offset l * lo[slot]; the products with l_A + l_B < NS are
// summed: NS = 2 -> 3 products (~2^-16 relative), NS = 3 -> 6 products
// (~2^-24).  The leading product x0*y0 and the smaller ones accumulate in
// separate FP32 registers; every 32-wide K chunk the leading one is folded
// into a two-float (hi, lo) sum with TwoSum (Knuth, TAOCP vol. 2, 4.2.2) and
// the small one is added to lo, so the accumulation error does not grow with
// K.  64 x 64 tile per CTA, 4 warps of 32 x 32.  Output FP64 or FP32 (flags
// bit1).
// ---------------------------------------------------------------------------
constexpr int HBM = 64, HBN = 64, HBK = 32, HPAD = 8;

__device__ __forceinline__ void mma_bf16_16816(float* c, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ void two_sum_acc(float& hi, float& lo, float x) {
  const float s = hi + x;
  const float bp = s - hi;
  const float ap = s - bp;
  lo += (hi - ap) + (x - bp);
  hi = s;
}

template <int NS>
__global__ void __launch_bounds__(128) gemm_bf16_split_kernel(const GGroup* __restrict__ groups,
                                                              const GSeg* __restrict__ segs,
                                                              const GTile* __restrict__ tiles, Bases bs) {
  __shared__ __align__(16) __nv_bfloat16 As[NS][HBM][HBK + HPAD];
  __shared__ __align__(16) __nv_bfloat16 Bs[NS][HBN][HBK + HPAD];
  const GTile tl = tiles[blockIdx.x];
  const GGroup g = groups[tl.g];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
  const int gid = lane >> 2, tig = lane & 3;
  float acc[2][4][4], accs[2][4][4], hi[2][4][4], lo[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int r = 0; r < 4; ++r) { acc[i][j][r] = 0.f; accs[i][j][r] = 0.f; hi[i][j][r] = 0.f; lo[i][j][r] = 0.f; }

  for (int si = g.seg0; si < g.seg1; ++si) {
    const GSeg sg = segs[si];
    const __nv_bfloat16* A0 = rptr<const __nv_bfloat16>(bs, sg.A);
    const __nv_bfloat16* B0 = rptr<const __nv_bfloat16>(bs, sg.B);
    const long long loA = sel_lo(bs, slot_of(sg.A)), loB = sel_lo(bs, slot_of(sg.B));
    for (int k0 = 0; k0 < sg.K; k0 += HBK) {
      for (int e = tid; e < HBM * HBK; e += 128) {
        int mm, kk;
        if (sg.tA) { mm = e % HBM; kk = e / HBM; } else { kk = e % HBK; mm = e / HBK; }
        const int gm = tl.m0 + mm, gk = k0 + kk;
        const bool in = gm < g.M && gk < sg.K;
        const long long o = sg.tA ? (long long)gk * sg.lda + gm : (long long)gm * sg.lda + gk;
#pragma unroll
        for (int l = 0; l < NS; ++l) As[l][mm][kk] = in ? A0[l * loA + o] : __float2bfloat16(0.f);
      }
      for (int e = tid; e < HBN * HBK; e += 128) {
        int nn, kk;
        if (sg.tB) { kk = e % HBK; nn = e / HBK; } else { nn = e % HBN; kk = e / HBN; }
        const int gn = tl.n0 + nn, gk = k0 + kk;
        const bool in = gn < g.N && gk < sg.K;
        const long long o = sg.tB ? (long long)gn * sg.ldb + gk : (long long)gk * sg.ldb + gn;
#pragma unroll
        for (int l = 0; l < NS; ++l) Bs[l][nn][kk] = in ? B0[l * loB + o] : __float2bfloat16(0.f);
      }
      __syncthreads();
#pragma unroll
      for (int pass = 0; pass < (NS == 2 ? 3 : 6); ++pass) {
        // (la, lb): NS=2: (0,0) (0,1) (1,0); NS=3 adds (0,2) (1,1) (2,0); small products first
        const int order = (NS == 2 ? 2 : 5) - pass;
        const int la = (order == 2 || order == 4) ? 1 : (order == 5 ? 2 : 0);
        const int lb = (order == 1 || order == 4) ? 1 : (order == 3 ? 2 : 0);
#pragma unroll
        for (int ks = 0; ks < HBK; ks += 16) {
          uint32_t af[2][4], bf[4][2];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int r0 = wm + 16 * i + gid;
            af[i][0] = *reinterpret_cast<const uint32_t*>(&As[la][r0][ks + 2 * tig]);
            af[i][1] = *reinterpret_cast<const uint32_t*>(&As[la][r0 + 8][ks + 2 * tig]);
            af[i][2] = *reinterpret_cast<const uint32_t*>(&As[la][r0][ks + 8 + 2 * tig]);
            af[i][3] = *reinterpret_cast<const uint32_t*>(&As[la][r0 + 8][ks + 8 + 2 * tig]);
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int c0 = wn + 8 * j + gid;
            bf[j][0] = *reinterpret_cast<const uint32_t*>(&Bs[lb][c0][ks + 2 * tig]);
            bf[j][1] = *reinterpret_cast<const uint32_t*>(&Bs[lb][c0][ks + 8 + 2 * tig]);
          }
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) mma_bf16_16816(order == 0 ? acc[i][j] : accs[i][j], af[i], bf[j]);
        }
      }
      __syncthreads();
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            two_sum_acc(hi[i][j][r], lo[i][j][r], acc[i][j][r]);
            lo[i][j][r] += accs[i][j][r];
            acc[i][j][r] = 0.f;
            accs[i][j][r] = 0.f;
          }
    }
  }
  const bool accum = g.flags & 1;
  const bool out_f32 = g.flags & 2;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int gm = tl.m0 + wm + 16 * i + gid + ((r >= 2) ? 8 : 0);
        const int gn = tl.n0 + wn + 8 * j + 2 * tig + (r & 1);
        if (gm >= g.M || gn >= g.N) continue;
        const long long o = (long long)gm * g.ldc + gn;
        const double v = (double)hi[i][j][r] + (double)lo[i][j][r];
        if (out_f32) {
          float* C = rptr<float>(bs, g.C) + o;
          *C = accum ? *C + (float)v : (float)v;
        } else {
          double* C = rptr<double>(bs, g.C) + o;
          *C = accum ? *C + v : v;
        }
      }
}

// ---------------------------------------------------------------------------
// W gather: dst[r, c] = sum_k coef_k src_k[r, c].  One CTA per item (or share of
// its rows), rows over the 8 warps, columns over the lanes.  FP64 in, FP64 out
// for the FP64 path.  Mixed path: the sources are the FP32 outputs of S1, so
// the sum and the split into bf16 levels run in FP32 (GB300 has about 1/64 of
// its FP32 rate in FP64); each level's remainder is exact in FP32.
//
// What bounds it: memory latency.  Most items have one or two terms, the ones
// that close a hop several dozen, and with one row and one load at a time per
// warp such an item alone took longer than all others.  The term records sit in
// shared memory, four rows and two terms are in flight per lane, and items are
// cut by rows according to their terms (upload), longest first.
// ---------------------------------------------------------------------------
constexpr int GT_TAB = 64;  // terms kept in shared memory (more: read as they come)

template <int NS>
__device__ __forceinline__ void store_split_f32(__nv_bfloat16* p, long long lo, float v) {
#pragma unroll
  for (int l = 0; l < NS; ++l) {
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    p[l * lo] = h;
    v -= __bfloat162float(h);
  }
}
// FP64 value: the first level is rounded from the double and its remainder
// (|r| <= 2^-9 |x|) is rounded to FP32 once, so the levels carry the value to
// about 2^-25 relative with two FP64 operations per element.
template <int NS>
__device__ __forceinline__ void store_split_f64(__nv_bfloat16* p, long long lo, double x) {
  const __nv_bfloat16 h0 = __double2bfloat16(x);
  p[0] = h0;
  store_split_f32<NS - 1>(p + lo, lo, __double2float_rn(x - (double)__bfloat162float(h0)));
}

template <int IN, int OUT>
__global__ void __launch_bounds__(256) gather_kernel(const GItem* __restrict__ items,
                                                     const GContrib* __restrict__ cs, Bases bs) {
  using T = typename std::conditional<IN == 0, double, float>::type;
  constexpr int JR = 4;
  __shared__ const T* tp[GT_TAB];
  __shared__ long long trs[GT_TAB];
  __shared__ T tc[GT_TAB];
  const GItem it = items[blockIdx.x];
  const int nk = it.c1 - it.c0;
  for (int k = threadIdx.x; k < min(nk, GT_TAB); k += 256) {
    const GContrib cb = cs[it.c0 + k];
    tp[k] = rptr<const T>(bs, cb.src);
    trs[k] = cb.src_rs;
    tc[k] = (T)cb.coef;
  }
  __syncthreads();
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int r = it.r0 + ty; r < it.rows; r += 8 * JR)
    for (int c = tx; c < it.cols; c += 32) {
      T acc[JR];
#pragma unroll
      for (int j = 0; j < JR; ++j) acc[j] = (T)0;
      auto load = [&](const T* p, long long rs, T* v) {
#pragma unroll
        for (int j = 0; j < JR; ++j) v[j] = r + 8 * j < it.rows ? p[(long long)(r + 8 * j) * rs + c] : (T)0;
      };
      auto add = [&](T f, const T* v) {
#pragma unroll
        for (int j = 0; j < JR; ++j) acc[j] = fma(f, v[j], acc[j]);
      };
      int k = 0;
      for (; k + 1 < min(nk, GT_TAB); k += 2) {
        T v0[JR], v1[JR];
        load(tp[k], trs[k], v0);
        load(tp[k + 1], trs[k + 1], v1);
        add(tc[k], v0);
        add(tc[k + 1], v1);
      }
      for (; k < nk; ++k) {
        T v0[JR];
        if (k < GT_TAB) {
          load(tp[k], trs[k], v0);
          add(tc[k], v0);
        } else {
          const GContrib cb = cs[it.c0 + k];
          load(rptr<const T>(bs, cb.src), cb.src_rs, v0);
          add((T)cb.coef, v0);
        }
      }
#pragma unroll
      for (int j = 0; j < JR; ++j) {
        if (r + 8 * j >= it.rows) continue;
        const long long d = (long long)(r + 8 * j) * it.dst_rs + c;
        if constexpr (OUT == 0) rptr<double>(bs, it.dst)[d] = (double)acc[j];
        else if constexpr (OUT == 1) rptr<float>(bs, it.dst)[d] = (float)acc[j];
        else if constexpr (IN == 0) store_split_f64<OUT>(rptr<__nv_bfloat16>(bs, it.dst) + d, sel_lo(bs, slot_of(it.dst)), acc[j]);
        else store_split_f32<OUT>(rptr<__nv_bfloat16>(bs, it.dst) + d, sel_lo(bs, slot_of(it.dst)), acc[j]);
      }
    }
}

// Strided 2-D copies, one item = rows x cols elements with arbitrary row and
// column strides on both sides.  The items are cut into 32 x 32 tiles, a CTA
// takes COPY_TILES of them (a list made with the plan: sized by the largest item,
// most CTAs of a grid had nothing to do, 12 us for 1 MB).  A tile goes through
// shared memory so that both the load and the store run along whichever side
// has unit stride (a transposing copy is coalesced on both ends).  NS = 0: FP64 -> FP64; NS = 2, 3: FP64 -> split
// bf16 levels at dst + l * lo[slot(dst)].
template <int NS>
__global__ void __launch_bounds__(256) tile_copy_kernel(const CItem* __restrict__ items, const CPart* __restrict__ parts,
                                                        Bases bs) {
  __shared__ double tile[32][33];
  const CPart part = parts[blockIdx.x];
  const CItem it = items[part.item];
  const double* src = rptr<const double>(bs, it.src);
  const int tcr = (it.rows + 31) >> 5, tcc = (it.cols + 31) >> 5;
  const int ntiles = tcr * tcc;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
  const bool src_rmaj = it.src_cs == 1 || it.src_rs != 1;   // src contiguous along c
  const bool dst_rmaj = it.dst_cs == 1 || it.dst_rs != 1;
  for (int t = part.first; t < min(ntiles, part.first + COPY_TILES); ++t) {
    const int r0 = (t / tcc) << 5, c0 = (t % tcc) << 5;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int a = ty + 8 * k;  // slow index within the tile
      const int r = src_rmaj ? r0 + a : r0 + tx, c = src_rmaj ? c0 + tx : c0 + a;
      if (r < it.rows && c < it.cols) {
        const double v = src[(long long)r * it.src_rs + (long long)c * it.src_cs];
        if (src_rmaj) tile[a][tx] = v;
        else tile[tx][a] = v;
      }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int a = ty + 8 * k;
      const int lr = dst_rmaj ? a : tx, lc = dst_rmaj ? tx : a;
      const int r = r0 + lr, c = c0 + lc;
      if (r < it.rows && c < it.cols) {
        const long long o = (long long)r * it.dst_rs + (long long)c * it.dst_cs;
        const double v = tile[lr][lc];
        if constexpr (NS == 0) rptr<double>(bs, it.dst)[o] = v;
        else store_split_f64<NS>(rptr<__nv_bfloat16>(bs, it.dst) + o, sel_lo(bs, slot_of(it.dst)), v);
      }
    }
    __syncthreads();
  }
}

// x (FP64, n) -> ns bf16 levels out[l * n + i], x ~ sum_l out[l].
__global__ void split_bf16_kernel(const double* __restrict__ x, long long n, int ns, __nv_bfloat16* __restrict__ out) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    if (ns == 2) store_split_f64<2>(out + i, n, x[i]);
    else store_split_f64<3>(out + i, n, x[i]);
  }
}


// ---------------------------------------------------------------------------
// Norms and dot products of flat vectors (the Lanczos steps: tt_lanczos.cu)
// ---------------------------------------------------------------------------
__global__ void sumsq_kernel(const double* __restrict__ v, long long n, double* __restrict__ partial) {
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)VT + threadIdx.x; i < n; i += (long long)gridDim.x * VT)
    acc = fma(v[i], v[i], acc);
  __shared__ double red[VT / 32];
  double s = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < VT / 32; ++q) t += red[q];
    partial[blockIdx.x * VEC_SUMS] = t;
  }
}

// out[j] = sum_b partial[b * VEC_SUMS + j] in a fixed order (deterministic)
__device__ void finalize_sums(const double* partial, int nblk, int nv, double* out) {
  // called by one warp
  const int lane = threadIdx.x & 31;
  for (int j = 0; j < nv; ++j) {
    double s = 0.0;
    for (int b = lane; b < nblk; b += 32) s += partial[b * VEC_SUMS + j];
    s = warp_sum(s);
    if (lane == 0) out[j] = s;
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

// ---------------------------------------------------------------------------
// Householder QR, one CTA per column-major matrix (ld = m).
// ---------------------------------------------------------------------------
constexpr int QRT = 256;
constexpr int QR_MAXN = 2048;

__device__ __forceinline__ void qr_one(const QrJob J, double* __restrict__ ws);

__global__ void __launch_bounds__(QRT) qr_kernel(const QrJob* __restrict__ jobs, double* __restrict__ ws,
                                                 const int* __restrict__ only, int* __restrict__ nrun) {
  if (only && !only[blockIdx.x]) return;  // masked launch: fallback sectors only
  if (nrun && threadIdx.x == 0) atomicAdd(nrun, 1);
  qr_one(jobs[blockIdx.x], ws);
}

// one matrix whose job record travels as a kernel argument (no device copy of it)
__global__ void __launch_bounds__(QRT) qr_byval_kernel(const QrJob J, double* __restrict__ ws) { qr_one(J, ws); }

__device__ __forceinline__ void qr_one(const QrJob J, double* __restrict__ ws) {
  const int m = J.m, n = J.n;
  double* A = ws + J.a;
  double* Qm = ws + J.q;
  double* R = ws + J.r;
  __shared__ double tau_s[QR_MAXN];
  __shared__ double red[QRT / 32];
  __shared__ double bcast;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, nw = QRT / 32;
  const int kmax = m < n ? m : n;
  for (int k = 0; k < kmax; ++k) {
    double* col = A + (long long)k * m;
    double s = 0.0;
    for (int i = k + 1 + threadIdx.x; i < m; i += QRT) s = fma(col[i], col[i], s);
    s = warp_sum(s);
    if (lane == 0) red[wp] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int q = 0; q < nw; ++q) t += red[q];
      double alpha = col[k];
      double tau = 0.0, scale = 0.0;
      if (t > 0.0) {
        double beta = -copysign(sqrt(alpha * alpha + t), alpha);
        tau = (beta - alpha) / beta;
        scale = 1.0 / (alpha - beta);
        col[k] = beta;
      }
      tau_s[k] = tau;
      bcast = scale;
    }
    __syncthreads();
    const double scale = bcast;
    if (tau_s[k] != 0.0)
      for (int i = k + 1 + threadIdx.x; i < m; i += QRT) col[i] *= scale;
    __syncthreads();
    const double tau = tau_s[k];
    if (tau != 0.0) {
      for (int j = k + 1 + wp; j < n; j += nw) {
        double* cj = A + (long long)j * m;
        double w = 0.0;
        for (int i = k + 1 + lane; i < m; i += 32) w = fma(col[i], cj[i], w);
        w = warp_sum(w) + cj[k];
        w *= tau;
        if (lane == 0) cj[k] -= w;
        for (int i = k + 1 + lane; i < m; i += 32) cj[i] = fma(-w, col[i], cj[i]);
      }
    }
    __syncthreads();
  }
  // R (n x n, column-major)
  for (long long e = threadIdx.x; e < (long long)n * n; e += QRT) {
    int i = (int)(e % n), j = (int)(e / n);
    R[e] = (i <= j && i < m) ? A[(long long)j * m + i] : 0.0;
  }
  // Q = H_0 ... H_{kmax-1} [I_n ; 0]   (columns j >= m stay zero)
  for (long long e = threadIdx.x; e < (long long)m * n; e += QRT) {
    int i = (int)(e % m), j = (int)(e / m);
    Qm[e] = (i == j) ? 1.0 : 0.0;
  }
  __syncthreads();
  for (int k = kmax - 1; k >= 0; --k) {
    const double tau = tau_s[k];
    if (tau == 0.0) continue;
    const double* v = A + (long long)k * m;
    for (int j = k + wp; j < n; j += nw) {
      double* qj = Qm + (long long)j * m;
      double w = 0.0;
      for (int i = k + 1 + lane; i < m; i += 32) w = fma(v[i], qj[i], w);
      w = warp_sum(w) + qj[k];
      w *= tau;
      if (lane == 0) qj[k] -= w;
      for (int i = k + 1 + lane; i < m; i += 32) qj[i] = fma(-w, v[i], qj[i]);
    }
    __syncthreads();
  }
  // sign convention diag(R) >= 0
  for (int k = wp; k < n; k += nw) {
    double d = (R[(long long)k * n + k] < 0.0) ? -1.0 : 1.0;
    __syncwarp();
    if (d < 0) {
      for (int i = lane; i < m; i += 32) Qm[(long long)k * m + i] = -Qm[(long long)k * m + i];
      for (int j = k + lane; j < n; j += 32) R[(long long)j * n + k] = -R[(long long)j * n + k];
    }
  }
}

__global__ void dot_finalize(const double* partial, int nblk, double* out) {
  __shared__ double s;
  finalize_sums(partial, nblk, 1, &s);
  __syncwarp();
  if (threadIdx.x == 0) *out = s;
}

__global__ void __launch_bounds__(VT) dot_kernel(const double* __restrict__ x, const double* __restrict__ y, long long n,
                                                 double* __restrict__ partial) {
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)VT + threadIdx.x; i < n; i += (long long)gridDim.x * VT)
    acc = fma(x[i], y[i], acc);
  __shared__ double red[VT / 32];
  double s = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < VT / 32; ++q) t += red[q];
    partial[blockIdx.x * VEC_SUMS] = t;
  }
}

// Local observables at one site: partial[b*2 + {0,1}] = sum over block b of
// A[a, pair, c] T[a, pair, c] w{n,d}(pair)  (T = EL A, right environment = 1).
__global__ void __launch_bounds__(256) local_obs_kernel(const ObsItem* __restrict__ items, const double* __restrict__ A,
                                                        const double* __restrict__ T, double* __restrict__ partial) {
  const ObsItem it = items[blockIdx.x];
  double sn = 0.0, sd = 0.0;
  const long long total = (long long)it.dl * it.m * it.dr;
  for (long long e = threadIdx.x; e < total; e += blockDim.x) {
    const int pr = (int)((e / it.dr) % it.m);
    const double v = A[it.off + e] * T[it.off + e];
    sn = fma(v, it.wn[pr], sn);
    sd = fma(v, it.wd[pr], sd);
  }
  __shared__ double red[2][8];
  sn = warp_sum(sn);
  sd = warp_sum(sd);
  if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = sn; red[1][threadIdx.x >> 5] = sd; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0, b = 0;
    for (int q = 0; q < 8; ++q) { a += red[0][q]; b += red[1][q]; }
    partial[blockIdx.x * 2] = a;
    partial[blockIdx.x * 2 + 1] = b;
  }
}

__global__ void local_obs_finalize(const double* __restrict__ partial, int n, double* __restrict__ out) {
  if (threadIdx.x != 0) return;
  double a = 0, b = 0;
  for (int i = 0; i < n; ++i) { a += partial[2 * i]; b += partial[2 * i + 1]; }
  out[0] += a;
  out[1] += b;
}

// rows of a column-major m x k matrix (ld) scaled by s[row]  /  columns scaled by s[col]
__global__ void scale_rc_kernel(double* __restrict__ a, long long ld, int rows, int cols, const double* __restrict__ s,
                                int by_col) {
  const long long total = (long long)rows * cols;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
    int r = (int)(e % rows), c = (int)(e / rows);
    a[r + c * ld] *= by_col ? s[c] : s[r];
  }
}

inline int grid_for(long long n) {
  long long g = (n + VT - 1) / VT;
  if (g > VEC_CTAS) g = VEC_CTAS;
  if (g < 1) g = 1;
  return (int)g;
}

}  // namespace

// ---------------------------------------------------------------------------
// host wrappers
// ---------------------------------------------------------------------------
cudaError_t launch_gemm_bf16(const DevGemm& g, const Bases& b, int nsplit, cudaStream_t s) {
  if (g.ntiles64 == 0) return cudaSuccess;
  if (nsplit == 2) gemm_bf16_split_kernel<2><<<g.ntiles64, 128, 0, s>>>(g.groups, g.segs, g.tiles64, b);
  else if (nsplit == 3) gemm_bf16_split_kernel<3><<<g.ntiles64, 128, 0, s>>>(g.groups, g.segs, g.tiles64, b);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

cudaError_t launch_gather(const DevGather& g, const Bases& b, int in_type, int out_type, cudaStream_t s) {
  if (g.nitems == 0) return cudaSuccess;
  if (in_type == 0 && out_type == 0) gather_kernel<0, 0><<<g.nitems, 256, 0, s>>>(g.items, g.contribs, b);
  else if (in_type == 1 && out_type == 2) gather_kernel<1, 2><<<g.nitems, 256, 0, s>>>(g.items, g.contribs, b);
  else if (in_type == 1 && out_type == 3) gather_kernel<1, 3><<<g.nitems, 256, 0, s>>>(g.items, g.contribs, b);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

cudaError_t launch_copy(const DevCopy& c, const Bases& b, cudaStream_t s) {
  if (c.nparts == 0) return cudaSuccess;
  tile_copy_kernel<0><<<c.nparts, 256, 0, s>>>(c.items, c.parts, b);
  return cudaGetLastError();
}

cudaError_t launch_split_bf16(const double* x, int64_t n, int nsplit, void* out, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  split_bf16_kernel<<<grid_for(n) * 2, VT, 0, s>>>(x, n, nsplit, reinterpret_cast<__nv_bfloat16*>(out));
  return cudaGetLastError();
}

cudaError_t launch_zero(void* p, size_t bytes, cudaStream_t s) { return cudaMemsetAsync(p, 0, bytes, s); }

cudaError_t launch_split_copy(const DevCopy& c, const Bases& b, int nsplit, cudaStream_t s) {
  if (c.nparts == 0) return cudaSuccess;
  if (nsplit == 2) tile_copy_kernel<2><<<c.nparts, 256, 0, s>>>(c.items, c.parts, b);
  else if (nsplit == 3) tile_copy_kernel<3><<<c.nparts, 256, 0, s>>>(c.items, c.parts, b);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

cudaError_t k_dot_plain(const double* x, const double* y, int64_t n, double* partial, double* out, cudaStream_t s) {
  int g = grid_for(n);
  dot_kernel<<<g, VT, 0, s>>>(x, y, n, partial);
  dot_finalize<<<1, 32, 0, s>>>(partial, g, out);
  return cudaGetLastError();
}

cudaError_t launch_local_obs(const ObsItem* items, int nitems, const double* A, const double* T, double* partial,
                             double* out, cudaStream_t s) {
  if (nitems == 0) return cudaSuccess;
  local_obs_kernel<<<nitems, 256, 0, s>>>(items, A, T, partial);
  local_obs_finalize<<<1, 32, 0, s>>>(partial, nitems, out);
  return cudaGetLastError();
}

cudaError_t launch_scale_rc(double* a, long long ld, int rows, int cols, const double* sv, int by_col, cudaStream_t s) {
  long long total = (long long)rows * cols;
  if (total == 0) return cudaSuccess;
  scale_rc_kernel<<<grid_for(total), VT, 0, s>>>(a, ld, rows, cols, sv, by_col);
  return cudaGetLastError();
}

cudaError_t launch_qr(const QrJob* jobs, int njobs, double* ws, cudaStream_t s) {
  if (njobs == 0) return cudaSuccess;
  qr_kernel<<<njobs, QRT, 0, s>>>(jobs, ws, nullptr, nullptr);
  return cudaGetLastError();
}

cudaError_t launch_qr_job(const QrJob& job, double* ws, cudaStream_t s) {
  qr_byval_kernel<<<1, QRT, 0, s>>>(job, ws);
  return cudaGetLastError();
}

cudaError_t launch_qr_masked(const QrJob* jobs, int njobs, double* ws, const int* only, int* nrun, cudaStream_t s) {
  if (njobs == 0) return cudaSuccess;
  qr_kernel<<<njobs, QRT, 0, s>>>(jobs, ws, only, nrun);
  return cudaGetLastError();
}

__global__ void plain_nrm_finalize(const double* partial, int nblk, KrylovState* ks, RhoScalars* rs) {
  __shared__ double s;
  finalize_sums(partial, nblk, 1, &s);
  __syncwarp();
  if (threadIdx.x != 0) return;
  double nrm = sqrt(s);
  ks->nrm = nrm;
  if (!isfinite(nrm) || nrm == 0.0) {
    rs->bad = 1;
    return;
  }
  rs->logscale += log(nrm);
}

cudaError_t k_normalise_inplace(double* v, int64_t n, double* partial, KrylovState* ks, RhoScalars* rs, cudaStream_t s) {
  int g = grid_for(n);
  sumsq_kernel<<<g, VT, 0, s>>>(v, n, partial);
  plain_nrm_finalize<<<1, 32, 0, s>>>(partial, g, ks, rs);
  scale_kernel<<<g, VT, 0, s>>>(v, n, &ks->nrm, nullptr, v);
  return cudaGetLastError();
}

}  // namespace tt

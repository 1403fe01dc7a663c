// Fixed-point BF16 digit operands for the exact-accumulation split GEMM
// (tt_tcgen05z.cu; Ozaki scheme, see tt_ozaki.cu for the arithmetic).
//
// A digit row holds K values v_k as four BF16 levels a0..a3 with
// v_k ~ 2^(e - 1054) (a0 2^24 + a1 2^16 + a2 2^8 + a3), e the largest biased
// FP64 exponent of the row, and e itself as an int16 next to the levels.
//  * digit_copy_kernel: FP64 rows (any row / element stride) -> digit rows
//    padded for TMA.
//  * gather_digits_kernel: the W-gather of the exact path: sums of two-float
//    (hi, lo) S1 outputs times MPO coefficients in two-float arithmetic
//    (TwoProd by FMA, TwoSum), then digits of every output row segment by
//    exact FP32 steps; two adjacent columns per lane, narrow rows packed
//    several to a warp.
// All arithmetic is FP32 / integer: GB300's FP64 pipe runs at ~1/64 of FP32.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "tt_fixed.h"
#include "tt_kernels.h"

namespace tt {

namespace {

__device__ __forceinline__ int slot_of(Ref r) { return (int)(r >> 56); }
__device__ __forceinline__ long long off_of(Ref r) { return (long long)(r & 0x00FFFFFFFFFFFFFFull); }

__device__ __forceinline__ int dexp(double v) {
  return (int)((static_cast<unsigned long long>(__double_as_longlong(v)) >> 52) & 0x7FF);
}
constexpr int DT = 256;

constexpr int GMAXC = 256;  // longest digit row (segment) of the exact path

// FP64 rows -> digit rows, one CTA per 32 rows of an item; every value is read
// once and kept in registers between the row exponent and the digits.
//   contiguous rows: a warp per row, two adjacent K per lane, so that a level's
//     store is a 32-bit word per lane;
//   strided rows (a transposed block): lanes along the rows (coalesced reads),
//     warps split K, the row exponent combined in shared memory; the digits
//     leave through shared memory, 64 K at a time (stored as computed, 2 bytes
//     to each of 32 rows, they took four times as long as the reads).
// Measured with one CTA per part instead of a grid sized by the largest item,
// and digits by byte permutes: D = 1024 site tensor and environments 32 -> 8 us
// a launch on average, D = 300 9.1 -> 4.2 us.
template <bool TOPDOWN>
__global__ void __launch_bounds__(DT) digit_copy_kernel(const DItem* __restrict__ items,
                                                        const CPart* __restrict__ parts, Bases bs) {
  const CPart part = parts[blockIdx.x];
  const DItem it = items[part.item];
  const int r0 = part.first;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double* src = reinterpret_cast<const double*>(sel_base(bs, slot_of(it.src))) + off_of(it.src);
  uint32_t* dst = reinterpret_cast<uint32_t*>(reinterpret_cast<__nv_bfloat16*>(sel_base(bs, slot_of(it.dst))) +
                                              off_of(it.dst));
  short* ex = reinterpret_cast<short*>(sel_base(bs, slot_of(it.e))) + off_of(it.e);
  const long long lo2 = sel_lo(bs, slot_of(it.dst)) / 2, drs2 = it.dst_rs / 2;  // in BF16 pairs
  constexpr int NP = GMAXC / 64;
  if (it.s_k == 1) {
    for (int q = warp; q < 32 && r0 + q < it.rows; q += DT / 32) {
      const int r = r0 + q;
      const double* sp = src + (long long)r * it.s_r;
      double v[NP][2];
      int m = 0;
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        const int k = 2 * lane + 64 * i;
        v[i][0] = k < it.cols ? sp[k] : 0.0;
        v[i][1] = k + 1 < it.cols ? sp[k + 1] : 0.0;
      }
#pragma unroll
      for (int i = 0; i < NP; ++i) m = max(m, max(dexp(v[i][0]), dexp(v[i][1])));
      m = __reduce_max_sync(0xffffffffu, m);
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        const int k = 2 * lane + 64 * i;
        if (k < it.cols) {
          uint32_t d0[4], d1[4];
          fixed_digit_bits<TOPDOWN>(v[i][0], m, d0);
          fixed_digit_bits<TOPDOWN>(v[i][1], m, d1);
#pragma unroll
          for (int lv = 0; lv < 4; ++lv) dst[lv * lo2 + r * drs2 + (k >> 1)] = __byte_perm(d0[lv], d1[lv], 0x7632);
        }
      }
      if (lane == 0) ex[(long long)r * it.e_rs] = (short)m;
    }
  } else {
    __shared__ int emax_s[32];
    __shared__ uint32_t stg[4][32][33];  // level, row, pair of K
    if (threadIdx.x < 32) emax_s[threadIdx.x] = 0;
    __syncthreads();
    const int r = r0 + lane;
    const bool in = r < it.rows;
    const double* sp = src + (long long)r * it.s_r;
    // this warp's K: 64 i + 8 warp + 0 .. 7
    double v[NP][8];
    int m = 0;
#pragma unroll
    for (int i = 0; i < NP; ++i)
      if (64 * i < it.cols) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int k = 64 * i + 8 * warp + q;
          v[i][q] = in && k < it.cols ? sp[(long long)k * it.s_k] : 0.0;
        }
      }
#pragma unroll
    for (int i = 0; i < NP; ++i)
      if (64 * i < it.cols) {
#pragma unroll
        for (int q = 0; q < 8; ++q) m = max(m, dexp(v[i][q]));
      }
    atomicMax(&emax_s[lane], m);
    __syncthreads();
    const int e = emax_s[lane];
    if (in && warp == 0) ex[(long long)r * it.e_rs] = (short)e;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      if (64 * i < it.cols) {  // (uniform)
#pragma unroll
        for (int q = 0; q < 8; q += 2) {
          uint32_t d0[4], d1[4];
          fixed_digit_bits<TOPDOWN>(v[i][q], e, d0);
          fixed_digit_bits<TOPDOWN>(v[i][q + 1], e, d1);
#pragma unroll
          for (int lv = 0; lv < 4; ++lv) stg[lv][lane][4 * warp + q / 2] = __byte_perm(d0[lv], d1[lv], 0x7632);
        }
        __syncthreads();
        const int np = min(32, (it.cols - 64 * i + 1) / 2);  // pairs with data
        for (int a = warp; a < 4 * 32; a += DT / 32) {
          const int lv = a >> 5, rr = a & 31;
          if (r0 + rr < it.rows && lane < np) dst[lv * lo2 + (r0 + rr) * drs2 + 32 * i + lane] = stg[lv][rr][lane];
        }
        __syncthreads();
      }
    }
  }
}

constexpr int GMAXK = 64;   // most MPO coefficients of one item (split in shared memory)

// One CTA per item (or share of its rows).  Each row is taken by a group of G
// lanes (G the smallest power of two with 2 G >= cols, at most 32), two adjacent
// columns per lane and PP such pairs, so that 32 / G rows share a warp when the
// item is narrow; the row exponent is a max-reduction inside the group.
//
// What bounds it: memory latency (see gather_kernel), then HBM: 8 bytes read per
// term and 8 written per element.  The term records are in shared memory, a
// warp has JR rows of PP pairs and two terms in flight (JR PP = 4), and items
// are cut by rows according to their terms, longest first.
struct GTerms {
  const float2* p[GMAXK];
  int rs[GMAXK];
  float2 f[GMAXK];  // coefficients as float pairs
};

template <int PP>
__device__ __forceinline__ void gather_rows(const GItem& it, const GTerms& t, int nk, const Bases& bs) {
  constexpr int JR = 4 / PP;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int lg = 0;
  while ((1 << lg) < 32 && 2 * (1 << lg) < it.cols) ++lg;
  const int G = 1 << lg, rpw = 32 >> lg;
  const int sub = lane >> lg, gl = lane & (G - 1);
  uint32_t* dst = reinterpret_cast<uint32_t*>(reinterpret_cast<__nv_bfloat16*>(sel_base(bs, slot_of(it.dst))) +
                                              off_of(it.dst));
  short* ex = reinterpret_cast<short*>(sel_base(bs, slot_of(it.e))) + off_of(it.e);
  const long long lo2 = sel_lo(bs, slot_of(it.dst)) / 2;  // level stride in BF16 pairs
  const int step = (DT / 32) * rpw;
  for (int rb = it.r0 + warp * rpw; rb < it.rows; rb += step * JR) {
    float h[JR][2 * PP], l[JR][2 * PP];
#pragma unroll
    for (int j = 0; j < JR; ++j)
#pragma unroll
      for (int i = 0; i < 2 * PP; ++i) { h[j][i] = 0.f; l[j][i] = 0.f; }
    auto load = [&](int k, float4 (*v)[PP]) {
#pragma unroll
      for (int j = 0; j < JR; ++j) {
        const int r = rb + sub + j * step;
        const float2* s = t.p[k] + (long long)r * t.rs[k];
        const bool al16 = (reinterpret_cast<uintptr_t>(s) & 15) == 0;
#pragma unroll
        for (int i = 0; i < PP; ++i) {
          const int c = 2 * (gl + G * i);
          float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
          if (r < it.rows && c < it.cols) {
            if (al16 && c + 1 < it.cols) {
              x = *reinterpret_cast<const float4*>(s + c);
            } else {
              const float2 v0 = s[c];
              const float2 v1 = c + 1 < it.cols ? s[c + 1] : make_float2(0.f, 0.f);
              x = make_float4(v0.x, v0.y, v1.x, v1.y);
            }
          }
          v[j][i] = x;
        }
      }
    };
    auto add = [&](int k, const float4 (*v)[PP]) {
      const float2 f = t.f[k];
#pragma unroll
      for (int j = 0; j < JR; ++j)
#pragma unroll
        for (int i = 0; i < PP; ++i) {
          df_fma(h[j][2 * i], l[j][2 * i], f.x, f.y, v[j][i].x, v[j][i].y);
          df_fma(h[j][2 * i + 1], l[j][2 * i + 1], f.x, f.y, v[j][i].z, v[j][i].w);
        }
    };
    int k = 0;
    for (; k + 1 < nk; k += 2) {
      float4 v0[JR][PP], v1[JR][PP];
      load(k, v0);
      load(k + 1, v1);
      add(k, v0);
      add(k + 1, v1);
    }
    if (k < nk) {
      float4 v0[JR][PP];
      load(k, v0);
      add(k, v0);
    }
#pragma unroll
    for (int j = 0; j < JR; ++j) {
      const int r = rb + sub + j * step;
      // renormalise every pair (TwoSum of h and l): after cancellation l may be
      // as large as h, and the digits below are taken from h and l separately
#pragma unroll
      for (int i = 0; i < 2 * PP; ++i) {
        const float sv = h[j][i] + l[j][i];
        const float bp = sv - h[j][i];
        l[j][i] = (h[j][i] - (sv - bp)) + (l[j][i] - bp);
        h[j][i] = sv;
      }
      int m = 0;
#pragma unroll
      for (int i = 0; i < PP; ++i) {
        const int c = 2 * (gl + G * i);
        if (c < it.cols) m = max(m, fexp(h[j][2 * i]));
        if (c + 1 < it.cols) m = max(m, fexp(h[j][2 * i + 1]));
      }
      for (int o = G >> 1; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
      // one exponent above the largest: |h + l| < 2^(m - 1023), so the scaled
      // values stay below 2^31 also after rounding
      if (m) m = m + 1;
      // scale 2^(1054 - m) as two exact power-of-two factors in the FP32 range
      const int sh = m ? 1054 - m : 0, sa = sh / 2, sb = sh - sa;
      const float fa = p2f(sa), fb = p2f(sb);
      if (r < it.rows) {
        uint32_t* drow = dst + ((long long)r * it.dst_rs >> 1);
#pragma unroll
        for (int i = 0; i < PP; ++i) {
          const int c = 2 * (gl + G * i);
          if (c < it.cols) {
            uint32_t d0[4], d1[4] = {0u, 0u, 0u, 0u};
            digits_of_pair((h[j][2 * i] * fa) * fb, (l[j][2 * i] * fa) * fb, d0);
            if (c + 1 < it.cols) digits_of_pair((h[j][2 * i + 1] * fa) * fb, (l[j][2 * i + 1] * fa) * fb, d1);
#pragma unroll
            for (int lv = 0; lv < 4; ++lv) drow[lv * lo2 + (c >> 1)] = __byte_perm(d0[lv], d1[lv], 0x7632);
          }
        }
        if (gl == 0) ex[(long long)r * it.e_rs] = (short)m;
      }
    }
  }
}

__global__ void __launch_bounds__(DT) gather_digits_kernel(const GItem* __restrict__ items,
                                                           const GContrib* __restrict__ cs, Bases bs) {
  const GItem it = items[blockIdx.x];
  // the item's terms, the MPO coefficients split into float pairs once per CTA
  // (FP64 arithmetic runs at ~1/64 of FP32 on GB300)
  __shared__ GTerms t;
  // the host rejects items with more terms; the clamp keeps the table in bounds
  const int nk = min(it.c1 - it.c0, GMAXK);
  for (int k = threadIdx.x; k < nk; k += DT) {
    const GContrib cb = cs[it.c0 + k];
    const float ch = (float)cb.coef;
    t.p[k] = reinterpret_cast<const float2*>(sel_base(bs, slot_of(cb.src))) + off_of(cb.src);
    t.rs[k] = (int)cb.src_rs;
    t.f[k] = make_float2(ch, (float)(cb.coef - (double)ch));
  }
  __syncthreads();
  if (it.cols <= 64) gather_rows<1>(it, t, nk, bs);
  else if (it.cols <= 128) gather_rows<2>(it, t, nk, bs);
  else gather_rows<GMAXC / 64>(it, t, nk, bs);
}

}  // namespace

cudaError_t launch_digit_copy(const DevDigit& d, const Bases& b, cudaStream_t s, bool topdown) {
  if (d.nparts == 0) return cudaSuccess;
  if (topdown) digit_copy_kernel<true><<<d.nparts, DT, 0, s>>>(d.items, d.parts, b);
  else digit_copy_kernel<false><<<d.nparts, DT, 0, s>>>(d.items, d.parts, b);
  return cudaGetLastError();
}

cudaError_t launch_gather_digits(const DevGather& g, const Bases& b, cudaStream_t s) {
  if (g.nitems == 0) return cudaSuccess;
  gather_digits_kernel<<<g.nitems, DT, 0, s>>>(g.items, g.contribs, b);
  return cudaGetLastError();
}

int gather_digits_max_cols() { return GMAXC; }
int gather_digits_max_contribs() { return GMAXK; }

}  // namespace tt

// Exact-accumulation split GEMM on the tensor cores for FP64 operands
// (Ozaki scheme: Ozaki, Ogita, Oishi, Rump, "Error-free transformations of
// matrix multiplication by using fast routines of matrix multiplication and
// its applications", Numer. Algorithms 59 (2012); here with fixed-point
// slices, as in the integer variants of that scheme).
//
// The grouped, segmented GEMM of the plans (C_g = sum over segments of
// A_seg B_seg, any transposition of A and B) reads FP64 operands directly.
// Per 32-wide K tile every row of the A tile and every column of the B tile is
// cut into four fixed-point digits relative to the largest binary exponent in
// that row (column) of the tile: v ~ 2^(e - 1054) F with the integer
// F = round(v 2^(1054 - e)), |F| <= 2^32, written as balanced base-256 digits
// F = a0 2^24 + a1 2^16 + a2 2^8 + a3, |a_s| <= 256.  The digits are exact in
// BF16, so every tensor-core product a_s b_t (|.| <= 2^16) is exact and a sum
// of at most 4 x 32 of them (< 2^24) is exact in the FP32 accumulator: the
// K tile's contribution of the digit pairs with s + t = d is an exact integer
// D_d.  The pairs with s + t <= 3 are kept (10 of 16); the tile contributes
// sum_d D_d 2^(eA + eB - 2060 - 8 d), which is added to a two-float (hi, lo)
// accumulator with TwoSum (Knuth, TAOCP vol. 2, 4.2.2) for d = 0, 1 and plain
// additions into lo for d = 2, 3.  Error: the digit truncation (<= 2^-33 of
// the row / column bound) and the dropped pairs, about 2^-32 of
// sum_k max_row |a| max_col |b| per K tile, against ~2^-24 for split-BF16
// with FP32 accumulation; no error grows with the number of K tiles beyond
// the two-float accumulation (~2^-48).
//
// The slicing is done on the fly from the FP64 operands in integer
// arithmetic (exponent and mantissa fields), because GB300's FP64 pipe runs at
// about 1/64 of its FP32 rate.  One CTA per 64 x 64 output tile, 16 warps of
// 16 x 16, mma.sync m16n8k16 (BF16 in, FP32 accumulate).
//
// Two K tiles are on their way while one is sliced and multiplied: every
// thread copies the eight values that it will slice itself (cp.async into its
// own slots, so no barrier guards them; 8-byte copies, as leading dimensions
// and offsets may be odd).  The 126 registers of a thread leave one CTA to an
// SM, so without that every K tile waited for its loads.  Lane = 8 rows x 4 K
// pairs: the digits of a pair go out as one word, and rows 20 words apart put
// stores and fragment loads into 32 banks.  Warps without a row or column of C
// neither slice nor multiply.
// What bounds it: issue slots of slicing and folding (some 30 integer operations
// a value, 25 FP32 operations an output and K tile) between the two barriers of a
// K tile.  Beta-step with loads, stores of single digits and four barriers in
// turn: D = 512 151.0 -> 148.4 ms, CL6x3 D = 1024 238.1 -> 236.3, D = 300 104.4 ->
// 102.8.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "tt_fixed.h"
#include "tt_kernels.h"

namespace tt {

namespace {

constexpr int OBM = 64, OBN = 64, OBK = 32, OPAD = 8, ODIG = 4;
constexpr int OT = 512;              // threads per CTA
constexpr int OEL = OBM * OBK / OT;  // tile elements per thread (4)
constexpr int OST = 2;               // K tiles in flight
static_assert(OEL == 4 && OBM == OBN, "part_row / pair_k");

__device__ __forceinline__ int slot_of(Ref r) { return (int)(r >> 56); }
__device__ __forceinline__ long long off_of(Ref r) { return (long long)(r & 0x00FFFFFFFFFFFFFFull); }

__device__ __forceinline__ int biased_exp(double v) {
  return (int)((static_cast<unsigned long long>(__double_as_longlong(v)) >> 52) & 0x7FF);
}

__device__ __forceinline__ void mma16816(float* c, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ void two_sum_into(float& hi, float& lo, float x) {
  const float s = hi + x;
  const float bp = s - hi;
  const float ap = s - bp;
  lo += (hi - ap) + (x - bp);
  hi = s;
}

// 2^x as a float for -126 <= x <= 127, else 0 (contributions below the FP32
// normal range are dropped; they are < 2^-126 in absolute value)
__device__ __forceinline__ float pow2f(int x) {
  return (x >= -126 && x <= 127) ? __int_as_float((x + 127) << 23) : 0.f;
}

// A thread's part of a 64 x 32 (rows x K) tile: one row, the K values
// pair_k(0), pair_k(0) + 1, pair_k(1), pair_k(1) + 1, in either storage order.
__device__ __forceinline__ int part_row(int tid) { return (tid & 7) + 8 * ((tid >> 5) & 7); }
__device__ __forceinline__ int pair_k(int tid, int i) { return 2 * (((tid >> 3) & 3) + 4 * (tid >> 8) + 8 * i); }

// dst (shared, one slot per thread, OT apart) <- the thread's values, 0 outside
__device__ __forceinline__ void copy_part(uint32_t dst, const double* __restrict__ P, long long ld, bool kmajor, int gr,
                                          int rmax, int k0, int kmax, int tid) {
#pragma unroll
  for (int i = 0; i < OEL; ++i) {
    const int gk = k0 + pair_k(tid, i >> 1) + (i & 1);
    const bool in = gr < rmax && gk < kmax;
    const double* src = in ? (kmajor ? P + (long long)gr * ld + gk : P + (long long)gk * ld + gr) : P;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(dst + i * OT * 8), "l"(src), "r"(in ? 8 : 0));
  }
}

// Largest biased exponent of each row of the tile into e[] (zeroed before): the
// four lanes of a row, then the two warps and pairs that share it.
__device__ __forceinline__ void row_exponents(const double* v, int tid, int* e) {
  int m = 0;
#pragma unroll
  for (int i = 0; i < OEL; ++i) m = max(m, biased_exp(v[i]));
  m = max(m, __shfl_xor_sync(0xffffffffu, m, 8));
  m = max(m, __shfl_xor_sync(0xffffffffu, m, 16));
  if ((tid & 31) < 8) atomicMax(&e[part_row(tid)], m);
}

// The thread's digits into a tile of ODIG x 64 x (OBK + OPAD)
template <bool TOPDOWN>
__device__ __forceinline__ void store_digits(const double* v, int emax, int tid, __nv_bfloat16* tile) {
#pragma unroll
  for (int i = 0; i < OEL; i += 2) {
    uint32_t d0[ODIG], d1[ODIG];
    fixed_digit_bits<TOPDOWN>(v[i], emax, d0);
    fixed_digit_bits<TOPDOWN>(v[i + 1], emax, d1);
    __nv_bfloat16* at = tile + part_row(tid) * (OBK + OPAD) + pair_k(tid, i >> 1);
#pragma unroll
    for (int s = 0; s < ODIG; ++s)
      *reinterpret_cast<uint32_t*>(at + s * OBM * (OBK + OPAD)) = __byte_perm(d0[s], d1[s], 0x7632);
  }
}

struct OzShared {
  double raw[OST][2][OEL * OT];  // [stage][A, B][value][thread]
  __nv_bfloat16 As[ODIG][OBM][OBK + OPAD];
  __nv_bfloat16 Bs[ODIG][OBN][OBK + OPAD];
  int eA[2][OBM], eB[2][OBN];
};

template <bool TOPDOWN>
__global__ void __launch_bounds__(OT) gemm_oz_kernel(const GGroup* __restrict__ groups, const GSeg* __restrict__ segs,
                                                      const GTile* __restrict__ tiles, Bases bs) {
  extern __shared__ __align__(16) unsigned char oz_smem[];
  OzShared& sh = *reinterpret_cast<OzShared*>(oz_smem);
  const GTile tl = tiles[blockIdx.x];
  const GGroup g = groups[tl.g];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = (warp >> 2) * 16, wn = (warp & 3) * 16;
  const int gid = lane >> 2, tig = lane & 3;
  const bool rows_a = tl.m0 + 8 * (warp & 7) < g.M, rows_b = tl.n0 + 8 * (warp & 7) < g.N;
  const bool live = tl.m0 + wm < g.M && tl.n0 + wn < g.N;

  float acc[ODIG][2][4], hi[2][4], lo[2][4];
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      hi[j][r] = 0.f;
      lo[j][r] = 0.f;
#pragma unroll
      for (int d = 0; d < ODIG; ++d) acc[d][j][r] = 0.f;
    }

  // the next K tile to fetch
  int fs = g.seg0, fk = 0;
  auto fetch = [&](int stage) {
    while (fs < g.seg1 && segs[fs].K <= fk) {
      ++fs;
      fk = 0;
    }
    if (fs < g.seg1) {
      const GSeg sg = segs[fs];
      const double* A = reinterpret_cast<const double*>(sel_base(bs, slot_of(sg.A))) + off_of(sg.A);
      const double* B = reinterpret_cast<const double*>(sel_base(bs, slot_of(sg.B))) + off_of(sg.B);
      // A logical M x K: stored M x K (tA = 0, K contiguous) or K x M (tA = 1);
      // B logical N x K: stored N x K (tB = 1) or K x N (tB = 0)
      const int row = part_row(tid);
      copy_part((uint32_t)__cvta_generic_to_shared(&sh.raw[stage][0][tid]), A, sg.lda, sg.tA == 0, tl.m0 + row, g.M, fk,
                sg.K, tid);
      copy_part((uint32_t)__cvta_generic_to_shared(&sh.raw[stage][1][tid]), B, sg.ldb, sg.tB == 1, tl.n0 + row, g.N, fk,
                sg.K, tid);
      fk += OBK;
    }
    asm volatile("cp.async.commit_group;\n");
  };
  int ntile = 0;
  for (int si = g.seg0; si < g.seg1; ++si) ntile += (segs[si].K + OBK - 1) / OBK;
  if (tid < OBM) sh.eA[0][tid] = 0;
  else if (tid < OBM + OBN) sh.eB[0][tid - OBM] = 0;
#pragma unroll
  for (int i = 0; i < OST; ++i) fetch(i);
  __syncthreads();

  for (int t0 = 0, cur = 0, stage = 0; t0 < ntile; ++t0, cur ^= 1, stage = stage + 1 == OST ? 0 : stage + 1) {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(OST - 1) : "memory");
    double va[OEL], vb[OEL];
#pragma unroll
    for (int i = 0; i < OEL; ++i) {
      va[i] = sh.raw[stage][0][i * OT + tid];
      vb[i] = sh.raw[stage][1][i * OT + tid];
    }
    if (rows_a) row_exponents(va, tid, sh.eA[cur]);
    if (rows_b) row_exponents(vb, tid, sh.eB[cur]);
    __syncthreads();  // exponents complete; every warp done with the last tile's digits
    if (tid < OBM) sh.eA[cur ^ 1][tid] = 0;
    else if (tid < OBM + OBN) sh.eB[cur ^ 1][tid - OBM] = 0;
    if (rows_a) store_digits<TOPDOWN>(va, sh.eA[cur][part_row(tid)], tid, &sh.As[0][0][0]);
    if (rows_b) store_digits<TOPDOWN>(vb, sh.eB[cur][part_row(tid)], tid, &sh.Bs[0][0][0]);
    fetch(stage);  // the values are in registers
    __syncthreads();
    if (!live) continue;
#pragma unroll
    for (int ks = 0; ks < OBK; ks += 16) {
      uint32_t af[ODIG][4];
#pragma unroll
      for (int s = 0; s < ODIG; ++s) {
        const int r0 = wm + gid;
        af[s][0] = *reinterpret_cast<const uint32_t*>(&sh.As[s][r0][ks + 2 * tig]);
        af[s][1] = *reinterpret_cast<const uint32_t*>(&sh.As[s][r0 + 8][ks + 2 * tig]);
        af[s][2] = *reinterpret_cast<const uint32_t*>(&sh.As[s][r0][ks + 8 + 2 * tig]);
        af[s][3] = *reinterpret_cast<const uint32_t*>(&sh.As[s][r0 + 8][ks + 8 + 2 * tig]);
      }
#pragma unroll
      for (int t = 0; t < ODIG; ++t) {
        uint32_t bf[2][2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int c0 = wn + 8 * j + gid;
          bf[j][0] = *reinterpret_cast<const uint32_t*>(&sh.Bs[t][c0][ks + 2 * tig]);
          bf[j][1] = *reinterpret_cast<const uint32_t*>(&sh.Bs[t][c0][ks + 8 + 2 * tig]);
        }
#pragma unroll
        for (int s = 0; s + t < ODIG; ++s)
#pragma unroll
          for (int j = 0; j < 2; ++j) mma16816(acc[s + t][j], af[s], bf[j]);
      }
    }
    // fold this K tile: D_d 2^(eA + eB - 2060 - 8 d) into (hi, lo)
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int m = wm + gid + ((r >= 2) ? 8 : 0);
        const int n = wn + 8 * j + 2 * tig + (r & 1);
        const int x = sh.eA[cur][m] + sh.eB[cur][n] - 2060;
        two_sum_into(hi[j][r], lo[j][r], acc[0][j][r] * pow2f(x));
        two_sum_into(hi[j][r], lo[j][r], acc[1][j][r] * pow2f(x - 8));
        lo[j][r] += acc[2][j][r] * pow2f(x - 16) + acc[3][j][r] * pow2f(x - 24);
#pragma unroll
        for (int d = 0; d < ODIG; ++d) acc[d][j][r] = 0.f;
      }
  }
  const bool accum = g.flags & 1;
  const bool out_f32 = g.flags & 2;
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int gm = tl.m0 + wm + gid + ((r >= 2) ? 8 : 0);
      const int gn = tl.n0 + wn + 8 * j + 2 * tig + (r & 1);
      if (gm >= g.M || gn >= g.N) continue;
      const long long o = (long long)gm * g.ldc + gn;
      const double v = (double)hi[j][r] + (double)lo[j][r];
      if (out_f32) {
        float* C = reinterpret_cast<float*>(sel_base(bs, slot_of(g.C))) + off_of(g.C) + o;
        *C = accum ? *C + (float)v : (float)v;
      } else {
        double* C = reinterpret_cast<double*>(sel_base(bs, slot_of(g.C))) + off_of(g.C) + o;
        *C = accum ? *C + v : v;
      }
    }
}

}  // namespace

cudaError_t launch_gemm_oz(const DevGemm& g, const Bases& b, cudaStream_t s, bool topdown) {
  if (g.ntiles64 == 0) return cudaSuccess;
  // 107 KB of shared memory; set on every call, as the attribute is per device
  auto run = [&](auto kernel) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(OzShared));
    if (e != cudaSuccess) return e;
    kernel<<<g.ntiles64, OT, sizeof(OzShared), s>>>(g.groups, g.segs, g.tiles64, b);
    return cudaGetLastError();
  };
  return topdown ? run(gemm_oz_kernel<true>) : run(gemm_oz_kernel<false>);
}

}  // namespace tt

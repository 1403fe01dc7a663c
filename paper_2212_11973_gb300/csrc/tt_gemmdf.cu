// Grouped GEMM in double-float arithmetic on the FP32 pipe: the mixed modes'
// CholeskyQR Gram and apply products, and the environment updates with
// env_precision 2.
//
// FP64 operands are split into float pairs (hi, lo) as they are staged, every
// product is formed by the FMA TwoProduct with the cross terms, every sum by
// TwoSum into an unnormalised (hi, lo) accumulator (Dekker; Knuth TAOCP vol. 2,
// 4.2.2): ~2^-46 relative per operation, K 2^-46 of sum |a| |b| per output.
// Output FP64.
//
// What bounds it: 12 FP32 operations per multiply-add, 10.7 multiply-adds per
// clock and SM against 2 on the FP64 pipe (or the FP64 tensor instruction), and
// enough tiles to go round: a gauge move at D = 1024 has 80 tiles of 64 x 64 and K
// = 467, which occupied half of the SMs for 90 us each.  So tiles are 32 x 32 with
// 8 outputs per thread, two chunks of 16 K in shared memory (the next one's loads
// in flight during the products), and parts of a tile outside the group (rows by
// 16, columns by 8) are skipped.  A chain of K chunks still takes ~150 clocks per
// K, so the gauge takes the FP64 kernel where that has less to do (df_beats_f64).
// Measured per launch, double-float against FP64: D = 1024 103 and 216 us, D =
// 512 90 and 38, D = 300 70 and 12.
#include <cuda_runtime.h>

#include <cstdint>

#include "tt_df.h"
#include "tt_kernels.h"

namespace tt {

namespace {

constexpr int DM = 32, DN = 32, DK = 16, DTH = 128;

__device__ __forceinline__ int slot_of(Ref r) { return (int)(r >> 56); }
__device__ __forceinline__ long long off_of(Ref r) { return (long long)(r & 0x00FFFFFFFFFFFFFFull); }

__global__ void __launch_bounds__(DTH) gemm_df_kernel(const FTile* __restrict__ tiles, const GSeg* __restrict__ segs,
                                                      Bases bs, bool exact_out) {
  __shared__ float2 As[2][DK][DM + 1];
  __shared__ float2 Bs[2][DK][DN + 1];
  const FTile tl = tiles[blockIdx.x];
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;  // rows ty, ty + 16; columns tx + 8 j
  float hi[2][4], lo[2][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) hi[i][j] = lo[i][j] = 0.f;

  // the chunk after the current one: segment, its operands and first K
  int si = tl.seg0, k0 = 0;
  double va[4], vb[4];
  bool ka = true, kb = true;
  // four elements of each operand per thread, coalesced for either storage order
  auto row_of = [&](bool kmajor, int i) { return kmajor ? (tid + DTH * i) / DK : (tid + DTH * i) % DM; };
  auto k_of = [&](bool kmajor, int i) { return kmajor ? (tid + DTH * i) % DK : (tid + DTH * i) / DM; };
  auto load = [&]() {
    const GSeg sg = segs[si];
    ka = sg.tA == 0;
    kb = sg.tB == 1;
    const double* A = reinterpret_cast<const double*>(sel_base(bs, slot_of(sg.A))) + off_of(sg.A);
    const double* B = reinterpret_cast<const double*>(sel_base(bs, slot_of(sg.B))) + off_of(sg.B);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int ra = row_of(ka, i), qa = k0 + k_of(ka, i), rb = row_of(kb, i), qb = k0 + k_of(kb, i);
      va[i] = ra < tl.rows && qa < sg.K
                  ? A[ka ? (long long)(tl.m0 + ra) * sg.lda + qa : (long long)qa * sg.lda + tl.m0 + ra]
                  : 0.0;
      vb[i] = rb < tl.cols && qb < sg.K
                  ? B[kb ? (long long)(tl.n0 + rb) * sg.ldb + qb : (long long)qb * sg.ldb + tl.n0 + rb]
                  : 0.0;
    }
    k0 += DK;
    if (k0 >= sg.K) {
      k0 = 0;
      ++si;
    }
  };
  auto stage = [&](int b) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      As[b][k_of(ka, i)][row_of(ka, i)] = df_split(va[i]);
      Bs[b][k_of(kb, i)][row_of(kb, i)] = df_split(vb[i]);
    }
  };
  if (si < tl.seg1) {
    load();
    stage(0);
    __syncthreads();
    for (int b = 0;; b ^= 1) {
      const bool more = si < tl.seg1;
      if (more) load();
#pragma unroll 4
      for (int kk = 0; kk < DK; ++kk) {
        float2 a[2], c[4];
#pragma unroll
        for (int i = 0; i < 2; ++i) a[i] = As[b][kk][ty + 16 * i];
#pragma unroll
        for (int j = 0; j < 4; ++j) c[j] = Bs[b][kk][tx + 8 * j];
#pragma unroll
        for (int i = 0; i < 2; ++i)
          if (16 * i < tl.rows) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (8 * j < tl.cols) {
                const float p = a[i].x * c[j].x;
                float e = fmaf(a[i].x, c[j].x, -p);
                e = fmaf(a[i].x, c[j].y, e);
                e = fmaf(a[i].y, c[j].x, e);
                const float s = hi[i][j] + p;
                const float bp = s - hi[i][j];
                lo[i][j] += ((hi[i][j] - (s - bp)) + (p - bp)) + e;
                hi[i][j] = s;
              }
          }
      }
      if (!more) break;
      stage(b ^ 1);  // (read last before the previous barrier)
      __syncthreads();
    }
  }
  double* C = reinterpret_cast<double*>(sel_base(bs, slot_of(tl.C))) + off_of(tl.C);
  const bool accum = tl.flags & 1;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = ty + 16 * i, q = tx + 8 * j;
      if (r >= tl.rows || q >= tl.cols) continue;
      double* c = C + (long long)r * tl.ldc + q;
      const double v = exact_out ? (double)hi[i][j] + (double)lo[i][j] : dbl_of_pair(hi[i][j], lo[i][j]);
      *c = accum ? *c + v : v;
    }
}

}  // namespace

int df_tile_size() { return DM; }

bool df_beats_f64(const GemmPlan& p) {
  // clocks: the FP64 kernel keeps every SM busy at 2 multiply-adds, with 1.3 for
  // its imbalance; this one its share of the tiles at 10.7, but at least one tile's
  // chain, ~150 per K with one warp on each scheduler, times 1.5 and with 20000 for
  // filling its pipeline (D = 300, K = 53: 23 us where the products alone take 4)
  double f64 = 0, df = 0, chain = 0;
  for (const GGroup& g : p.groups) {
    double k = 0;
    for (int s = g.seg0; s < g.seg1; ++s) k += p.segs[s].K;
    f64 += ((g.M + 7) / 8 * 8) * (double)((g.N + 7) / 8 * 8) * k / 2;
    df += ((g.M + DM - 1) / DM) * (double)((g.N + DN - 1) / DN) * k * (DM * DN * 12 / 128);
    chain = k > chain ? k : chain;
  }
  const double td = df / 152;
  return 1.5 * (td > 150 * chain ? td : 150 * chain) + 20000 < 1.3 * f64 / 152 + 5000;
}

cudaError_t launch_gemm_df(const DevGemm& g, const Bases& b, cudaStream_t s, bool exact_out) {
  if (g.ntilesd == 0) return cudaSuccess;
  gemm_df_kernel<<<g.ntilesd, DTH, 0, s>>>(g.tilesd, g.segs, b, exact_out);
  return cudaGetLastError();
}

}  // namespace tt

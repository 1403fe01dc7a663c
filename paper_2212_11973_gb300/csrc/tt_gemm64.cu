// FP64 grouped GEMM on the FP64 tensor instruction (mma.sync m8n8k4): every
// FP64 contraction of the sweep (H_eff, bond, environment and absorb plans of
// the FP64 mode, the measurement and the QR factors of every mode).
//
// What bounds it: GB300 executes 2 FP64 multiply-adds per clock and SM, by
// DFMA and by DMMA alike (measured: one m8n8k4 per 512 clocks and SM sub-
// partition), 1.2 TFLOP/s in all.  Memory and latency hide behind that with a
// few warps, so what counts is (1) no multiply-adds on padding and (2) the
// same amount of work for each of the 608 sub-partitions.  Sectors have 3 to
// 200 states, so the tile is cut into 8 x 8 blocks and blocks outside the
// group are skipped, K is padded only to the next multiple of 4, and the four
// warps of a CTA (one per sub-partition) take every fourth K step of one
// T x T tile and are summed in warp order at the end (deterministic).  A
// fragment comes straight from global memory into registers (32 or 64
// contiguous bytes per row; 4 B per clock and SM at T = 8), prefetched a few
// steps ahead across segment boundaries; no shared memory, no barrier in the
// loop.
//
// T and the number of warps on a tile are chosen per plan (f64_shape): the
// largest of 32, 16, 8 whose longest tile is at most a quarter of one SM's (or,
// for one-warp tiles, one sub-partition's) share of the plan.  Where no K is
// above 128 a tile belongs to one warp: splitting 3 to 12 K steps over four
// warps leaves some of them idle, and the sum of the four shares costs as much
// FP64 work as 3 of the K steps' multiply-adds per output.
//
// Measured against 64 x 64 DFMA tiles with a K loop per CTA (which padded a
// sector of 12 to 64 and left most SMs idle behind a few long tiles): FP64
// beta-step of a 4x8 cylinder at D = 256 961 -> 162 ms (140 -> 135 ms by the
// one-warp tiles later), of the 2x2 cluster at D = 64 24.3 -> 5.4 ms;
// measurement and QR factors of a D = 300 exact-split step 249 -> 217 ms.  The
// smaller CholeskyQR products of the mixed modes run here too (df_beats_f64
// draws the line): double-float on 64 x 64 tiles took 31 ms of a D = 300 step
// and 43 of a D = 512 one, here 4 and 10.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "tt_kernels.h"

namespace tt {

namespace {

__device__ __forceinline__ int slot_of(Ref r) { return (int)(r >> 56); }
__device__ __forceinline__ long long off_of(Ref r) { return (long long)(r & 0x00FFFFFFFFFFFFFFull); }

__device__ __forceinline__ void dmma(double* c, double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
               : "+d"(c[0]), "+d"(c[1])
               : "d"(a), "d"(b));
}

// K steps (4 deep) of one warp: steps wk, wk + WK, ... counted through all
// segments of the tile
struct KIter {
  const GSeg* segs;
  const Bases* bs;
  int si, seg1, t, n4, K, s0, wk;
  const double *pa, *pb;          // this lane's first element of the segment
  long long ars, brs, aks, bks;   // strides along the tile row / column and K
  int lr, lk, m0, n0;

  template <int WK>
  __device__ __forceinline__ void open() {
    const GSeg sg = segs[si];
    K = sg.K;
    n4 = (K + 3) >> 2;
    ars = sg.tA ? 1 : sg.lda;
    aks = sg.tA ? sg.lda : 1;
    brs = sg.tB ? sg.ldb : 1;
    bks = sg.tB ? 1 : sg.ldb;
    pa = reinterpret_cast<const double*>(sel_base(*bs, slot_of(sg.A))) + off_of(sg.A) + (m0 + lr) * ars + lk * aks;
    pb = reinterpret_cast<const double*>(sel_base(*bs, slot_of(sg.B))) + off_of(sg.B) + (n0 + lr) * brs + lk * bks;
    t = (wk - s0) & (WK - 1);
  }
  // position on this warp's next step; false past the end
  template <int WK>
  __device__ __forceinline__ bool settle() {
    while (t >= n4) {
      s0 += n4;
      if (++si >= seg1) return false;
      open<WK>();
    }
    return true;
  }
};

template <int NB>
struct Frag {
  double a[NB], b[NB];
};

template <int T, int PF, int WK>
__global__ void __launch_bounds__(128) gemm_f64_kernel(const FTile* __restrict__ tiles, int ntiles,
                                                       const GSeg* __restrict__ segs, Bases bs) {
  constexpr int NB = T / 8;
  constexpr int LD = T + (T > 8 ? 4 : 0);  // staging row (bank spread of the double2 stores)
  __shared__ __align__(16) double red[WK == 1 ? 1 : 4][WK == 1 ? 2 : T * LD];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ti = WK == 1 ? blockIdx.x * 4 + warp : blockIdx.x;
  if (WK == 1 && ti >= ntiles) return;
  const FTile tl = tiles[ti];
  const int lr = lane >> 2, lk = lane & 3;
  const int mb = (tl.rows + 7) >> 3, nb = (tl.cols + 7) >> 3;  // 8 x 8 blocks in use (uniform)
  double acc[NB][NB][2];
#pragma unroll
  for (int i = 0; i < NB; ++i)
#pragma unroll
    for (int j = 0; j < NB; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;

  if (tl.seg0 < tl.seg1) {
    KIter it;
    it.segs = segs;
    it.bs = &bs;
    it.si = tl.seg0;
    it.seg1 = tl.seg1;
    it.s0 = 0;
    it.wk = WK == 1 ? 0 : warp;
    it.lr = lr;
    it.lk = lk;
    it.m0 = tl.m0;
    it.n0 = tl.n0;
    it.open<WK>();
    Frag<NB> f[PF];
    bool ok[PF];
    auto load = [&](Frag<NB>& q) {
      const bool kin = 4 * it.t + lk < it.K;
      const double* a = it.pa + (long long)(4 * it.t) * it.aks;
      const double* b = it.pb + (long long)(4 * it.t) * it.bks;
#pragma unroll
      for (int i = 0; i < NB; ++i) q.a[i] = (kin && 8 * i + lr < tl.rows) ? a[8 * i * it.ars] : 0.0;
#pragma unroll
      for (int j = 0; j < NB; ++j) q.b[j] = (kin && 8 * j + lr < tl.cols) ? b[8 * j * it.brs] : 0.0;
      it.t += WK;
    };
#pragma unroll
    for (int p = 0; p < PF; ++p) {
      ok[p] = it.si < it.seg1 && it.settle<WK>();
      if (ok[p]) load(f[p]);
    }
    bool more = ok[0];
    while (more) {
#pragma unroll
      for (int p = 0; p < PF; ++p) {
        if (!ok[p]) {
          more = false;
          break;
        }
#pragma unroll
        for (int i = 0; i < NB; ++i)
#pragma unroll
          for (int j = 0; j < NB; ++j)
            if (i < mb && j < nb) dmma(acc[i][j], f[p].a[i], f[p].b[j]);
        ok[p] = it.si < it.seg1 && it.settle<WK>();
        if (ok[p]) load(f[p]);
      }
    }
  }
  double* C = reinterpret_cast<double*>(sel_base(bs, slot_of(tl.C))) + off_of(tl.C);
  const bool accum = tl.flags & 1;
  if (WK == 1) {
#pragma unroll
    for (int i = 0; i < NB; ++i)
#pragma unroll
      for (int j = 0; j < NB; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int r = 8 * i + lr, c = 8 * j + 2 * lk + h;
          if (r >= tl.rows || c >= tl.cols) continue;
          double* p = C + (long long)r * tl.ldc + c;
          *p = accum ? *p + acc[i][j][h] : acc[i][j][h];
        }
    return;
  }
  // the four K shares summed in warp order, rows written along their columns
#pragma unroll
  for (int i = 0; i < NB; ++i)
#pragma unroll
    for (int j = 0; j < NB; ++j)
      *reinterpret_cast<double2*>(&red[warp][(8 * i + lr) * LD + 8 * j + 2 * lk]) =
          make_double2(acc[i][j][0], acc[i][j][1]);
  __syncthreads();
  for (int e = threadIdx.x; e < T * T; e += 128) {
    const int r = e / T, c = e % T;
    if (r >= tl.rows || c >= tl.cols) continue;
    const int o = r * LD + c;
    const double v = ((red[0][o] + red[1][o]) + red[2][o]) + red[3][o];
    double* p = C + (long long)r * tl.ldc + c;
    *p = accum ? *p + v : v;
  }
}

}  // namespace

F64Shape f64_shape(const GemmPlan& p) {
  // clocks of one SM: 2 multiply-adds each
  double total = 0, kmax = 0;
  for (const GGroup& g : p.groups) {
    double k = 0;
    for (int s = g.seg0; s < g.seg1; ++s) k += (p.segs[s].K + 3) / 4 * 4;
    total += 0.5 * ((g.M + 7) / 8 * 8) * (double)((g.N + 7) / 8 * 8) * k;
    kmax = std::max(kmax, k);
  }
  const double share = total / 152;
  if (kmax <= 128)
    for (int T : {16, 8})
      if (4 * 4 * 0.5 * T * T * kmax <= share) return {T, 1};
  for (int T : {32, 16})
    if (4 * 0.5 * T * T * kmax <= share) return {T, 4};
  return {8, 4};
}

// (16 x 16 where that gives every SM sub-partition a tile)
F64Shape f64_shape_ordered(const GemmPlan& p) {
  size_t tiles = 0;
  for (const GGroup& g : p.groups) tiles += (size_t)((g.M + 15) / 16) * ((g.N + 15) / 16);
  return {tiles >= 4 * 152 ? 16 : 8, 1};
}

std::vector<FTile> f64_tiles(const GemmPlan& p, int T) {
  std::vector<std::pair<int, int>> order;  // longest K first
  for (size_t g = 0; g < p.groups.size(); ++g) {
    int k = 0;
    for (int s = p.groups[g].seg0; s < p.groups[g].seg1; ++s) k += p.segs[s].K;
    order.push_back({-k, (int)g});
  }
  std::stable_sort(order.begin(), order.end());
  std::vector<FTile> out;
  for (auto& og : order) {
    const GGroup& g = p.groups[og.second];
    for (int m0 = 0; m0 < g.M; m0 += T)
      for (int n0 = 0; n0 < g.N; n0 += T)
        out.push_back(FTile{g.C + (Ref)((int64_t)m0 * g.ldc + n0), m0, n0, std::min(T, g.M - m0), std::min(T, g.N - n0),
                            g.seg0, g.seg1, g.ldc, g.flags});
  }
  return out;
}

cudaError_t launch_gemm_f64(const DevGemm& g, const Bases& b, cudaStream_t s) {
  if (g.ntilesf == 0) return cudaSuccess;
  const int gw = (g.ntilesf + 3) / 4;
  if (g.tf == 32) gemm_f64_kernel<32, 1, 4><<<g.ntilesf, 128, 0, s>>>(g.tilesf, g.ntilesf, g.segs, b);
  else if (g.tf == 16 && g.wkf == 1) gemm_f64_kernel<16, 2, 1><<<gw, 128, 0, s>>>(g.tilesf, g.ntilesf, g.segs, b);
  else if (g.tf == 16) gemm_f64_kernel<16, 2, 4><<<g.ntilesf, 128, 0, s>>>(g.tilesf, g.ntilesf, g.segs, b);
  else if (g.tf == 8 && g.wkf == 1) gemm_f64_kernel<8, 4, 1><<<gw, 128, 0, s>>>(g.tilesf, g.ntilesf, g.segs, b);
  else if (g.tf == 8) gemm_f64_kernel<8, 4, 4><<<g.ntilesf, 128, 0, s>>>(g.tilesf, g.ntilesf, g.segs, b);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

}  // namespace tt

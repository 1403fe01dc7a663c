// Persistent, warp-specialised split-BF16 grouped GEMM on the 5th-generation
// tensor cores (sm_103a): operands as NS bf16 levels, the level products l_A +
// l_B < NS, folded every two pieces of at most 64 of K into a two-float TwoSum sum.
//
// Laid out as the digit kernel (tt_tcgen05z.cu): one CTA per SM walks 128 x 64
// output tiles; warp 0 streams the level tiles by TMA into a ring of
// shared-memory stages (K chunks of 64, or of 32 where no segment is longer than
// 128), warp 1 issues the MMAs, warps 2-9 fold a finished accumulator while the
// next fold group's MMAs run in the other buffer, and write the tile's hi + lo
// as FP32 or FP64 through a per-warp staging buffer.  The products of one order
// d = l_A + l_B share an accumulator (D_0 .. D_{NS-1}, 64 TMEM columns each), so
// level l of A meets the B levels 0 .. NS-1-l, which lie one after the other, in
// one MMA of N = 64 (NS - l).  D_0 goes through TwoSum, the smaller orders into
// lo.  Where a plan has fewer tiles than SMs, `split` CTAs share a tile's
// segments and the last to arrive adds their sums in part order.
//
// What bounds it: the chain of segments (18 to 42 of K = 3 to 180) behind each
// tile; see the digit kernel.  D = 512, all four launches of an H_eff and a bond
// apply, average: 29 -> 25 us from one lane fencing and loading each segment's
// maps, K chunks of 64 throughout, six MMAs per 16 K and rows stored as they came
// (S1, whose tiles have one segment each and are bound by their output, 23 us; with
// the shared-memory reads of the output one by one it took 40).
//
// Every wait is bounded by wait_ns; a role whose wait runs out raises a shared
// abort flag that the other roles' waits observe, the CTA records the error,
// drains its own TMA copies and MMAs (fixed budget), frees its TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "tt_df.h"
#include "tt_kernels.h"
#include "tt_tc_ptx.h"

namespace tt {

namespace {

using namespace tcx;

constexpr int PBM = 128, PBN = 64, PIECE = 64;  // two pieces to a fold group
constexpr uint32_t PTMEM_COLS = 512;
constexpr int PEPI = 8;  // epilogue warps
constexpr int PTHREADS = 64 + 32 * PEPI;
constexpr int PSTG_WARP = 16 * 16;  // staging per epilogue warp: 16 rows x 16 columns of 8 bytes
constexpr int PSTG_BYTES = PEPI * PSTG_WARP * 8;
constexpr size_t PSMEM = 222 * 1024;  // dynamic shared memory (the item table is static)

template <int NS, int BK>
struct PCfg {
  static constexpr int A_BYTES = PBM * BK * 2, B_BYTES = PBN * BK * 2;  // per level
  static constexpr int STAGE_BYTES = NS * (A_BYTES + B_BYTES);
  static constexpr int STAGES = (int)((PSMEM - PSTG_BYTES - 1024) / STAGE_BYTES);
};

// Pieces (at most PIECE of K each, within a segment) of the tile part: the sum over
// its segments, by the whole warp
__device__ __forceinline__ int part_pieces(const TileItem& q, const GSeg* segs) {
  if (q.n <= 1) return (q.K0 + PIECE - 1) / PIECE;
  int t = 0;
  for (int s = threadIdx.x & 31; s < q.n; s += 32) t += (segs[q.seg(s)].K + PIECE - 1) / PIECE;
  return __reduce_add_sync(0xffffffffu, t);
}

// OUT32: every group of the launch writes FP32 (flags bit 1), else FP64.
// BYLEVEL (BK = 64): the order of a padded state's first beta-step (tt_settle.cu):
// the level products of a piece one after the other, those of order 0 into one
// accumulator and all others into a second, both folded by one formula.
template <int NS, int BK, bool OUT32, bool BYLEVEL>
__global__ void __launch_bounds__(PTHREADS, 1) gemm_tcp_kernel(const GGroup* __restrict__ groups,
                                                               const GSeg* __restrict__ segs,
                                                               const GTile* __restrict__ tiles, int nitems, int split,
                                                               const CUtensorMap* __restrict__ maps, Bases bs,
                                                               uint64_t* __restrict__ scratch,
                                                               unsigned* __restrict__ tickets, int* __restrict__ err,
                                                               long long wait_ns) {
  using C = PCfg<NS, BK>;
  constexpr int S = C::STAGES;
  constexpr int BUF = 64 * NS;                       // TMEM columns of one accumulator buffer
  static_assert(S >= 2 && 2 * BUF <= (int)PTMEM_COLS && (!BYLEVEL || BK == PIECE), "stages and accumulators");
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[S], empty_bar[S], accf[2], acce[2];
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s, issued_s, consumed_s, last_commit_s, last_accf_s;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  volatile int* abort_f = &abort_s;
  __shared__ TileItem table[TITEMS];

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // the CTA's i-th item, in shared memory (beyond the table in a slot of the warp;
  // an item and its successor may be in use together)
  __shared__ TileItem own[(PTHREADS / 32)][2];
  auto item = [&](int i) -> const TileItem& {
    if (i < TITEMS) return table[i];
    TileItem& o = own[warp][i & 1];
    __syncwarp();
    if (lane == 0) o = load_item(groups, segs, tiles, bs, (OUT32 ? 4 : 8), blockIdx.x + i * gridDim.x, split);
    __syncwarp();
    return o;
  };
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)),
                 "r"(PTMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 32) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], PEPI);
    }
    abort_s = 0;
    issued_s = 0;
    consumed_s = 0;
    last_commit_s = -1;
    last_accf_s = -1;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  int kl0 = 0;
  if (warp == 0) kl0 = first_segments(groups, segs, tiles, maps, split);
  else load_items(table, groups, segs, tiles, maps, bs, (OUT32 ? 4 : 8), nitems, split);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_base_s;

  if (warp == 0) {
    // ---------------- producer ----------------
    int it = 0;
    bool stop = false;  // the abort flag, read once for the whole warp: lanes that saw
                        // it at different times would wait for each other in item()
    for (int i = 0; blockIdx.x + i * gridDim.x < nitems && !stop; ++i) {
      const TileItem& q = item(i);
      for (int s0 = 0; s0 < q.n && !stop; s0 += 32) {
        int kl = q.K0;
        if (i == 0 && s0 == 0) {
          kl = kl0;
        } else if (q.n > 1 || i >= TITEMS) {
          const int sl = q.seg(min(s0 + lane, q.n - 1));
          kl = segs[sl].K;
          fence_maps(maps, sl);
          __syncwarp();
        }
        for (int s = s0; s < min(q.n, s0 + 32) && !stop; ++s) {
          const int K = __shfl_sync(0xffffffffu, kl, s - s0);
          if (lane == 0) {
            const CUtensorMap* ma = maps + 4 * q.seg(s) + 3;
            const CUtensorMap* mb = ma - 1;
            for (int k0 = 0; k0 < K; k0 += BK) {
              const int sg = it % S;
              if (!wait_ab(&empty_bar[sg], ((it / S) & 1) ^ 1, wait_ns, abort_f, err)) break;
              uint8_t* st = smem + sg * C::STAGE_BYTES;
              mbar_expect_tx(&full_bar[sg], C::STAGE_BYTES);
#pragma unroll
              for (int l = 0; l < NS; ++l) tma_load_3d(st + l * C::A_BYTES, ma, k0, q.m0, l, &full_bar[sg]);
#pragma unroll
              for (int l = 0; l < NS; ++l)
                tma_load_3d(st + NS * C::A_BYTES + l * C::B_BYTES, mb, k0, q.n0, l, &full_bar[sg]);
              ++it;
              issued_s = it;
            }
          }
          stop = __any_sync(0xffffffffu, *abort_f);
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    constexpr uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(PBM >> 4) << 24);
    int it = 0, fg = 0;
    bool ok = true;
    for (int i = 0; blockIdx.x + i * gridDim.x < nitems && ok; ++i) {
      const TileItem& q = item(i);
      int kl = q.K0, c = 0;  // c: piece within the part
      const int T = part_pieces(q, segs);
      for (int s = 0; s < q.n && ok; ++s) {
        if ((s & 31) == 0 && q.n > 1) kl = segs[q.seg(min(s + lane, q.n - 1))].K;
        const int K = __shfl_sync(0xffffffffu, kl, s & 31);
        if (lane == 0) {
          for (int k0 = 0; k0 < K && ok; k0 += BK) {
            const int b = fg & 1;
            const bool first = (c & 1) == 0 && k0 % PIECE == 0;
            if (first) {
              ok = wait_ab(&acce[b], ((fg >> 1) & 1) ^ 1, wait_ns, abort_f, err);
              if (!ok) break;
            }
            const int sg = it % S;
            ok = wait_ab(&full_bar[sg], (it / S) & 1, wait_ns, abort_f, err);
            if (!ok) break;
            consumed_s = it + 1;
            fence_after();
            const uint32_t tb = tmem + BUF * b;
            const uint32_t sa = smem_u32(smem + sg * C::STAGE_BYTES);
            const uint32_t sb = sa + NS * C::A_BYTES;
            if (BYLEVEL) {
#pragma unroll
              for (int p = 0; p < NS * (NS + 1) / 2; ++p) {
                const int la = (p == 2 || p == 4) ? 1 : (p == 5 ? 2 : 0), lb = (p == 1 || p == 4) ? 1 : (p == 3 ? 2 : 0);
#pragma unroll
                for (int kk = 0; kk < BK / 16; ++kk)
                  umma_f16(tb + (p ? 64 : 0), desc_of<BK>(sa + la * C::A_BYTES + kk * 32),
                           desc_of<BK>(sb + lb * C::B_BYTES + kk * 32), idesc0 | ((uint32_t)(PBN >> 3) << 17),
                           (!first || p > 1 || kk > 0) ? 1u : 0u);
              }
            } else {
              const int nk = (min(BK, K - k0) + 15) >> 4;  // 16-wide steps with data
              for (int kk = 0; kk < nk; ++kk) {
                const uint64_t bd = desc_of<BK>(sb + kk * 32);
#pragma unroll
                for (int l = 0; l < NS; ++l)
                  umma_f16(tb + 64 * l, desc_of<BK>(sa + l * C::A_BYTES + kk * 32), bd,
                           idesc0 | ((uint32_t)((PBN * (NS - l)) >> 3) << 17), (!first || kk > 0 || l > 0) ? 1u : 0u);
              }
            }
            umma_commit(&empty_bar[sg]);
            last_commit_s = it;
            ++it;
            if (k0 + BK < K && (k0 + BK) % PIECE != 0) continue;  // the piece goes on
            ++c;
            if ((c & 1) == 0 || c == T) {
              umma_commit(&accf[b]);
              last_accf_s = fg;
              ++fg;
            }
          }
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
      }
    }
  } else {
    // ---------------- epilogue: fold, write per tile ----------------
    // warp w reads TMEM lanes 32 (w % 4) .. + 31 and folds columns 32 h .. + 31
    const int q = warp & 3, h = (warp - 2) >> 2;
    const uint32_t lane_off = (uint32_t)(32 * q) << 16;
    uint64_t* stg = reinterpret_cast<uint64_t*>(smem + S * C::STAGE_BYTES) + (warp - 2) * PSTG_WARP;
    int fg = 0;
    bool ok = true;
    float hi[32], lo[32];
    for (int i = 0; blockIdx.x + i * gridDim.x < nitems && ok; ++i) {
      const TileItem& z = item(i);
      if (z.part >= z.parts) continue;
#pragma unroll
      for (int i = 0; i < 32; ++i) { hi[i] = 0.f; lo[i] = 0.f; }
      const int units = (part_pieces(z, segs) + 1) / 2;
      for (int f = 0; f < units; ++f) {
        const int b = fg & 1;
        ok = __all_sync(0xffffffffu, wait_ab(&accf[b], (fg >> 1) & 1, wait_ns, abort_f, err));
        if (!ok) break;
        fence_after();
        const uint32_t tb = tmem + BUF * b + lane_off + 32 * h;
#pragma unroll
        for (int cb = 0; cb < 32; cb += 16) {
          constexpr int ND = BYLEVEL ? 2 : NS;  // accumulators
          uint32_t dv[ND][16];
#pragma unroll
          for (int d = 0; d < ND; ++d) tmem_ld16_nw(tb + 64 * d + cb, dv[d]);
          tmem_wait_ld16(dv[0]);
#pragma unroll
          for (int d = 1; d < ND; ++d) tmem_dep16(dv[d]);
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            float u = __uint_as_float(dv[ND - 1][i]);
#pragma unroll
            for (int d = ND - 2; d >= 1; --d) u += __uint_as_float(dv[d][i]);
            if (BYLEVEL) {
              const float x = __uint_as_float(dv[0][i]), h0 = hi[cb + i];
              if (f == 0) {
                hi[cb + i] = x;
                lo[cb + i] = u;
              } else {
                const float sv = h0 + x;
                const float bp = sv - h0;
                lo[cb + i] += ((h0 - (sv - bp)) + (x - bp)) + u;
                hi[cb + i] = sv;
              }
            } else {
              two_sum_into(hi[cb + i], lo[cb + i], __uint_as_float(dv[0][i]));
              lo[cb + i] += u;
            }
          }
        }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acce[b]);
        ++fg;
      }
      if (!ok) break;
      if (z.parts > 1 && !gather_parts(z, (blockIdx.x + i * gridDim.x) / split, split, PEPI, warp - 2, scratch, tickets, hi, lo)) continue;
#pragma unroll
      for (int cb = 0; cb < 32; cb += 16) {
        if (OUT32) {
          store_block16(stg, [&](int k) { return (uint64_t)__float_as_uint(hi[cb + k] + lo[cb + k]); },
                        reinterpret_cast<float*>(z.C), z.ldc, z.m0 + 32 * q, z.n0 + 32 * h + cb, z.M, z.N, z.flags & 1);
        } else {
          double v[16];
          dbl_of_pairs<16>(hi + cb, lo + cb, v, BYLEVEL);
          store_block16(stg, [&](int k) { return (uint64_t)__double_as_longlong(v[k]); },
                        reinterpret_cast<double*>(z.C), z.ldc, z.m0 + 32 * q, z.n0 + 32 * h + cb, z.M, z.N, z.flags & 1);
        }
      }
    }
  }

  fence_before();
  __syncthreads();
  fence_after();
  if (abort_s && tid == 0) {
    // drain what this CTA still has in flight: TMA chunks issued but not
    // consumed (each the newest phase of its stage barrier), the MMAs up to
    // the last stage commit, the last accumulator commit
    for (int c = consumed_s; c < issued_s; ++c) mbar_wait(&full_bar[c % S], (c / S) & 1, DRAIN_NS);
    if (last_commit_s >= 0) mbar_wait(&empty_bar[last_commit_s % S], (last_commit_s / S) & 1, DRAIN_NS);
    if (last_accf_s >= 0) mbar_wait(&accf[last_accf_s & 1], (last_accf_s >> 1) & 1, DRAIN_NS);
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(PTMEM_COLS) : "memory");
}

int sm_count() {
  static const int n = [] {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
      cudaGetLastError();
      return 148;
    }
    return v;
  }();
  return n;
}

}  // namespace

cudaError_t launch_gemm_tcp(const GGroup* groups, const GSeg* segs, const GTile* tiles, int ntiles, int split,
                            int kbox, const void* maps, const Bases& b, int nsplit, bool out32, void* scratch,
                            unsigned* tickets, int* err, long long wait_ns, cudaStream_t s, bool bylevel) {
  if (ntiles == 0) return cudaSuccess;
  if (bylevel && (kbox != 64 || split != 1)) return cudaErrorInvalidValue;
  if ((kbox != 32 && kbox != 64) || split < 1 || (split > 1 && (!scratch || !tickets))) return cudaErrorInvalidValue;
  const int nitems = ntiles * split, grid = nitems < sm_count() ? nitems : sm_count();
  auto run = [&](auto kernel) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PSMEM);
    if (e != cudaSuccess) return e;
    kernel<<<grid, PTHREADS, PSMEM, s>>>(groups, segs, tiles, nitems, split, (const CUtensorMap*)maps, b,
                                         (uint64_t*)scratch, tickets, err, wait_ns);
    return cudaGetLastError();
  };
  auto pick = [&](auto ns) {
    constexpr int NS = decltype(ns)::value;
    if (bylevel) return out32 ? run(gemm_tcp_kernel<NS, 64, true, true>) : run(gemm_tcp_kernel<NS, 64, false, true>);
    if (kbox == 64) return out32 ? run(gemm_tcp_kernel<NS, 64, true, false>) : run(gemm_tcp_kernel<NS, 64, false, false>);
    return out32 ? run(gemm_tcp_kernel<NS, 32, true, false>) : run(gemm_tcp_kernel<NS, 32, false, false>);
  };
  if (nsplit == 2) return pick(std::integral_constant<int, 2>{});
  if (nsplit == 3) return pick(std::integral_constant<int, 3>{});
  return cudaErrorInvalidValue;
}

}  // namespace tt

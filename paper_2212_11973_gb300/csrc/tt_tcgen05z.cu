// Exact-accumulation split GEMM on the 5th-generation tensor cores (sm_103a).
//
// Operands are fixed-point BF16 digits (Ozaki scheme with one exponent per
// operand row and GEMM segment; see tt_ozaki.cu for the arithmetic): a row
// with largest biased exponent e holds v ~ 2^(e - 1054) F, F = a0 2^24 +
// a1 2^16 + a2 2^8 + a3, |a_s| <= 256, the four digit levels stored like
// split-BF16 levels (K-major, rows padded to 8, level l at l * lo[slot]) and
// the int16 exponents per row next to them.  Every tensor-core product of
// two digits is exact and, for a segment of K <= 256, every sum of the digit
// pairs with s + t = d is an integer below 2^24, exact in the FP32 TMEM
// accumulator.  The kernel keeps the ten pairs with s + t <= 3 in four TMEM
// accumulators D_0..D_3 and, once per segment, the epilogue warps add
// sum_d D_d 2^(eA + eB - 2060 - 8 d) to a two-float (hi, lo) sum in
// registers (TwoSum for d = 0, 1): ~2^-32 of the rows' bounds, with no
// rounding that grows with K.
//
// Structure as gemm_tcp_kernel (tt_tcgen05p.cu): persistent, one CTA per SM,
// 128 x 64 output tiles; warp 0 streams the digit tiles into a ring of two
// shared-memory stages of 64 K (A 4 x 16 KB, B 4 x 8 KB) or four of 32, warp 1 issues the MMAs of
// a segment into one of two TMEM buffers (4 accumulators x 64 columns each),
// warps 2-9 fold a finished buffer while the next segment's MMAs run in the
// other (two warps per TMEM lane quarter, 32 columns each, so that every SM
// sub-partition has two folding warps), and write each finished tile as FP64
// or as a two-float pair (flags bit 1) through a per-warp, XOR-swizzled
// shared-memory staging buffer (coalesced 128-byte row stores, no cross-warp
// barrier).  Waits are bounded as in the other tcgen05 kernels.
//
// What bounds it: the chain of 18 to 42 short segments (K = 3 to 180) behind
// each output tile at small D, shared-memory and L2 bandwidth of the operands and
// the output stores at D = 1024; never the tensor pipe.  So
//   (1) 16-wide K steps past a segment's end are skipped, and plans whose segments
//       are at most 64 long (D up to ~350) use chunks of 32, four in flight (D =
//       1024, whose longer segments feed fine from two stages of 64, was 15 %
//       slower with them);
//   (2) the items of a CTA are read side by side into shared memory before the
//       roles start; a segment's tensor maps are fenced and its K and exponent
//       references read by the lanes of a warp, 32 segments at a time; exponents
//       are loaded one segment ahead of the wait;
//   (3) where a plan has fewer tiles than SMs, `split` CTAs share a tile's
//       segments: each writes its two-float sums to scratch and the last to
//       arrive (a ticket per tile and folding warp, no CTA waits for another)
//       adds them in part order;
//   (4) FP64 outputs are put together by integer operations, and all stores of
//       16 rows are in flight together.
// Measured, a launch: S3, B1 and B2 at D = 300 40 -> 19 us on average; S3 at D =
// 1024 205 -> 150 us, S1 133 -> 121 us (25 tiles a CTA, each a single segment:
// its stores are half of the time).
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

constexpr int ZBM = 128, ZBN = 64, ZDIG = 4;
constexpr int ZMAXSTAGES = 4;
constexpr int ZRING_BYTES = 2 * ZDIG * (ZBM + ZBN) * 64 * 2;  // 192 KB of operand stages
constexpr uint32_t ZTMEM_COLS = 512;
constexpr int ZEPI = 8;  // epilogue warps
constexpr int ZTHREADS = 64 + 32 * ZEPI;
constexpr int ZMAXK = 256;  // longest segment whose digit sums stay exact
// epilogue staging, after the TMA stages: per epilogue warp 16 rows x 16
// columns of 8-byte outputs
constexpr int ZSTG_WARP = 16 * 16;
constexpr int ZSTG_BYTES = ZEPI * ZSTG_WARP * 8;

// PAIR: every group of the launch writes two-float pairs (flags bit 1), else
// FP64 (accumulating with flags bit 0); one kernel per output form keeps the
// FP64 conversions out of the pair kernel entirely
template <bool PAIR, int ZBK>
__global__ void __launch_bounds__(ZTHREADS, 1) gemm_tcz_kernel(const GGroup* __restrict__ groups,
                                                               const GSeg* __restrict__ segs,
                                                               const GTile* __restrict__ tiles, int nitems, int split,
                                                               const CUtensorMap* __restrict__ maps, Bases bs,
                                                               uint64_t* __restrict__ scratch,
                                                               unsigned* __restrict__ tickets, int* __restrict__ err,
                                                               long long wait_ns, bool exact_out) {
  constexpr int ZA_BYTES = ZBM * ZBK * 2, ZB_BYTES = ZBN * ZBK * 2;  // per digit level
  constexpr int ZSTAGE_BYTES = ZDIG * (ZA_BYTES + ZB_BYTES);
  constexpr int ZSTAGES = ZRING_BYTES / ZSTAGE_BYTES;
  static_assert(ZSTAGES <= ZMAXSTAGES && ZSTAGES * ZSTAGE_BYTES == ZRING_BYTES, "operand ring");
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[ZSTAGES], empty_bar[ZSTAGES], accf[2], acce[2];
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s, issued_s, consumed_s, last_commit_s, last_accf_s;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  volatile int* abort_f = &abort_s;
  __shared__ TileItem table[TITEMS];

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // the CTA's i-th item, in shared memory (beyond the table in a slot of the warp;
  // an item and its successor may be in use together)
  __shared__ TileItem own[(ZTHREADS / 32)][2];
  auto item = [&](int i) -> const TileItem& {
    if (i < TITEMS) return table[i];
    TileItem& o = own[warp][i & 1];
    __syncwarp();
    if (lane == 0) o = load_item(groups, segs, tiles, bs, 8, blockIdx.x + i * gridDim.x, split);
    __syncwarp();
    return o;
  };
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)),
                 "r"(ZTMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 32) {
    for (int s = 0; s < ZSTAGES; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], ZEPI);
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
  else load_items(table, groups, segs, tiles, maps, bs, 8, nitems, split);
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
            for (int k0 = 0; k0 < K; k0 += ZBK) {
              const int sg = it % ZSTAGES;
              if (!wait_ab(&empty_bar[sg], ((it / ZSTAGES) & 1) ^ 1, wait_ns, abort_f, err)) break;
              uint8_t* st = smem + sg * ZSTAGE_BYTES;
              mbar_expect_tx(&full_bar[sg], ZSTAGE_BYTES);
#pragma unroll
              for (int l = 0; l < ZDIG; ++l) tma_load_3d(st + l * ZA_BYTES, ma, k0, q.m0, l, &full_bar[sg]);
#pragma unroll
              for (int l = 0; l < ZDIG; ++l)
                tma_load_3d(st + ZDIG * ZA_BYTES + l * ZB_BYTES, mb, k0, q.n0, l, &full_bar[sg]);
              ++it;
              issued_s = it;
            }
          }
          stop = __any_sync(0xffffffffu, *abort_f);
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: one fold unit per segment ----------------
    // A digit s times the B digits 0 .. 3 - s in one instruction: the B levels lie
    // one after the other, 64 rows each, so they are an operand of N = 64 (4 - s)
    // rows, and its products belong to D_s .. D_3, 64 TMEM columns each.  Four
    // instructions per 16 K instead of ten, and A is read 4 times, not 10
    // (operands from shared memory, 128 bytes per clock, bound the MMAs here)
    constexpr uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(ZBM >> 4) << 24);
    int it = 0, fg = 0;
    bool ok = true;
    for (int i = 0; blockIdx.x + i * gridDim.x < nitems && ok; ++i) {
      const TileItem& q = item(i);
      int kl = q.K0;
      for (int s = 0; s < q.n && ok; ++s) {
        if ((s & 31) == 0 && q.n > 1) kl = segs[q.seg(min(s + lane, q.n - 1))].K;
        const int K = __shfl_sync(0xffffffffu, kl, s & 31);
        if (lane == 0) {
          const int b = fg & 1;
          ok = wait_ab(&acce[b], ((fg >> 1) & 1) ^ 1, wait_ns, abort_f, err);
          fence_after();
          const uint32_t tb = tmem + 256 * b;
          for (int k0 = 0; k0 < K && ok; k0 += ZBK) {
            const int sg = it % ZSTAGES;
            ok = wait_ab(&full_bar[sg], (it / ZSTAGES) & 1, wait_ns, abort_f, err);
            if (!ok) break;
            consumed_s = it + 1;
            fence_after();
            const uint32_t sa = smem_u32(smem + sg * ZSTAGE_BYTES);
            const int nk = (min(ZBK, K - k0) + 15) >> 4;  // 16-wide steps with data
            for (int kk = 0; kk < nk; ++kk) {
              const uint64_t bd = desc_of<ZBK>(sa + ZDIG * ZA_BYTES + kk * 32);
#pragma unroll
              for (int s = 0; s < ZDIG; ++s)
                umma_f16(tb + 64 * s, desc_of<ZBK>(sa + s * ZA_BYTES + kk * 32), bd,
                         idesc0 | ((uint32_t)((ZBN * (ZDIG - s)) >> 3) << 17), (k0 > 0 || kk > 0 || s > 0) ? 1u : 0u);
            }
            umma_commit(&empty_bar[sg]);
            last_commit_s = it;
            ++it;
          }
          if (ok) {
            umma_commit(&accf[b]);
            last_accf_s = fg;
            ++fg;
          }
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
      }
    }
  } else {
    // ---------------- epilogue: fold per segment, write per tile ----------------
    // warp w reads TMEM lanes 32 (w % 4) .. + 31 (the quarter its SM sub-
    // partition may access) and folds columns 32 h .. 32 h + 31 of them
    const int q = warp & 3, h = (warp - 2) >> 2;
    const uint32_t lane_off = (uint32_t)(32 * q) << 16;
    uint64_t* stg = reinterpret_cast<uint64_t*>(smem + ZRING_BYTES) + (warp - 2) * ZSTG_WARP;
    int fg = 0;
    bool ok = true;
    float hi[32], lo[32];
    // row exponents of the segment at hand: this lane's row, and the column of
    // which it holds the exponent for the others
    int ea = 0, eb = 0;
    auto exps = [&](const TileItem& t, const short* pa, int sa, const short* pb, int sb, int& xa, int& xb) {
      const int row = t.m0 + 32 * q + lane, col = t.n0 + 32 * h + lane;
      xa = t.n > 0 && row < t.M ? (int)pa[(long long)row * sa] : 0;
      xb = t.n > 0 && col < t.N ? (int)pb[(long long)col * sb] : 0;
    };
    for (int i = 0; blockIdx.x + i * gridDim.x < nitems && ok; ++i) {
      const TileItem& z = item(i);
      // exponent references of 32 segments, one per lane; the exponents of the
      // segment (or the next item's first segment) after the current one are in
      // flight while it is waited for
      unsigned long long ral = 0, rbl = 0;
      int sal = 0, sbl = 0;
      auto refs = [&](int s) {
        const GSeg* sp = segs + z.seg(min(s + lane, z.n - 1));
        ral = reinterpret_cast<unsigned long long>(exps_ptr(bs, sp->eA));
        rbl = reinterpret_cast<unsigned long long>(exps_ptr(bs, sp->eB));
        sal = sp->eas;
        sbl = sp->ebs;
      };
      if (z.n > 1) refs(0);
      if (i == 0) exps(z, z.pa, z.eas, z.pb, z.ebs, ea, eb);
#pragma unroll
      for (int i = 0; i < 32; ++i) { hi[i] = 0.f; lo[i] = 0.f; }
      if (z.n == 0) {
        if (blockIdx.x + (i + 1) * gridDim.x < nitems) {
          const TileItem& nx = item(i + 1);
          exps(nx, nx.pa, nx.eas, nx.pb, nx.ebs, ea, eb);
        }
        if (z.part >= z.parts) continue;  // (no segment left for this part)
      }
      for (int s = 0; s < z.n; ++s) {
        int ean = 0, ebn = 0;
        if (s + 1 < z.n) {
          if (((s + 1) & 31) == 0) refs(s + 1);
          const int l = (s + 1) & 31;
          exps(z, reinterpret_cast<const short*>(__shfl_sync(0xffffffffu, ral, l)), __shfl_sync(0xffffffffu, sal, l),
               reinterpret_cast<const short*>(__shfl_sync(0xffffffffu, rbl, l)), __shfl_sync(0xffffffffu, sbl, l), ean, ebn);
        } else if (blockIdx.x + (i + 1) * gridDim.x < nitems) {
          const TileItem& nx = item(i + 1);
          exps(nx, nx.pa, nx.eas, nx.pb, nx.ebs, ean, ebn);
        }
        const int b = fg & 1;
        ok = __all_sync(0xffffffffu, wait_ab(&accf[b], (fg >> 1) & 1, wait_ns, abort_f, err));
        if (!ok) break;
        fence_after();
        // the scale of D_0 at (row, column) is 2^(eA + eB - 2060): as a biased
        // FP32 exponent xa + eB, clamped to [0, 254] (0: below the normal
        // range, dropped like the digits below it)
        const int xa = ea - 2060 + 127;
        const uint32_t tb = tmem + 256 * b + lane_off + 32 * h;
        const bool first = s == 0;
#pragma unroll
        for (int cb = 0; cb < 32; cb += 16) {
          uint32_t dv[ZDIG][16];
#pragma unroll
          for (int d = 0; d < ZDIG; ++d) tmem_ld16_nw(tb + 64 * d + cb, dv[d]);
          tmem_wait_ld16(dv[0]);
#pragma unroll
          for (int d = 1; d < ZDIG; ++d) tmem_dep16(dv[d]);
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const int xe = xa + __shfl_sync(0xffffffffu, eb, cb + i);
            const float sc = __int_as_float(min(max(xe, 0), 254) << 23);
            // D_0 + D_1 2^-8 as an exact pair (sv, ev) (TwoSum), D_2 2^-16 and
            // D_3 2^-24 into ev, then the pair scaled by the power of two sc (a
            // product of its own: fused into the sums below, the same but where it
            // is subnormal, it would round once less)
            const float d0 = __uint_as_float(dv[0][i]);
            const float p1 = __uint_as_float(dv[1][i]) * 0.00390625f;
            const float sv = d0 + p1;
            const float bp = sv - d0;
            float ev = (d0 - (sv - bp)) + (p1 - bp);
            ev = fmaf(__uint_as_float(dv[2][i]), 1.52587890625e-05f, ev);
            ev = fmaf(__uint_as_float(dv[3][i]), 5.9604644775390625e-08f, ev);
            const float s2 = __fmul_rn(sv, sc), e2 = __fmul_rn(ev, sc);
            if (first) {
              hi[cb + i] = s2;
              lo[cb + i] = e2;
            } else {
              two_sum_into(hi[cb + i], lo[cb + i], s2);
              lo[cb + i] += e2;
            }
          }
        }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acce[b]);
        ++fg;
        ea = ean;
        eb = ebn;
      }
      if (!ok) break;
      if (z.parts > 1 && !gather_parts(z, (blockIdx.x + i * gridDim.x) / split, split, ZEPI, warp - 2, scratch, tickets, hi, lo)) continue;
      // the finished 32 x 32 block
#pragma unroll
      for (int cb = 0; cb < 32; cb += 16) {
        if (PAIR) {
          store_block16(
              stg,
              [&](int k) {
                return ((uint64_t)__float_as_uint(lo[cb + k]) << 32) | (uint64_t)__float_as_uint(hi[cb + k]);
              },
              reinterpret_cast<uint64_t*>(z.C), z.ldc, z.m0 + 32 * q, z.n0 + 32 * h + cb, z.M, z.N, false);
        } else {
          double v[16];
          dbl_of_pairs<16>(hi + cb, lo + cb, v, exact_out);
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
    for (int c = consumed_s; c < issued_s; ++c) mbar_wait(&full_bar[c % ZSTAGES], (c / ZSTAGES) & 1, DRAIN_NS);
    if (last_commit_s >= 0) mbar_wait(&empty_bar[last_commit_s % ZSTAGES], (last_commit_s / ZSTAGES) & 1, DRAIN_NS);
    if (last_accf_s >= 0) mbar_wait(&accf[last_accf_s & 1], (last_accf_s >> 1) & 1, DRAIN_NS);
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ZTMEM_COLS) : "memory");
}

int sm_count_z() {
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

int tcz_max_k() { return ZMAXK; }
size_t tcz_smem_bytes() { return (size_t)ZRING_BYTES + ZSTG_BYTES + 1024; }

int tcz_split(int ntiles, int max_segs) {
  if (ntiles <= 0) return 1;
  const int room = sm_count_z() / ntiles;
  // at least four segments to a part: with two, six ladders stepped side by side
  // (each CTA takes a whole SM) lost 4 % to the larger grids
  return room < 2 || max_segs < 8 ? 1 : (room < max_segs / 4 ? room : max_segs / 4);
}
size_t tcz_scratch_bytes(int ntiles, int split) { return split > 1 ? (size_t)ntiles * split * ZBM * ZBN * 8 : 0; }
size_t tcz_tickets(int ntiles) { return (size_t)ntiles * ZEPI; }

cudaError_t launch_gemm_tcz(const GGroup* groups, const GSeg* segs, const GTile* tiles, int ntiles, int split,
                            int kbox, const void* maps, const Bases& b, void* scratch, unsigned* tickets, int* err,
                            long long wait_ns, bool pair, cudaStream_t s, bool exact_out) {
  if (ntiles == 0) return cudaSuccess;
  if ((kbox != 32 && kbox != 64) || split < 1 || (split > 1 && (!scratch || !tickets))) return cudaErrorInvalidValue;
  const size_t smem = tcz_smem_bytes();
  const int nitems = ntiles * split, grid = nitems < sm_count_z() ? nitems : sm_count_z();
  auto run = [&](auto kernel) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<grid, ZTHREADS, smem, s>>>(groups, segs, tiles, nitems, split, (const CUtensorMap*)maps, b,
                                        (uint64_t*)scratch, tickets, err, wait_ns, exact_out);
    return cudaGetLastError();
  };
  if (pair) return kbox == 64 ? run(gemm_tcz_kernel<true, 64>) : run(gemm_tcz_kernel<true, 32>);
  return kbox == 64 ? run(gemm_tcz_kernel<false, 64>) : run(gemm_tcz_kernel<false, 32>);
}

}  // namespace tt

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
// each output tile at small D, shared-memory and L2 bandwidth of the operands at
// D = 1024; never the tensor pipe.  So (1) 16-wide K steps past a segment's end
// are skipped, and plans whose segments are at most 64 long (D up to ~350) use
// chunks of 32, four in flight (D = 300: 40 -> 24 us a launch; D = 1024, whose
// longer segments feed fine from two stages of 64, was 15 % slower with them);
// (2) a segment's tensor maps are
// fenced and its K and exponent references read by the lanes of a warp, 32
// segments at a time, and the row exponents of the next segment are loaded
// before the wait for the current one; (3) where a plan has fewer tiles than
// SMs, `split` CTAs share a tile's segments: each writes its two-float sums to
// scratch and the last to arrive (a ticket per tile and folding warp, no CTA
// waits for another) adds them in part order.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

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
// epilogue staging, after the TMA stages: per epilogue warp 32 rows x 16
// columns of 8-byte outputs, column c of row r at word r * 16 + (c ^ (r & 15))
constexpr int ZSTG_WARP = 32 * 16;
constexpr int ZSTG_BYTES = ZEPI * ZSTG_WARP * 8;

__device__ __forceinline__ void mbar_arrive_z(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool wait_z(uint64_t* bar, uint32_t parity, long long budget, volatile int* abort_f,
                                       int* err) {
  if (mbar_test_wait(bar, parity)) return true;
  const unsigned long long t0 = globaltimer();
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort_f) return false;
    if (budget <= 0 || (long long)(globaltimer() - t0) > budget) {
      *abort_f = 1;
      if (err) atomicExch(err, 1);
      return false;
    }
  }
}

// 16 TMEM columns of this warp's lane quarter, not yet waited for: the caller
// issues tmem_wait_ld16() with one set of registers and tmem_dep16() with
// every other set before reading them (the registers pass through those asm
// statements, so no use is scheduled before the wait)
__device__ __forceinline__ void tmem_ld16_nw(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld16(uint32_t* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}
__device__ __forceinline__ void tmem_dep16(uint32_t* r) {
  asm volatile(""
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}

__device__ __forceinline__ void two_sum_z(float& hi, float& lo, float x) {
  const float s = hi + x;
  const float bp = s - hi;
  const float ap = s - bp;
  lo += (hi - ap) + (x - bp);
  hi = s;
}

// UMMA shared-memory descriptor, K-major, rows of BK elements in one swizzle
// span (64: 128 bytes, 32: 64 bytes), 8-row groups contiguous
template <int BK>
__device__ __forceinline__ uint64_t desc_of(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)1 << 16;                    // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)((8 * BK * 2) >> 4) << 32;  // stride byte offset
  d |= (uint64_t)1 << 46;                    // descriptor version
  d |= (uint64_t)(BK == 64 ? 2 : 4) << 61;   // SWIZZLE_128B / SWIZZLE_64B
  return d;
}

// one part of a tile: segments seg0 + part, + split, ... (n of them)
struct ZItem {
  GTile tl;
  GGroup g;
  int part, parts, n;
};
__device__ __forceinline__ ZItem item_of(const GGroup* groups, const GTile* tiles, int w, int split) {
  ZItem it;
  it.tl = tiles[w / split];
  it.g = groups[it.tl.g];
  const int nseg = it.g.seg1 - it.g.seg0;
  it.part = w % split;
  it.parts = max(1, min(split, nseg));
  it.n = it.part < it.parts ? (nseg - it.part + it.parts - 1) / it.parts : 0;
  return it;
}

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
                                                               long long wait_ns) {
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

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
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
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_base_s;

  if (warp == 0) {
    // ---------------- producer ----------------
    int it = 0, fenced = -1;  // group whose first 32 segments' maps this CTA has fenced
    for (int w = blockIdx.x; w < nitems && !*abort_f; w += gridDim.x) {
      const ZItem q = item_of(groups, tiles, w, split);
      for (int s0 = 0; s0 < q.n; s0 += 32) {
        const int sl = q.g.seg0 + q.part + min(s0 + lane, q.n - 1) * q.parts;
        const int kl = segs[sl].K;
        if (fenced != q.tl.g || q.n > 32) {
          const uint64_t ma = reinterpret_cast<uint64_t>(maps + 3 * sl), mb = ma + 2 * sizeof(CUtensorMap);
          asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(ma) : "memory");
          asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(mb) : "memory");
          asm volatile("prefetch.tensormap [%0];" ::"l"(ma) : "memory");
          asm volatile("prefetch.tensormap [%0];" ::"l"(mb) : "memory");
          fenced = q.parts == 1 ? q.tl.g : -1;
          __syncwarp();
        }
        for (int s = s0; s < min(q.n, s0 + 32); ++s) {
          const int K = __shfl_sync(0xffffffffu, kl, s - s0);
          if (lane == 0) {
            const int si = q.g.seg0 + q.part + s * q.parts;
            const CUtensorMap* ma = maps + 3 * si;
            const CUtensorMap* mb = ma + 2;
            for (int k0 = 0; k0 < K; k0 += ZBK) {
              const int sg = it % ZSTAGES;
              if (!wait_z(&empty_bar[sg], ((it / ZSTAGES) & 1) ^ 1, wait_ns, abort_f, err)) break;
              uint8_t* st = smem + sg * ZSTAGE_BYTES;
              mbar_expect_tx(&full_bar[sg], ZSTAGE_BYTES);
#pragma unroll
              for (int l = 0; l < ZDIG; ++l) tma_load_3d(st + l * ZA_BYTES, ma, k0, q.tl.m0, l, &full_bar[sg]);
#pragma unroll
              for (int l = 0; l < ZDIG; ++l)
                tma_load_3d(st + ZDIG * ZA_BYTES + l * ZB_BYTES, mb, k0, q.tl.n0, l, &full_bar[sg]);
              ++it;
              issued_s = it;
            }
          }
          __syncwarp();
          if (*abort_f) break;
        }
        if (*abort_f) break;
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
    for (int w = blockIdx.x; w < nitems && ok; w += gridDim.x) {
      const ZItem q = item_of(groups, tiles, w, split);
      int kl = 0;
      for (int s = 0; s < q.n && ok; ++s) {
        if ((s & 31) == 0) kl = segs[q.g.seg0 + q.part + min(s + lane, q.n - 1) * q.parts].K;
        const int K = __shfl_sync(0xffffffffu, kl, s & 31);
        if (lane == 0) {
          const int b = fg & 1;
          ok = wait_z(&acce[b], ((fg >> 1) & 1) ^ 1, wait_ns, abort_f, err);
          fence_after();
          const uint32_t tb = tmem + 256 * b;
          for (int k0 = 0; k0 < K && ok; k0 += ZBK) {
            const int sg = it % ZSTAGES;
            ok = wait_z(&full_bar[sg], (it / ZSTAGES) & 1, wait_ns, abort_f, err);
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
    for (int w = blockIdx.x; w < nitems && ok; w += gridDim.x) {
      const ZItem z = item_of(groups, tiles, w, split);
      const GTile tl = z.tl;
      const GGroup& g = z.g;
      if (z.part >= z.parts) continue;
      const int row = tl.m0 + 32 * q + lane;
      const int col_l = tl.n0 + 32 * h + lane;  // the column whose exponent this lane loads
#pragma unroll
      for (int i = 0; i < 32; ++i) { hi[i] = 0.f; lo[i] = 0.f; }
      // exponent references of 32 segments, one per lane; the exponents of the
      // segment after the current one are in flight while it is waited for
      unsigned long long ral = 0, rbl = 0;
      int sal = 0, sbl = 0;
      auto refs = [&](int s) {
        const GSeg* sp = segs + g.seg0 + z.part + min(s + lane, z.n - 1) * z.parts;
        ral = sp->eA;
        rbl = sp->eB;
        sal = sp->eas;
        sbl = sp->ebs;
      };
      auto exps = [&](int s, int& ea, int& eb) {
        const int l = s & 31;
        const Ref ra = __shfl_sync(0xffffffffu, ral, l), rb = __shfl_sync(0xffffffffu, rbl, l);
        const int sa = __shfl_sync(0xffffffffu, sal, l), sb = __shfl_sync(0xffffffffu, sbl, l);
        const short* pa = reinterpret_cast<const short*>(sel_base(bs, slot_of(ra))) + off_of(ra);
        const short* pb = reinterpret_cast<const short*>(sel_base(bs, slot_of(rb))) + off_of(rb);
        ea = row < g.M ? (int)pa[(long long)row * sa] : 0;
        eb = col_l < g.N ? (int)pb[(long long)col_l * sb] : 0;
      };
      int ea = 0, eb = 0;
      if (z.n > 0) {
        refs(0);
        exps(0, ea, eb);
      }
      for (int s = 0; s < z.n; ++s) {
        int ean = 0, ebn = 0;
        if (s + 1 < z.n) {
          if (((s + 1) & 31) == 0) refs(s + 1);
          exps(s + 1, ean, ebn);
        }
        const int b = fg & 1;
        ok = __all_sync(0xffffffffu, wait_z(&accf[b], (fg >> 1) & 1, wait_ns, abort_f, err));
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
            // D_3 2^-24 into ev, then the pair scaled by the power of two sc
            const float d0 = __uint_as_float(dv[0][i]);
            const float p1 = __uint_as_float(dv[1][i]) * 0.00390625f;
            const float sv = d0 + p1;
            const float bp = sv - d0;
            float ev = (d0 - (sv - bp)) + (p1 - bp);
            ev = fmaf(__uint_as_float(dv[2][i]), 1.52587890625e-05f, ev);
            ev = fmaf(__uint_as_float(dv[3][i]), 5.9604644775390625e-08f, ev);
            const float s2 = sv * sc, e2 = ev * sc;
            if (first) {
              hi[cb + i] = s2;
              lo[cb + i] = e2;
            } else {
              two_sum_z(hi[cb + i], lo[cb + i], s2);
              lo[cb + i] += e2;
            }
          }
        }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_z(&acce[b]);
        ++fg;
        ea = ean;
        eb = ebn;
      }
      if (!ok) break;
      if (z.parts > 1) {
        // this part's sums to scratch, 32 rows contiguous per column; the last
        // part to arrive adds all of them in part order
        const int t = w / split;
        uint64_t* sc = scratch + ((size_t)t * split * ZEPI + (warp - 2)) * 1024 + lane;
        uint64_t* mine = sc + (size_t)z.part * ZEPI * 1024;
#pragma unroll
        for (int i = 0; i < 32; ++i)
          __stcg(mine + 32 * i, ((uint64_t)__float_as_uint(lo[i]) << 32) | (uint64_t)__float_as_uint(hi[i]));
        __threadfence();
        __syncwarp();
        unsigned arrived = 0;
        if (lane == 0) arrived = atomicInc(&tickets[t * ZEPI + warp - 2], z.parts - 1);
        arrived = __shfl_sync(0xffffffffu, arrived, 0);
        if (arrived != (unsigned)(z.parts - 1)) continue;
        __threadfence();
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const uint64_t v = __ldcg(sc + 32 * i);
          hi[i] = __uint_as_float((uint32_t)v);
          lo[i] = __uint_as_float((uint32_t)(v >> 32));
        }
        for (int p = 1; p < z.parts; ++p) {
          const uint64_t* o = sc + (size_t)p * ZEPI * 1024;
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const uint64_t v = __ldcg(o + 32 * i);
            two_sum_z(hi[i], lo[i], __uint_as_float((uint32_t)v));
            lo[i] += __uint_as_float((uint32_t)(v >> 32));
          }
        }
      }
      // the finished 32 x 32 block, 16 columns at a time through this warp's
      // staging buffer: one row per lane on the way in, 16 lanes per row (128
      // contiguous bytes) on the way out
      const bool accum = g.flags & 1;
      const int c_l = lane & 15;
      uint64_t* const Cb = reinterpret_cast<uint64_t*>(sel_base(bs, slot_of(g.C))) + off_of(g.C);
#pragma unroll
      for (int cb = 0; cb < 32; cb += 16) {
        if (PAIR) {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            stg[lane * 16 + (i ^ (lane & 15))] =
                ((uint64_t)__float_as_uint(lo[cb + i]) << 32) | (uint64_t)__float_as_uint(hi[cb + i]);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            stg[lane * 16 + (i ^ (lane & 15))] =
                (uint64_t)__double_as_longlong((double)hi[cb + i] + (double)lo[cb + i]);
        }
        __syncwarp();
        const int col = tl.n0 + 32 * h + cb + c_l;
        for (int rr = lane >> 4; rr < 32; rr += 2) {
          const int grow = tl.m0 + 32 * q + rr;
          if (grow < g.M && col < g.N) {
            const long long o = (long long)grow * g.ldc + col;
            const uint64_t bits = stg[rr * 16 + (c_l ^ (rr & 15))];
            if (PAIR || !accum) {
              Cb[o] = bits;
            } else {
              double* Cp = reinterpret_cast<double*>(Cb + o);
              *Cp += __longlong_as_double((long long)bits);
            }
          }
        }
        __syncwarp();
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
  return room < 2 || max_segs < 4 ? 1 : (room < max_segs / 2 ? room : max_segs / 2);
}
size_t tcz_scratch_bytes(int ntiles, int split) { return split > 1 ? (size_t)ntiles * split * ZBM * ZBN * 8 : 0; }
size_t tcz_tickets(int ntiles) { return (size_t)ntiles * ZEPI; }

cudaError_t launch_gemm_tcz(const GGroup* groups, const GSeg* segs, const GTile* tiles, int ntiles, int split,
                            int kbox, const void* maps, const Bases& b, void* scratch, unsigned* tickets, int* err,
                            long long wait_ns, bool pair, cudaStream_t s) {
  if (ntiles == 0) return cudaSuccess;
  if ((kbox != 32 && kbox != 64) || split < 1 || (split > 1 && (!scratch || !tickets))) return cudaErrorInvalidValue;
  const size_t smem = tcz_smem_bytes();
  const int nitems = ntiles * split, grid = nitems < sm_count_z() ? nitems : sm_count_z();
  auto run = [&](auto kernel) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<grid, ZTHREADS, smem, s>>>(groups, segs, tiles, nitems, split, (const CUtensorMap*)maps, b,
                                        (uint64_t*)scratch, tickets, err, wait_ns);
    return cudaGetLastError();
  };
  if (pair) return kbox == 64 ? run(gemm_tcz_kernel<true, 64>) : run(gemm_tcz_kernel<true, 32>);
  return kbox == 64 ? run(gemm_tcz_kernel<false, 64>) : run(gemm_tcz_kernel<false, 32>);
}

}  // namespace tt

// Inline PTX helpers of the tcgen05 GEMM kernels (sm_103a): mbarriers with
// bounded waits, 3-D TMA tile loads, UMMA shared-memory descriptors (K-major,
// 128-byte swizzle), tcgen05.mma / commit, and 32-column TMEM loads / stores.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

#include "tt_kernels.h"

namespace tt {
namespace tcx {

// budget of the waits that drain an aborted CTA's own copies and MMAs (these
// always complete; the budget only keeps a wrong phase from spinning forever)
constexpr long long DRAIN_NS = 2000000000ll;

static __device__ __forceinline__ int slot_of(Ref r) { return (int)(r >> 56); }
static __device__ __forceinline__ long long off_of(Ref r) { return (long long)(r & 0x00FFFFFFFFFFFFFFull); }

static __device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

static __device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

static __device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

static __device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t phase) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(phase)
      : "memory");
  return ok != 0;
}

static __device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t phase) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(phase)
      : "memory");
  return ok != 0;
}

static __device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// Wait for the phase of parity `phase` to complete, for at most budget_ns
// nanoseconds (one non-blocking test when the budget is <= 0); false when the
// budget expired.
static __device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t phase, long long budget_ns) {
  if (mbar_test_wait(bar, phase)) return true;
  if (budget_ns <= 0) return false;
  const unsigned long long t0 = globaltimer();
  while (true) {
    if (mbar_try_wait(bar, phase)) return true;
    if ((long long)(globaltimer() - t0) > budget_ns) return false;
  }
}

static __device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}

// UMMA shared-memory descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart (SBO), version 1 (sm_100 family).
static __device__ __forceinline__ uint64_t make_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)1 << 16;               // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;     // stride byte offset
  d |= (uint64_t)1 << 46;               // descriptor version
  d |= (uint64_t)2 << 61;               // SWIZZLE_128B
  return d;
}

static __device__ __forceinline__ void umma_f16(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

static __device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

// 32 TMEM columns of the warp's lane quarter; the wait is in the same asm
// statement, so no use of the registers can be scheduled before it
static __device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

static __device__ __forceinline__ void tmem_st32(uint32_t taddr, const float* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
      "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])),
      "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])),
      "r"(__float_as_uint(v[11])), "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])),
      "r"(__float_as_uint(v[14])), "r"(__float_as_uint(v[15])), "r"(__float_as_uint(v[16])),
      "r"(__float_as_uint(v[17])), "r"(__float_as_uint(v[18])), "r"(__float_as_uint(v[19])),
      "r"(__float_as_uint(v[20])), "r"(__float_as_uint(v[21])), "r"(__float_as_uint(v[22])),
      "r"(__float_as_uint(v[23])), "r"(__float_as_uint(v[24])), "r"(__float_as_uint(v[25])),
      "r"(__float_as_uint(v[26])), "r"(__float_as_uint(v[27])), "r"(__float_as_uint(v[28])),
      "r"(__float_as_uint(v[29])), "r"(__float_as_uint(v[30])), "r"(__float_as_uint(v[31]))
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

static __device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
static __device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// ---- persistent kernels (tt_tcgen05p.cu, tt_tcgen05z.cu) ----

static __device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

static __device__ __forceinline__ bool wait_ab(uint64_t* bar, uint32_t parity, long long budget, volatile int* abort_f,
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
static __device__ __forceinline__ void tmem_ld16_nw(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
static __device__ __forceinline__ void tmem_wait_ld16(uint32_t* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}
static __device__ __forceinline__ void tmem_dep16(uint32_t* r) {
  asm volatile(""
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}

static __device__ __forceinline__ void two_sum_into(float& hi, float& lo, float x) {
  const float s = hi + x;
  const float bp = s - hi;
  const float ap = s - bp;
  lo += (hi - ap) + (x - bp);
  hi = s;
}

// UMMA shared-memory descriptor, K-major, rows of BK elements in one swizzle
// span (64: 128 bytes, 32: 64 bytes), 8-row groups contiguous
template <int BK>
static __device__ __forceinline__ uint64_t desc_of(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)1 << 16;                    // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)((8 * BK * 2) >> 4) << 32;  // stride byte offset
  d |= (uint64_t)1 << 46;                    // descriptor version
  d |= (uint64_t)(BK == 64 ? 2 : 4) << 61;   // SWIZZLE_128B / SWIZZLE_64B
  return d;
}

// Segments of part `part` of `parts`: every parts-th pair of the group's, so that
// the split-BF16 kernel's fold groups are those of an undivided tile where every
// segment is one piece.
static __device__ __forceinline__ int part_count(int nseg, int split) { return max(1, min(split, (nseg + 1) >> 1)); }
static __device__ __forceinline__ int part_segs(int nseg, int parts, int part) {
  const int pairs = (nseg + 1) >> 1;
  if (part >= parts || nseg == 0) return 0;
  return 2 * ((pairs - part + parts - 1) / parts) - ((nseg & 1) && (pairs - 1) % parts == part ? 1 : 0);
}

// One part of a tile and what the roles need of its group and first segment:
// segments seg(0) .. seg(n - 1).
struct TileItem {
  void* C;                 // output of the group
  const short *pa, *pb;    // row exponents of the first segment's operands (digits)
  int m0, n0, M, N;
  int ldc, flags;
  int seg0, parts, part, n;
  int K0, eas, ebs;        // first segment
  __device__ __forceinline__ int seg(int s) const { return seg0 + (s >> 1) * 2 * parts + (s & 1); }
};
static __device__ __forceinline__ const short* exps_ptr(const Bases& bs, Ref r) {
  return reinterpret_cast<const short*>(sel_base(bs, slot_of(r))) + off_of(r);
}
static __device__ __forceinline__ TileItem load_item(const GGroup* groups, const GSeg* segs, const GTile* tiles,
                                                     const Bases& bs, int esize, int w, int split) {
  TileItem it;
  const GTile tl = tiles[w / split];
  const GGroup g = groups[tl.g];
  const int nseg = g.seg1 - g.seg0;
  it.part = w % split;
  it.parts = part_count(nseg, split);
  it.n = part_segs(nseg, it.parts, it.part);
  it.seg0 = g.seg0 + 2 * it.part;
  it.C = reinterpret_cast<char*>(sel_base(bs, slot_of(g.C))) + off_of(g.C) * esize;  // esize: bytes of an output
  it.m0 = tl.m0;
  it.n0 = tl.n0;
  it.M = g.M;
  it.N = g.N;
  it.ldc = g.ldc;
  it.flags = g.flags;
  it.K0 = it.eas = it.ebs = 0;
  it.pa = it.pb = nullptr;
  if (it.n > 0) {
    const GSeg& s = segs[it.seg0];
    it.K0 = s.K;
    it.pa = exps_ptr(bs, s.eA);
    it.pb = exps_ptr(bs, s.eB);
    it.eas = s.eas;
    it.ebs = s.ebs;
  }
  return it;
}
// The records of a CTA's first TITEMS items are loaded side by side before the
// roles start (tile -> group -> segment is a chain of three loads, which each
// role would go through for each tile), with the fences of the tensor maps of
// those with a single segment, by warps 1 and up; warp 0, the producer, meanwhile
// fences its first item's maps itself (first_segments).
constexpr int TITEMS = 40;
static __device__ __forceinline__ void fence_maps(const CUtensorMap* maps, int seg) {
  const uint64_t ma = reinterpret_cast<uint64_t>(maps + 4 * seg + 3), mb = ma - sizeof(CUtensorMap);
  asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(ma) : "memory");
  asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(mb) : "memory");
  asm volatile("prefetch.tensormap [%0];" ::"l"(ma) : "memory");
  asm volatile("prefetch.tensormap [%0];" ::"l"(mb) : "memory");
}
// K and map fences of the first 32 segments of the CTA's first item, one per lane
static __device__ __forceinline__ int first_segments(const GGroup* groups, const GSeg* segs, const GTile* tiles,
                                                     const CUtensorMap* maps, int split) {
  const GGroup g = groups[tiles[blockIdx.x / split].g];
  const int nseg = g.seg1 - g.seg0, parts = part_count(nseg, split), part = blockIdx.x % split;
  const int n = part_segs(nseg, parts, part);
  if (n == 0) return 0;
  const int at = min((int)(threadIdx.x & 31), n - 1);
  const int s = g.seg0 + 2 * part + (at >> 1) * 2 * parts + (at & 1);
  fence_maps(maps, s);
  return segs[s].K;
}
static __device__ __forceinline__ void load_items(TileItem* table, const GGroup* groups, const GSeg* segs,
                                                  const GTile* tiles, const CUtensorMap* maps, const Bases& bs, int esize,
                                                  int nitems, int split) {
  for (int i = threadIdx.x - 32; i < TITEMS; i += blockDim.x - 32) {
    const int w = blockIdx.x + i * gridDim.x;
    if (w >= nitems) break;
    const TileItem it = load_item(groups, segs, tiles, bs, esize, w, split);
    table[i] = it;
    if (it.n == 1) fence_maps(maps, it.seg0);  // (longer chains: by the producer, 32 at a time)
  }
}

// 16 columns of a warp's 32 x 32 block to global memory: bits(i) is the output of
// this lane's row (row0 + lane) and column col0 + i, 8 bytes or the low 4 (T =
// uint64_t / double / float; accum: added to what is there).  16 rows at a time
// through the warp's 2 KB of staging, XOR-swizzled, so that a row's 16 columns are
// one contiguous store and all eight of a lane's are in flight (one by one, each
// waited for its shared-memory load: 5000 clocks a tile, half of S1's time).
template <class T, class F>
static __device__ __forceinline__ void store_block16(uint64_t* stg, F bits, T* C, int ldc, int row0,
                                                     int col0, int M, int N, bool accum) {
  const int lane = threadIdx.x & 31, l = lane & 15, hf = lane >> 4;
  const int col = col0 + l;
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    if (hf == half) {
#pragma unroll
      for (int i = 0; i < 16; ++i) stg[l * 16 + (i ^ l)] = bits(i);
    }
    __syncwarp();
    uint64_t u[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) u[t] = stg[(2 * t + hf) * 16 + (l ^ (2 * t + hf))];
    const int row = row0 + 16 * half + hf;
    T* p = C + (long long)row * ldc + col;
    const long long step = 2ll * ldc;
    if (col < N) {
      if (accum) {
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          T v;
          memcpy(&v, &u[t], sizeof(T));
          if (row + 2 * t < M) p[t * step] += v;
        }
      } else {
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          T v;
          memcpy(&v, &u[t], sizeof(T));
          if (row + 2 * t < M) p[t * step] = v;
        }
      }
    }
    __syncwarp();
  }
}

// This part's 32 x 32 two-float sums (warp ew of nw epilogue warps; row per lane,
// hi / lo of 32 columns) to scratch, 32 rows contiguous per column; in the last
// part to arrive, the sums of all parts in part order and true.  tickets: one per
// tile and warp, zero before and after.
static __device__ __forceinline__ bool gather_parts(const TileItem& z, int tile, int split, int nw, int ew,
                                                    uint64_t* scratch, unsigned* tickets, float* hi, float* lo) {
  const int lane = threadIdx.x & 31;
  uint64_t* sc = scratch + ((size_t)tile * split * nw + ew) * 1024 + lane;
  uint64_t* mine = sc + (size_t)z.part * nw * 1024;
#pragma unroll
  for (int i = 0; i < 32; ++i)
    __stcg(mine + 32 * i, ((uint64_t)__float_as_uint(lo[i]) << 32) | (uint64_t)__float_as_uint(hi[i]));
  __threadfence();
  __syncwarp();
  unsigned arrived = 0;
  if (lane == 0) arrived = atomicInc(&tickets[tile * nw + ew], z.parts - 1);
  arrived = __shfl_sync(0xffffffffu, arrived, 0);
  if (arrived != (unsigned)(z.parts - 1)) return false;
  __threadfence();
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    const uint64_t v = __ldcg(sc + 32 * i);
    hi[i] = __uint_as_float((uint32_t)v);
    lo[i] = __uint_as_float((uint32_t)(v >> 32));
  }
  for (int p = 1; p < z.parts; ++p) {
    const uint64_t* o = sc + (size_t)p * nw * 1024;
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      const uint64_t v = __ldcg(o + 32 * i);
      two_sum_into(hi[i], lo[i], __uint_as_float((uint32_t)v));
      lo[i] += __uint_as_float((uint32_t)(v >> 32));
    }
  }
  return true;
}

}  // namespace tcx
}  // namespace tt

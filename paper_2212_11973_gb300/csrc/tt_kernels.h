// Launch wrappers of the device kernels (tt_kernels.cu).  Every wrapper is
// asynchronous on the given stream and returns the cudaError_t of the launch.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "tt_core.h"

namespace tt {

// Slot table passed by value to the plan-driven kernels: base pointer of each
// slot and, for split-BF16 buffers, the element offset of the "lo" half.
struct Bases {
  void* p[8];
  long long lo[8];
};

#ifdef __CUDACC__
// bs.p[slot] by selects: indexing the by-value kernel argument with a
// run-time slot would copy the array to local memory first
__device__ __forceinline__ void* sel_base(const Bases& bs, int slot) {
  void* p = bs.p[0];
#pragma unroll
  for (int k = 1; k < 8; ++k)
    if (slot == k) p = bs.p[k];
  return p;
}
__device__ __forceinline__ long long sel_lo(const Bases& bs, int slot) {
  long long v = bs.lo[0];
#pragma unroll
  for (int k = 1; k < 8; ++k)
    if (slot == k) v = bs.lo[k];
  return v;
}
#endif

// Device copies of a plan.
struct DevGemm {
  GGroup* groups = nullptr;
  GSeg* segs = nullptr;
  GTile* tiles64 = nullptr;   // 64 x 64 output tiles
  FTile* tilesd = nullptr;    // double-float kernel's tiles
  FTile* tilesf = nullptr;    // FP64 kernel: tf x tf output tiles on wkf warps
  int ngroups = 0, nsegs = 0, ntiles64 = 0, ntilesf = 0, tf = 0, wkf = 0, ntilesd = -1;
  double flops = 0;
};
struct DevGather {
  GItem* items = nullptr;
  GContrib* contribs = nullptr;
  int nitems = 0;
  double elems = 0;
};
// copies and digit copies: one CTA per part, an item and its first 32 x 32 tile
// (of COPY_TILES) or digit row (of 32)
struct CPart {
  int item, first;
};
constexpr int COPY_TILES = 2;
struct DevCopy {
  CItem* items = nullptr;
  CPart* parts = nullptr;
  int nparts = 0;
};
struct DevDigit {
  DItem* items = nullptr;
  CPart* parts = nullptr;
  int nparts = 0;
};

// Device-side Krylov bookkeeping of one Lanczos exponential.
struct KrylovState {
  double alpha[17];
  double beta[17];
  double h[17];     // first Gram-Schmidt pass
  double h2[17];    // second
  double c[17];
  double nb;        // ||v||
  double hscale;    // max(|alpha_j| + beta_j)
  double resid;     // ||v|| beta_K |c_K|
  double nrm;       // norm of the result (before normalisation)
  int kdim;         // Krylov dimension in use
  int broken;       // breakdown seen
  int bad;          // NaN / Inf seen
  unsigned ticket;  // CTAs arrived at the current reduction (zero between launches)
};

// Global accumulators of a state (device).
struct RhoScalars {
  double logscale;
  double resid_max;
  int bad;
  int pad;
};

// FP64 GEMM (tt_gemm64.cu) on the tile list f64_tiles(plan, T): T x T tiles, each
// on wk warps that share its K steps.
struct F64Shape {
  int T, wk;
};
F64Shape f64_shape(const GemmPlan& p);
// one-warp tiles: every output a single sum over ascending K, whatever T
F64Shape f64_shape_ordered(const GemmPlan& p);
std::vector<FTile> f64_tiles(const GemmPlan& p, int T);
cudaError_t launch_gemm_f64(const DevGemm& g, const Bases& b, cudaStream_t s);
// The same in double-float arithmetic on the FP32 pipe (~2^-46 per operation),
// on f64_tiles(plan, df_tile_size()).
int df_tile_size();
// whether the double-float kernel is the faster one for a plan
bool df_beats_f64(const GemmPlan& p);
// exact_out: hi + lo rounded as by an FP64 addition.
cudaError_t launch_gemm_df(const DevGemm& g, const Bases& b, cudaStream_t s, bool exact_out = false);
// Exact-accumulation split GEMM (tt_ozaki.cu): FP64 operands of the FP64
// plans, four fixed-point BF16 digits per K tile, ~2^-32 normwise.  topdown: digits
// rounded from the top level down (tt_fixed.h).
cudaError_t launch_gemm_oz(const DevGemm& g, const Bases& b, cudaStream_t s, bool topdown = false);
// nsplit = 2 (3 products) or 3 (6 products); operand level l at offset l * lo[slot]
cudaError_t launch_gemm_bf16(const DevGemm& g, const Bases& b, int nsplit, cudaStream_t s);
// in_type / out_type: 0 = double, 1 = float, 2 / 3 = split bf16 with that many levels
cudaError_t launch_gather(const DevGather& g, const Bases& b, int in_type, int out_type, cudaStream_t s);
cudaError_t launch_copy(const DevCopy& c, const Bases& b, cudaStream_t s);
cudaError_t launch_split_bf16(const double* x, int64_t n, int nsplit, void* out /* bf16[nsplit*n] */, cudaStream_t s);
cudaError_t launch_zero(void* p, size_t bytes, cudaStream_t s);
// strided FP64 -> split-bf16 copy (levels at dst + l * lo[slot(dst)])
cudaError_t launch_split_copy(const DevCopy& c, const Bases& b, int nsplit, cudaStream_t s);
// tcgen05 grouped GEMM (tt_tcgen05.cu): K-major A and B, 128 x 128 tiles, maps =
// 4 CUtensorMap per segment in global memory: A (box 64 K x 128 rows), B (64 x
// 128), B (kbox x 64), A (kbox x 128).
size_t tc_smem_bytes(int nsplit);
// Persistent warp-specialised variant (tt_tcgen05p.cu): 128 x 64 tiles, one
// CTA per SM, TMA ring / MMA warp / fold-and-epilogue warps, the same
// arithmetic and maps.
// out32: every group writes FP32 (flags bit 1), else FP64; split, kbox, scratch
// and tickets as for launch_gemm_tcz below; bylevel: the products of 64 of K level
// by level into two sums (kbox 64, split 1).
cudaError_t launch_gemm_tcp(const GGroup* groups, const GSeg* segs, const GTile* tiles128x64, int ntiles, int split,
                            int kbox, const void* maps, const Bases& b, int nsplit, bool out32, void* scratch,
                            unsigned* tickets, int* err, long long wait_ns, cudaStream_t s, bool bylevel = false);
// Exact-accumulation split GEMM on tcgen05 (tt_tcgen05z.cu): digit operands
// (4 levels + int16 row exponents, GSeg.eA / eB), persistent 128 x 64 tiles,
// maps with boxes of kbox = 64 (128-byte swizzle) or 32 (64-byte) K;
// segments of K <= tcz_max_k(); output FP64 or two-float pairs
// (flags bit 1, the same in every group of a launch: pair).
int tcz_max_k();
size_t tcz_smem_bytes();
// split CTAs share the segments of a tile (tcz_split: where the tiles leave SMs
// idle); they need scratch of tcz_scratch_bytes and tcz_tickets zeroed counters
// (left at zero).
int tcz_split(int ntiles, int max_segs);
size_t tcz_scratch_bytes(int ntiles, int split);
size_t tcz_tickets(int ntiles);
cudaError_t launch_gemm_tcz(const GGroup* groups, const GSeg* segs, const GTile* tiles128x64, int ntiles, int split,
                            int kbox, const void* maps, const Bases& b, void* scratch, unsigned* tickets, int* err,
                            long long wait_ns, bool pair, cudaStream_t s, bool exact_out = false);
// Digit producers (tt_digits.cu): FP64 rows -> digit rows; the W-gather of
// the exact path (two-float S1 outputs -> digit rows of T2, rows up to
// gather_digits_max_cols() long, at most gather_digits_max_contribs() MPO
// terms per item).
cudaError_t launch_digit_copy(const DevDigit& d, const Bases& b, cudaStream_t s, bool topdown = false);
cudaError_t launch_gather_digits(const DevGather& g, const Bases& b, cudaStream_t s);
int gather_digits_max_cols();
int gather_digits_max_contribs();
// err: set to 1 by a CTA whose bounded wait (budget wait_ns) ran out.
cudaError_t launch_gemm_tc(const GGroup* groups, const GSeg* segs, const GTile* tiles128, int ntiles,
                           const void* maps, const Bases& b, int nsplit, int* err, long long wait_ns, cudaStream_t s);

// Lanczos exponential on flat FP64 vectors of length n (tt_lanczos.cu).  Q holds
// the Krylov basis with leading dimension ldq; `partial` is scratch of
// VEC_CTAS * VEC_SUMS doubles; ks->ticket must be zero before the first use.
// Most CTAs of a vector reduction (2 x 152 SMs), and sums per CTA of one
// (Krylov dimension 16 and one): kernels and their scratch go by these.
constexpr int VEC_CTAS = 304, VEC_SUMS = 17;
// ks reset, ks->nb = |x|, q0 = x / |x|
cudaError_t k_lanczos_begin(const double* x, int64_t n, double* partial, KrylovState* ks, double* q0, cudaStream_t s);
// step k of K after w = H q_k: alpha_k, beta_k and q_{k+1} (in Q); the last
// step leaves the normalised coefficients of exp(t T) e_1 in ks and adds the
// log of the norm to rs.  Three launches, two for the last step.
cudaError_t k_lanczos_step(double* Q, int64_t ldq, int k, int K, double* w, int64_t n, double* partial, KrylovState* ks,
                           RhoScalars* rs, double breakdown_tol, double t, cudaStream_t s);
// y = sum_j ks->c[j] q_j
cudaError_t k_lanczos_end(const double* Q, int64_t ldq, const KrylovState* ks, double* y, int64_t n, cudaStream_t s);

// The same exponential, the digit gather and the Cholesky factors in the fixed
// arithmetic of a padded state's first beta-step (tt_settle.cu).
cudaError_t k_settle_begin(const double* x, int64_t n, double* partial, KrylovState* ks, double* q0, cudaStream_t s);
cudaError_t k_settle_step(double* Q, int64_t ldq, int k, int K, double* w, int64_t n, double* partial, KrylovState* ks,
                          double breakdown_tol, cudaStream_t s);
cudaError_t k_settle_end(const double* Q, int64_t ldq, KrylovState* ks, double t, int K, double* y, int64_t n,
                         double* partial, RhoScalars* rs, cudaStream_t s);
cudaError_t launch_gather_digits_rows(const DevGather& g, const Bases& b, cudaStream_t s);
cudaError_t launch_chol_rows(const CholJob* jobs, int njobs, double* ws, int* fail, cudaStream_t s, int maxn, bool df);

// v /= ||v||, logscale += ln ||v|| (rs->bad set on zero / non-finite norm)
cudaError_t k_normalise_inplace(double* v, int64_t n, double* partial, KrylovState* ks, RhoScalars* rs, cudaStream_t s);

// Householder QR of a batch of column-major matrices in workspace `ws`.
cudaError_t launch_qr(const QrJob* jobs, int njobs, double* ws, cudaStream_t s);
// The same factorisation of one matrix over the whole GPU (tt_qrgrid.cu): A, Q
// (m x n) and R (n x n) column-major, not overlapping; scratch of
// qr_grid_scratch(m, n) bytes.  qr_grid_ctas: the CTAs it takes, 0 where it does not
// apply.  *done is false where the device refused the launch; otherwise *err points
// at a device int that is set when a bounded wait (wait_ns) ran out.
cudaError_t qr_grid_ctas(int m, int n, int* ctas);
size_t qr_grid_scratch(int m, int n);
cudaError_t launch_qr_grid(const double* A, int m, int n, int ctas, double* Q, double* R, void* scratch,
                           long long wait_ns, cudaStream_t s, int** err, bool* done);
// one job passed by value (the record is a kernel argument, not device memory)
cudaError_t launch_qr_job(const QrJob& job, double* ws, cudaStream_t s);
// the same, only for the jobs whose only[job] != 0
// Householder QR of the jobs whose flag in `only` is set; *nrun (if not null)
// counts the sectors factorised.
cudaError_t launch_qr_masked(const QrJob* jobs, int njobs, double* ws, const int* only, int* nrun, cudaStream_t s);
// Cholesky + triangular inverse per job (shifted on request); fail[sec] set on
// a non-positive pivot.
// maxn: the largest n of the jobs (those up to 232 in shared memory); df:
// double-float arithmetic (~2^-46) instead of FP64.
cudaError_t launch_chol_inv(const CholJob* jobs, int njobs, double* ws, int* fail, cudaStream_t s, int maxn = 0,
                            bool df = false);
// Sign fix diag(R) >= 0 done inside launch_qr.

// Per-block item of the local measurement (d = 4 local space, <= 4 pairs).
struct ObsItem {
  long long off;
  int dl, m, dr, pad;
  double wn[4], wd[4];
};
// out[0] += sum A T w_n ; out[1] += sum A T w_d  (partial: 2 * nitems doubles)
cudaError_t launch_local_obs(const ObsItem* items, int nitems, const double* A, const double* T, double* partial,
                             double* out, cudaStream_t s);
// column-major a (ld): by_col ? a[:, c] *= s[c] : a[r, :] *= s[r]
cudaError_t launch_scale_rc(double* a, long long ld, int rows, int cols, const double* sv, int by_col, cudaStream_t s);

// *out = x . y (deterministic two-stage reduction)
cudaError_t k_dot_plain(const double* x, const double* y, int64_t n, double* partial, double* out, cudaStream_t s);

}  // namespace tt

// The device arithmetic of tt_df.h compiled for the host (the few CUDA bit
// intrinsics it uses restated here).  Test infrastructure only.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>

template <class To, class From>
static To bits(From v) {
  To r;
  static_assert(sizeof(To) == sizeof(From), "bit cast");
  std::memcpy(&r, &v, sizeof r);
  return r;
}
static unsigned __float_as_uint(float f) { return bits<unsigned>(f); }
static float __uint_as_float(unsigned u) { return bits<float>(u); }
static long long __double_as_longlong(double d) { return bits<long long>(d); }
static double __longlong_as_double(long long v) { return bits<double>(v); }
static double __hiloint2double(int hi, int lo) {
  return bits<double>(((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo);
}
static unsigned __funnelshift_rc(unsigned lo, unsigned hi, unsigned n) {
  const uint64_t v = ((uint64_t)hi << 32) | lo;
  return (unsigned)(v >> (n < 32 ? n : 32));
}
static float __double2float_rn(double d) { return (float)d; }

// CUDA's rsqrtf is within 2 ulp: h_ulps away from the rounded one
static int h_off = 0;
static float rsqrtf(float x) {
  return __uint_as_float(__float_as_uint((float)(1.0 / std::sqrt((double)x))) + (unsigned)h_off);
}

#include "tt_df.h"

extern "C" void h_pairs(const float* hi, const float* lo, double* out, int64_t n) {
  for (int64_t i = 0; i < n; ++i) out[i] = tt::dbl_of_pair(hi[i], lo[i]);
}

// 1 / sqrt and sqrt of pairs, rsqrtf `off` ulps from the rounded one
extern "C" void h_roots(const double* d, int off, double* rh, double* rl, double* sh, double* sl, int64_t n) {
  h_off = off;
  for (int64_t i = 0; i < n; ++i) {
    float2 v = tt::df_split(d[i]);
    v = tt::df_two_sum(v.x, v.y);
    const float2 r = tt::df_rsqrt(v), s = tt::df_sqrt(v, r);
    rh[i] = r.x; rl[i] = r.y; sh[i] = s.x; sl[i] = s.y;
  }
}

// a[i] - sum over 8 of b c, as a rank-8 update takes them
extern "C" void h_rank8(const double* a, const double* b, const double* c, double* out, int64_t n) {
  auto pair = [](double v) { const float2 p = tt::df_split(v); return tt::df_two_sum(p.x, p.y); };
  for (int64_t i = 0; i < n; ++i) {
    float2 acc = pair(a[i]);
    for (int s = 0; s < 8; ++s) {
      tt::df_fnms(acc, pair(b[8 * i + s]), pair(c[8 * i + s]));
      tt::df_tidy(acc);
    }
    out[i] = (double)acc.x + (double)acc.y;
  }
}

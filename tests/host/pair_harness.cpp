// The device arithmetic of tt_df.h compiled for the host (the few CUDA bit
// intrinsics it uses restated here).  Test infrastructure only.
#include <cuda_runtime.h>

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

#include "tt_df.h"

extern "C" void h_pairs(const float* hi, const float* lo, double* out, int64_t n) {
  for (int64_t i = 0; i < n; ++i) out[i] = tt::dbl_of_pair(hi[i], lo[i]);
}

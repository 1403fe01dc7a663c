// Double-float device arithmetic: a value as a pair of floats (Dekker; Knuth TAOCP
// vol. 2, 4.2.2), for work that GB300's FP64 pipe (2 multiply-adds per clock and
// SM, 72 clocks for one in a dependent chain) would hold up.
#pragma once
#include <cuda_runtime.h>

namespace tt {

// v = hi + lo: hi the top 24 significant bits of v (truncated), lo the other
// 29 rounded to 24 (error <= 2^-47 |v|), by integer operations on the FP64 bit
// pattern (no FP64 arithmetic); zero for zero and FP64 subnormals, FP64
// conversions for |v| outside [2^-97, 2^127]
__device__ __forceinline__ float2 df_split(double v) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(v));
  const int e = (int)((b >> 52) & 0x7FF);
  if (e == 0) return make_float2(0.f, 0.f);
  if (e < 926 || e > 1150) {
    const float h = __double2float_rn(v);
    return make_float2(h, __double2float_rn(v - (double)h));
  }
  const unsigned sg = (unsigned)(b >> 32) & 0x80000000u;
  const float hi = __uint_as_float(sg | ((unsigned)(e - 896) << 23) | (unsigned)((b >> 29) & 0x7FFFFFu));
  // low 29 mantissa bits times 2^(e - 1075) = (ml 2^-29) 2^(e - 1046), e - 1046 >= -120
  const float lo = ((float)(unsigned)(b & 0x1FFFFFFFull) * 1.862645149230957e-09f) *
                   __uint_as_float((unsigned)(e - 1046 + 127) << 23);
  return make_float2(hi, __uint_as_float(__float_as_uint(lo) | sg));
}

// FP64 value of a normal float by integer operations (exponent rebias and
// mantissa shift); zero for zero and float subnormals
__device__ __forceinline__ double dbl_of_float(float f) {
  const unsigned u = __float_as_uint(f);
  const unsigned e = (u >> 23) & 0xFF;
  if (e == 0) return 0.0;
  const unsigned long long b = ((unsigned long long)(u & 0x80000000u) << 32) |
                               ((unsigned long long)(e - 127 + 1023) << 52) |
                               ((unsigned long long)(u & 0x7FFFFFu) << 29);
  return __longlong_as_double((long long)b);
}

// hi + lo as FP64 by integer operations (two conversions and an addition on the
// FP64 pipe cost 192 clocks of an SM sub-partition per warp): renormalised by
// TwoSum to |t| <= ulp(s) / 2, then the mantissas added, t's truncated at 2^-53 of
// s.  Infinities and NaN pass through; FP32 subnormals give zero.
__device__ __forceinline__ double dbl_of_pair(float hi, float lo) {
  const float s = hi + lo;
  const float bp = s - hi;
  const float t = (hi - (s - bp)) + (lo - bp);
  const unsigned us = __float_as_uint(s), ut = __float_as_uint(t);
  int es = (us >> 23) & 0xFF;
  const int et = (ut >> 23) & 0xFF;
  const unsigned sign = us & 0x80000000u;
  if (es == 0) return 0.0;
  if (es == 255)
    return __hiloint2double((int)(sign | 0x7FF00000u | ((us & 0x7FFFFFu) >> 3)), (int)(us << 29));
  const unsigned mt = et ? (ut & 0x7FFFFFu) | 0x800000u : 0u;
  const int sh = es - et - 29;  // >= -5
  const unsigned T = sh >= 0 ? (sh < 32 ? mt >> sh : 0u) : mt << -sh;
  unsigned long long m = (unsigned long long)((us & 0x7FFFFFu) | 0x800000u) << 29;
  m = ((us ^ ut) >> 31) ? m - T : m + T;
  if (!(m >> 52)) {  // s a power of two, t of the other sign
    m <<= 1;
    --es;
  }
  return __longlong_as_double((long long)(((unsigned long long)sign << 32) | ((unsigned long long)(es + 896) << 52) |
                                          (m & 0xFFFFFFFFFFFFFull)));
}

}  // namespace tt

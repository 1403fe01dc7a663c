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
// FP64 pipe cost 192 clocks of an SM sub-partition per warp): renormalised by TwoSum
// to |t| <= ulp(s) / 2, then the mantissas added and rounded at half an ulp of the
// result (to nearest; of t what lies below half an ulp is dropped, error below 2^-53
// of the sum).  Sums outside [2^-71, 2^128) set `fp64` (the result is then no use):
// columns that a state gives no weight go down to FP32 subnormals and beyond, and
// their direction counts.
__device__ __forceinline__ double pair_bits(float hi, float lo, bool& fp64) {
  const float s = hi + lo;
  const float bp = s - hi;
  const float t = (hi - (s - bp)) + (lo - bp);
  const unsigned us = __float_as_uint(s), ut = __float_as_uint(t);
  const int es = (us >> 23) & 0xFF;
  fp64 = fp64 || ((unsigned)(es - 56) > 198u && s != 0.f);
  // in units of 2^-53 of s's leading bit: s in bits 30 .. 53, t at es - et >= 24
  // below it (none of it from 56 on; a zero t has et = 0)
  const unsigned T = __funnelshift_rc((ut & 0x7FFFFFu) << 6 | 0x20000000u, 0u, es - (int)((ut >> 23) & 0xFF) - 24);
  const unsigned long long ms = (unsigned long long)((us & 0x7FFFFFu) | 0x800000u) << 30;
  const unsigned long long m = ((us ^ ut) >> 31) ? ms - T : ms + T;
  const bool low = !(m >> 53);  // s a power of two, t of the other sign
  // (53 bits; the leading one, or a carry out of them, goes into the exponent)
  const unsigned long long v = ((unsigned long long)(es + (low ? 894 : 895)) << 52) + (low ? m : (m + 1) >> 1);
  return __longlong_as_double(
      (long long)(((unsigned long long)(us & 0x80000000u) << 32) + (s == 0.f ? 0ull : v)));
}
__device__ __forceinline__ double dbl_of_pair(float hi, float lo) {
  bool fp64 = false;
  const double v = pair_bits(hi, lo, fp64);
  return fp64 ? (double)hi + (double)lo : v;
}
// of N pairs, with one branch for all of them; exact: rounded as an FP64 addition
template <int N>
__device__ __forceinline__ void dbl_of_pairs(const float* hi, const float* lo, double* v, bool exact) {
  bool fp64 = exact;
  if (!exact) {
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = pair_bits(hi[i], lo[i], fp64);
  }
  if (fp64) {
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = (double)hi[i] + (double)lo[i];
  }
}

// Arithmetic on normalised pairs (|lo| <= ulp(hi) / 2), ~2^-46 relative.
__device__ __forceinline__ float2 df_two_sum(float s, float t) {
  const float h = s + t;
  const float bp = h - s;
  return make_float2(h, (s - (h - bp)) + (t - bp));
}
__device__ __forceinline__ float2 df_mul(float2 a, float2 b) {
  const float p = a.x * b.x;
  float e = fmaf(a.x, b.x, -p);
  e = fmaf(a.x, b.y, e);
  e = fmaf(a.y, b.x, e);
  return df_two_sum(p, e);
}
// a - b c; the result is not normalised
__device__ __forceinline__ void df_fnms(float2& a, float2 b, float2 c) {
  const float p = b.x * c.x;
  float e = fmaf(b.x, c.x, -p);  // b.x c.x = p + e exactly
  e = fmaf(b.x, c.y, e);
  e = fmaf(b.y, c.x, e);
  const float s = a.x - p;  // a.x - p = s + t exactly
  const float bp = s - a.x;
  const float t = (a.x - (s - bp)) + (-p - bp);
  a.y += t - e;
  a.x = s;
}
// normalises in three operations (Dekker's order: the high part is the larger, or
// both are rounding errors of what cancelled).  Without it after each of 8 terms
// the low part grows, and a Cholesky factor of n = 180 is 1.5 times further from
// its matrix (rms of R^T R - G: 1.6e-15 against 1.1e-15 of the diagonal).
__device__ __forceinline__ void df_tidy(float2& a) {
  const float h = a.x + a.y;
  a.y = a.y - (h - a.x);
  a.x = h;
}
// 1 / sqrt(d): y the float rsqrt and e = 1 - d y^2 as a pair (|e| < 2^-20), then
// y (1 + e / 2 + 3 e^2 / 8) with the product by e / 2 as a pair: 2^-46.9 (in one FP32
// term: 2^-44)
__device__ __forceinline__ float2 df_rsqrt(float2 d) {
  const float y = rsqrtf(d.x);
  const float qh = y * y, ql = fmaf(y, y, -qh);
  const float th = d.x * qh;
  float tl = fmaf(d.x, qh, -th);
  tl = fmaf(d.x, ql, tl);
  tl = fmaf(d.y, qh, tl);
  const float2 e = df_two_sum(1.f - th, -tl);
  const float g = 0.5f * y, p = g * e.x;
  const float q = fmaf(y, fmaf(0.375f * e.x, e.x, 0.5f * e.y), fmaf(g, e.x, -p));
  const float2 r = df_two_sum(y, p);
  return df_two_sum(r.x, r.y + q);
}
// sqrt(d) from ip = 1 / sqrt(d): s = d ip, corrected by (d - s^2) ip / 2
__device__ __forceinline__ float2 df_sqrt(float2 d, float2 ip) {
  const float2 s = df_mul(d, ip);
  float2 r = d;
  df_fnms(r, s, s);
  return df_two_sum(s.x, fmaf((r.x + r.y) * 0.5f, ip.x, s.y));
}

}  // namespace tt

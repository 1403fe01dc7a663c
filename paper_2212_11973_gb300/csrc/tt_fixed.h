// Fixed-point digits of FP64 and two-float values for the exact-accumulation split
// (Ozaki scheme; see tt_ozaki.cu), in 32-bit integer and FP32 operations.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace tt {

// Balanced base-256 digits of F = round(v 2^(1054 - emax)), emax >= the biased
// exponent of v (so |F| <= 2^32): F = a0 2^24 + a1 2^16 + a2 2^8 + a3 with a1,
// a2, a3 in [-128, 127] (TOPDOWN: each digit the rounding of what is left, so that
// a1 and a2 may be 128; 0.4 % of the values differ, and with them the products
// of the lowest orders that are dropped), returned as the bits of the FP32 integers (|a| <= 256,
// so their upper halves are the BF16 digits).  Zero and subnormal v give 0.
// With F' = F + 2^23 + 2^15 + 2^7 the digits are F' >> 24 and the lower bytes of
// F' less 128; a byte b becomes a float as 2^23 + b (a byte permute), less
// 2^23 + 128.
template <bool TOPDOWN>
__device__ __forceinline__ void fixed_digit_bits(double v, int emax, uint32_t* d) {
  const uint32_t vh = (uint32_t)__double2hiint(v), vl = (uint32_t)__double2loint(v);
  const int E = (int)((vh >> 20) & 0x7FF);
  const uint32_t mh = (vh & 0xFFFFFu) | 0x100000u;  // 53-bit mantissa mh:vl
  const int s = 20 + emax - E;                      // shift less one, >= 20
  // (mantissa >> s) + 1 >> 1, at most 33 bits
  uint32_t lo = s < 32 ? __funnelshift_r(vl, mh, s) : (s < 64 ? mh >> (s - 32) : 0u);
  uint32_t hi = s < 32 ? mh >> s : 0u;
  const bool carry = lo == 0xFFFFFFFFu;
  lo += 1u;
  hi += carry ? 1u : 0u;
  lo = __funnelshift_r(lo, hi, 1);
  hi >>= 1;
  if (E == 0) { lo = 0u; hi = 0u; }
  // signed, plus the bias: 64-bit two's complement
  long long F = (long long)(((unsigned long long)hi << 32) | lo);
  F = (vh >> 31) ? -F : F;
  const float bias = 8388736.f;  // 2^23 + 128
  if (TOPDOWN) {
    // a digit plus 128: what the digits above leave, biased to be positive, plus half
    const uint32_t g = (uint32_t)F;
    const uint32_t u1 = (((g + 0x800000u) & 0xFFFFFFu) + 0x8000u) >> 16;
    const uint32_t u2 = (((g + 0x8000u) & 0xFFFFu) + 0x80u) >> 8;
    const uint32_t u3 = (g + 0x80u) & 0xFFu;
    d[0] = __float_as_uint((float)(int)((F + 0x800000ll) >> 24));
    d[1] = __float_as_uint(__uint_as_float(0x4B000000u | u1) - bias);
    d[2] = __float_as_uint(__uint_as_float(0x4B000000u | u2) - bias);
    d[3] = __float_as_uint(__uint_as_float(0x4B000000u | u3) - bias);
    return;
  }
  F += 0x808080ll;
  const uint32_t g = (uint32_t)F;
  const int a0 = (int)(F >> 24);
  d[0] = __float_as_uint((float)a0);
  d[1] = __float_as_uint(__uint_as_float(__byte_perm(g, 0x4B000000u, 0x7542)) - bias);
  d[2] = __float_as_uint(__uint_as_float(__byte_perm(g, 0x4B000000u, 0x7541)) - bias);
  d[3] = __float_as_uint(__uint_as_float(__byte_perm(g, 0x4B000000u, 0x7540)) - bias);
}

// biased FP64 exponent of a float (0 for zero / subnormal)
__device__ __forceinline__ int fexp(float v) {
  const int e = (__float_as_int(v) >> 23) & 0xFF;
  return e == 0 ? 0 : e + 896;
}

// 2^x for -126 <= x <= 127 from the exponent field
__device__ __forceinline__ float p2f(int x) { return __int_as_float((x + 127) << 23); }

// two-float c (hi, lo) += coef * (xh + xl), coef split into (ch, cl)
__device__ __forceinline__ void df_fma(float& sh, float& sl, float ch, float cl, float xh, float xl) {
  const float p = ch * xh;
  const float pe = fmaf(ch, xh, -p) + (ch * xl + cl * xh);
  const float s = sh + p;
  const float bp = s - sh;
  const float ap = s - bp;
  sl += ((sh - ap) + (p - bp)) + pe;
  sh = s;
}

// Balanced base-256 digits of round(S + Sl) (a normalised two-float value,
// |Sl| <= ulp(S) / 2, |S| < 2^31, scaled so that the row's bound is 2^31), in
// FP32 arithmetic only: every step is exact, the roundings are those of rintf.  Returned as the BF16 bit
// patterns (the digits are integers of magnitude <= 256, so their FP32 and
// BF16 forms agree in the upper 16 bits).
__device__ __forceinline__ void digits_of_pair(float S, float Sl, uint32_t* d) {
  const float R = rintf(S);
  const float f = (S - R) + Sl;
  const float a0 = rintf(R * 5.9604644775390625e-08f);   // R / 2^24
  const float rem = (R - a0 * 16777216.f) + rintf(f);    // |rem| < 2^24
  const float a1 = rintf(rem * 1.52587890625e-05f);      // rem / 2^16
  const float r1 = rem - a1 * 65536.f;
  const float a2 = rintf(r1 * 0.00390625f);              // r1 / 2^8
  const float a3 = r1 - a2 * 256.f;
  d[0] = __float_as_uint(a0);
  d[1] = __float_as_uint(a1);
  d[2] = __float_as_uint(a2);
  d[3] = __float_as_uint(a3);
}

}  // namespace tt

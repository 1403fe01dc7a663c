// Fixed-point digits of FP64 values for the exact-accumulation split (Ozaki
// scheme; see tt_ozaki.cu), in 32-bit integer and FP32 operations.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace tt {

// Balanced base-256 digits of F = round(v 2^(1054 - emax)), emax >= the biased
// exponent of v (so |F| <= 2^32): F = a0 2^24 + a1 2^16 + a2 2^8 + a3 with a1,
// a2, a3 in [-128, 127], returned as the bits of the FP32 integers (|a| <= 256,
// so their upper halves are the BF16 digits).  Zero and subnormal v give 0.
// With F' = F + 2^23 + 2^15 + 2^7 the digits are F' >> 24 and the lower bytes of
// F' less 128; a byte b becomes a float as 2^23 + b (a byte permute), less
// 2^23 + 128.
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
  F += 0x808080ll;
  const uint32_t g = (uint32_t)F;
  const int a0 = (int)(F >> 24);
  const float bias = 8388736.f;  // 2^23 + 128
  d[0] = __float_as_uint((float)a0);
  d[1] = __float_as_uint(__uint_as_float(__byte_perm(g, 0x4B000000u, 0x7542)) - bias);
  d[2] = __float_as_uint(__uint_as_float(__byte_perm(g, 0x4B000000u, 0x7541)) - bias);
  d[3] = __float_as_uint(__uint_as_float(__byte_perm(g, 0x4B000000u, 0x7540)) - bias);
}

}  // namespace tt

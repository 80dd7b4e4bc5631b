// Conversions between FP32 and FP64 on the integer pipe.
//
// This part issues FP64 instructions, conversions included, at about 1.6 per
// clock per SM, so a kernel that touches every sample in FP64 is bound by their
// number.  A conversion is a handful of 32-bit integer operations (128 per clock
// per SM); both functions return exactly what the casts do.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace vl {
namespace bits {

// (float)d, round to nearest even
__device__ __forceinline__ float to_float(double d) {
  const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
  const uint32_t e = (hi >> 20) & 0x7ffu;
  if (e - 897u > 252u) return (float)d;  // zero, or outside the normal FP32 range
  // exponent (mod 2^9) and the leading 23 mantissa bits, exponent rebiased
  uint32_t f = (__funnelshift_l(lo, hi, 3) - (896u << 23)) & 0x7fffffffu;
  const uint32_t rem = lo << 3;  // what is cut off, half an ulp = 2^31
  f += rem > 0x80000000u || (rem == 0x80000000u && (f & 1u));
  return __uint_as_float(f | (hi & 0x80000000u));
}

// (double)f
__device__ __forceinline__ double to_double(float f) {
  const uint32_t b = __float_as_uint(f), m = b & 0x7fffffffu;
  if (m - 0x00800000u > 0x7effffffu && m != 0u) return (double)f;  // subnormal, inf, nan
  const uint32_t hi = (b & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u);
  return __hiloint2double((int)hi, (int)(b << 29));
}

// 2^e as a double, -1022 <= e <= 1023
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((e + 1023) << 20, 0); }

}  // namespace bits
}  // namespace vl

// FP64 <-> pair of FP32 (hi + lo) through integer operations, host and device.
// GB300 issues two FP64 operations or conversions per cycle and SM, and the plain
// forms (round, widen, subtract, round; widen, widen, add) bound the permutations:
// 16 columns of 327,680 values in 62 (with the column maxima) and out 45 us, with
// these 53 and 31.
#pragma once

#include "h2_digits.hpp"   // bits_float

namespace h2 {

__host__ __device__ __forceinline__ uint32_t float_bits(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  uint32_t b;
  std::memcpy(&b, &f, sizeof b);
  return b;
#endif
}
__host__ __device__ __forceinline__ uint64_t double_bits(double v) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(v);
#else
  uint64_t b;
  std::memcpy(&b, &v, sizeof b);
  return b;
#endif
}
__host__ __device__ __forceinline__ double bits_double(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double v;
  std::memcpy(&v, &b, sizeof v);
  return v;
#endif
}

// hi = v rounded to 24 bits, lo = the rest rounded to 24 bits; |lo| <= ulp(hi) / 2
__host__ __device__ __forceinline__ void double_to_pair(double v, float &hi, float &lo) {
  const uint64_t w = double_bits(v);
  const uint32_t e = (uint32_t)(w >> 52) & 0x7ffu;
  if (e - 953u <= 170u) {   // 2^-70 <= |v| < 2^101: both parts are normal
    const uint32_t sign = (uint32_t)(w >> 32) & 0x80000000u;
    // the significand rounded to 23 fraction bits (a carry steps the exponent); the
    // exponent rebased by 896 = 1023 - 127, modulo 2^32
    const uint32_t u = (uint32_t)((w + (1ull << 28)) >> 29) - (896u << 23);
    hi = bits_float((u & 0x7fffffffu) | sign);
    // the 29 bits below, from -2^28 to 2^28 - 1 units of 2^(e - 1075)
    const int32_t t = (int32_t)((uint32_t)w << 3) >> 3;
    lo = (float)t * bits_float(((e - 948u) << 23) | sign);
  } else {
    hi = (float)v;
    lo = (float)(v - (double)hi);
  }
}

// f widened (exact)
__host__ __device__ __forceinline__ double widen(float f) {
  const uint32_t b = float_bits(f), a = b & 0x7fffffffu;
  if (a - 0x00800000u < 0x7f000000u)   // normal
    return bits_double(((uint64_t)((b & 0x80000000u) | ((a >> 3) + (896u << 20))) << 32) | (uint64_t)(a << 29));
  return a == 0u ? bits_double((uint64_t)b << 32) : (double)f;
}

}  // namespace h2

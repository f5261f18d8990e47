// convert.cuh -- exact FP32 -> FP64 conversion on bit patterns.
//
// Every FP32 value is exactly representable in FP64; the conversion only
// re-biases the exponent (127 -> 1023), moves the 23 fraction bits to the top
// of the 52, normalises subnormal inputs (an FP32 subnormal m 2^-149 is a
// normal FP64 number) and keeps zeros, infinities and NaNs (payload moved the
// same way).  Done in the integer pipe because this part issues two FP64
// instructions per clock per SM.  Host-compilable so that it can be checked
// against the compiler's conversion for every class of input.
#pragma once
#include <stdint.h>

#if defined(__CUDACC__)
#define CONV_HD __host__ __device__ __forceinline__
#else
#define CONV_HD static inline
#endif

CONV_HD int conv_clz32(uint32_t x) {
#if defined(__CUDA_ARCH__)
  return __clz(x);
#else
  return x ? __builtin_clz(x) : 32;
#endif
}

CONV_HD uint64_t f32_to_f64_bits(uint32_t b) {
  const uint64_t sign = (uint64_t)(b >> 31) << 63;
  const uint32_t e = (b >> 23) & 0xffu, m = b & 0x7fffffu;
  if (e == 0xffu) return sign | (0x7ffull << 52) | ((uint64_t)m << 29);
  if (e != 0u) return sign | ((uint64_t)(e + 896u) << 52) | ((uint64_t)m << 29);
  if (m == 0u) return sign;
  const int sh = conv_clz32(m) - 8;  // moves the leading bit to position 23
  return sign | ((uint64_t)(897 - sh) << 52) | ((uint64_t)((m << sh) & 0x7fffffu) << 29);
}

// Whether f32_pair_sum_bits covers hi + lo: the larger is normal, the other zero or
// normal and less than 2^29 times smaller, so the sum has at most 53 bits.
CONV_HD bool f32_pair_sum_covers(uint32_t hi, uint32_t lo) {
  const uint32_t mh = hi & 0x7fffffffu, ml = lo & 0x7fffffffu;
  const uint32_t a = mh > ml ? mh : ml, b = mh > ml ? ml : mh;
  return a - 0x00800000u < 0x7f000000u && (b == 0u || (b >= 0x00800000u && (a >> 23) - (b >> 23) <= 28u));
}

// hi + lo as binary64 bits, exactly, with integer operations: mantissas on the
// smaller exponent's grid, one 64-bit addition, the leading bit moved to place.
CONV_HD uint64_t f32_pair_sum_bits(uint32_t hi, uint32_t lo) {
  const uint32_t mh = hi & 0x7fffffffu, ml = lo & 0x7fffffffu;
  const uint32_t a = mh > ml ? mh : ml, b = mh > ml ? ml : mh;
  const uint32_t sign = (mh > ml ? hi : lo) & 0x80000000u;  // equal magnitudes: 0 or twice, both of lo's sign
  const uint32_t ea = a >> 23;
  const uint32_t d = b ? ea - (b >> 23) : 0u;
  const uint64_t big = (uint64_t)((a & 0x7fffffu) | 0x800000u) << d;
  const uint32_t small = b ? (b & 0x7fffffu) | 0x800000u : 0u;
  const uint64_t m = (int32_t)(hi ^ lo) < 0 ? big - small : big + small;
  if (m == 0) return 0;  // exact cancellation: +0
  const uint32_t top = (uint32_t)(m >> 32);
  const int lz = top ? conv_clz32(top) : 32 + conv_clz32((uint32_t)m);
  // leading bit 63 - lz of m counts 2^(63 - lz + ea - d - 150)
  const uint32_t e = 63u - (uint32_t)lz + ea - d - 150u + 1023u;
  return ((uint64_t)sign << 32) + ((uint64_t)(e - 1u) << 52) + (m << (lz - 11));
}

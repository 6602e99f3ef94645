// convert.cuh -- float <-> double in integer arithmetic: conversions to and
// from 64-bit types run at GB300's float64 rate, a small fraction of its
// integer rate.
#pragma once
#include <cstdint>
#include <cstring>

namespace nlc {

__host__ __device__ __forceinline__ unsigned float_bits(float v) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(v);
#else
  unsigned b;
  memcpy(&b, &v, 4);
  return b;
#endif
}
__host__ __device__ __forceinline__ float float_of(unsigned b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float v;
  memcpy(&v, &b, 4);
  return v;
#endif
}
__host__ __device__ __forceinline__ double double_of(unsigned hi, unsigned lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double((int)hi, (int)lo);
#else
  const uint64_t b = ((uint64_t)hi << 32) | lo;
  double v;
  memcpy(&v, &b, 8);
  return v;
#endif
}
__host__ __device__ __forceinline__ unsigned hi_word(double v) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2hiint(v);
#else
  uint64_t b;
  memcpy(&b, &v, 8);
  return (unsigned)(b >> 32);
#endif
}
__host__ __device__ __forceinline__ unsigned lo_word(double v) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2loint(v);
#else
  uint64_t b;
  memcpy(&b, &v, 8);
  return (unsigned)b;
#endif
}

// Exact float -> double in integer arithmetic (conversions to and from
// 64-bit types run at the float64 rate).  Denormals count as zero, as in the
// rest of the float32 code (-ftz).
__host__ __device__ __forceinline__ double widen(float v) {
  const unsigned b = float_bits(v), m = b & 0x7fffffffu;
  unsigned hi = (m >> 3) + 0x38000000u;           // rebias 127 -> 1023
  hi = m >= 0x7f800000u ? hi + 0x38000000u : hi;  // infinities and NaN
  hi = m < 0x00800000u ? 0u : hi;
  const unsigned lo = m < 0x00800000u ? 0u : b << 29;
  return double_of(hi | (b & 0x80000000u), lo);
}
__host__ __device__ __forceinline__ double widen(double v) { return v; }

// The nearest float (ties to even), likewise in integer arithmetic; results
// below the normal range are zero.
__host__ __device__ __forceinline__ float narrow(double v) {
  const unsigned hi = hi_word(v), lo = lo_word(v), m = hi & 0x7fffffffu;
  unsigned f = ((m - 0x38000000u) << 3) | (lo >> 29);
  const unsigned rest = lo & 0x1fffffffu;
  f += (rest > 0x10000000u || (rest == 0x10000000u && (f & 1u))) ? 1u : 0u;
  f = m < 0x38100000u ? 0u : f;                                // below 2^-126
  f = m >= 0x47f00000u ? 0x7f800000u : f;                      // 2^128 and above
  f = m > 0x7ff00000u || (m == 0x7ff00000u && lo) ? 0x7fffffffu : f;  // NaN
  return float_of(f | (hi & 0x80000000u));
}
template <class G>
__host__ __device__ __forceinline__ G store_as(double v) {
  if constexpr (sizeof(G) == 4)
    return narrow(v);
  else
    return v;
}

}  // namespace nlc

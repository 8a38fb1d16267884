// fdlb_cvt.cuh -- binary32 <-> binary64 conversions on the integer pipe.
//
// GB300 converts between the two on the binary64 pipe, 2 values per clock and
// SM, which bounds the kernels that set or read a state of binary32 pairs: at
// 2048 x 2048 cells of 128 populations, a pair's three binary64 operations
// take 2.6 ms.  The widening and the round-to-nearest-even below give the same
// bits as the conversions (to which narrow still sends values outside
// binary32's normal range).
#pragma once

#include <cstdint>
#include <cstring>

#include "fdlb_mp9.cuh"  // dbits, dfrom

namespace fdlb {

__device__ __forceinline__ uint32_t fbits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t b;
  std::memcpy(&b, &x, 4);
  return b;
#endif
}
__device__ __forceinline__ float ffrom(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float x;
  std::memcpy(&x, &b, 4);
  return x;
#endif
}

// (double)x, without a branch: denormals are scaled by 2^64 first, infinities
// and NaN get the larger exponent field
__device__ __forceinline__ double widen(float x) {
  const bool small = (fbits(x) & 0x7fffffffu) < 0x00800000u;
  const uint32_t b = fbits(small ? x * 18446744073709551616.0f : x), m = b & 0x7fffffffu;
  uint32_t hi = (m >> 3) + (small ? 832u << 20 : 896u << 20);
  hi += m >= 0x7f800000u ? 896u << 20 : 0u;
  hi = m == 0 ? 0u : hi;
  return dfrom((long long)(((uint64_t)((b & 0x80000000u) | hi) << 32) | (b << 29)));
}

// (float)v, round to nearest even
__device__ __forceinline__ float narrow(double v) {
  const uint64_t b = (uint64_t)dbits(v);
  const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b, m = hi & 0x7fffffffu;
  // binary32 normals: exponents 2^-126 .. 2^127
  if (m - (897u << 20) >= (254u << 20) && (m | lo) != 0) return (float)v;
  uint32_t u = (m << 3 | lo >> 29) - (896u << 23);
  const uint32_t rem = lo & 0x1fffffffu;
  u += rem > 0x10000000u || (rem == 0x10000000u && (u & 1u));
  if ((m | lo) == 0) u = 0;
  return ffrom((hi & 0x80000000u) | u);
}

// v as the unevaluated sum of two binary32 values
__device__ __forceinline__ void split_pair(double v, float& h, float& l) {
  h = narrow(v);
  l = narrow(v - widen(h));
}

}  // namespace fdlb

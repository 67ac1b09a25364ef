// Conversions of FP64 values to narrower formats on the integer pipe.
#pragma once
#include <string.h>

#include "ok_internal.cuh"

namespace okgb {

// GB300's FP64 pipe, the conversions to and from FP64 with it, runs at 1/58 of the FP32 rate, so the
// kernels that only pass FP64 data on are bound by their conversions.  These give bit for bit what
// the conversion gives, from 32-bit integer operations, and use the conversion itself outside the
// range where the integer form holds.
__host__ __device__ __forceinline__ void double_words(double d, unsigned& hi, unsigned& lo) {
#ifdef __CUDA_ARCH__
  hi = (unsigned)__double2hiint(d);
  lo = (unsigned)__double2loint(d);
#else
  unsigned long long D;
  memcpy(&D, &d, sizeof D);
  hi = (unsigned)(D >> 32);
  lo = (unsigned)D;
#endif
}
__host__ __device__ __forceinline__ float float_bits(unsigned u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float f;
  memcpy(&f, &u, sizeof f);
  return f;
#endif
}

// The 24 leading bits of |d|'s significand in place of a float's, biased exponent ed - 896 beside it; `low` the 29
// bits that follow.  `ok`: |d| in [2^-74, 2^127).
struct SplitBits {
  unsigned top, low, sign, ed;
  bool ok;
};
__host__ __device__ __forceinline__ SplitBits split_bits(double d) {
  unsigned h, l;
  double_words(d, h, l);
  SplitBits s;
  s.ed = (h >> 20) & 0x7ffu;
  s.sign = h & 0x80000000u;
  s.top = ((h & 0x7fffffffu) - (896u << 20)) << 3 | l >> 29;   // (exponent - 896) << 23 | 23 bits
  s.low = l & 0x1fffffffu;
  s.ok = s.ed - (1023u - 74u) <= 74u + 126u;
  return s;
}

// d rounded to odd at 24 bits: rounding the result to 22 bits or fewer (to FP16) rounds d itself.
__host__ __device__ __forceinline__ float float_odd_of(double d) {
  const SplitBits s = split_bits(d);
  if (!s.ok) return (float)d;   // |d| < 2^-74 is zero in FP16 and |d| >= 2^127 infinite, however rounded here
  return float_bits(s.sign | s.top | (s.low != 0u));
}

// Double-float split of d: hi = RN_float(d), lo = RN_float(d - hi), the value dd(d) defines (lo is a
// normal float or zero in the range of the integer form).
__host__ __device__ __forceinline__ dd split_df(double d) {
  const SplitBits s = split_bits(d);
  if (!s.ok) return dd(d);
  const unsigned up = s.low > 0x10000000u - (s.top & 1u);
  int rem = (int)s.low - (int)(up << 29);   // |rem| <= 2^28: half a float ulp
  if (s.sign) rem = -rem;
  // lo = rem 2^(ed - 1075) (zero stays +0), the power of two a normal float
  const float scale = float_bits((s.ed - 1075u + 127u) << 23);
#ifdef __CUDA_ARCH__
  const float lo = __int2float_rn(rem) * scale;
#else
  const float lo = (float)rem * scale;
#endif
  return dd(float_bits(s.sign | (s.top + up)), lo);
}

}  // namespace okgb

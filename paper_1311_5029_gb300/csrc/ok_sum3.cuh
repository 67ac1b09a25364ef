// Sums with more than FP64's accuracy on the FP32 pipes (the training step's loss and gradient).
#pragma once
#include <math.h>

#include "ok_internal.cuh"

namespace okgb {

// The product as a rounded value of its own: never contracted into the sum that follows.
__host__ __device__ __forceinline__ float mul_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  volatile float p = a * b;
  return p;
#endif
}

// s + t + u: three floats of falling size, what each sum drops caught by the next (Ogita, Rump and Oishi, SIAM J.
// Sci. Comput. 26 (2005)).
struct Sum3 {
  float s, t, u;
  __host__ __device__ __forceinline__ double value() const { return (double)s + ((double)t + (double)u); }
};
// acc += x; returns the exact rounding error (Knuth).
__host__ __device__ __forceinline__ float two_sum(float& acc, float x) {
  const float s = acc + x, bb = s - acc;
  const float e = (acc - (s - bb)) + (x - bb);
  acc = s;
  return e;
}
__host__ __device__ __forceinline__ Sum3 operator+(Sum3 a, Sum3 b) {
  const float r = two_sum(a.s, b.s), q = two_sum(a.t, b.t);
  a.u += b.u + (q + two_sum(a.t, r));
  return a;
}
// a += (d + e)^2, d + e a difference and its rounding error (|e| <= 2^-24 |d|).
__host__ __device__ __forceinline__ void add_square(Sum3& a, float d, float e) {
  const float p = mul_rn(d, d), q = fmaf(d, d, -p);        // d^2 = p + q
  const float c = 2.f * d, x = mul_rn(c, e), y = fmaf(c, e, -x);  // 2 d e = x + y
  float r = two_sum(a.s, p);
  r = two_sum(a.t, r);
  r += two_sum(a.t, q);
  r += two_sum(a.t, x);
  a.u += r + (y + mul_rn(e, e));
}
__host__ __device__ __forceinline__ void add_square(Sum3& a, float d) {
  const float p = mul_rn(d, d), q = fmaf(d, d, -p);
  float r = two_sum(a.s, p);
  r = two_sum(a.t, r);
  a.u += r + two_sum(a.t, q);
}

// v[0] += |x|^2, v[1] += |o - x|^2 over N complex numbers.  Each of the two sums is taken in three floats (some 70
// bits) when its own largest component, of x or of o - x, lies in [2^-40, 2^40]: there a square and
// its rounding error fit FP32's range, and what a smaller component loses below 2^-149 is 2^-69 of the sum or less.
// Otherwise, and with NaN, it is taken in FP64 component by component.
template <int N>
__host__ __device__ __forceinline__ void loss_chunk(const float2 (&o)[N], const float2 (&x)[N], double (&v)[2]) {
  float mx = 0.f, md = 0.f;
  bool nan = false;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const float dr = o[k].x - x[k].x, di = o[k].y - x[k].y;
    mx = fmaxf(fmaxf(mx, fabsf(x[k].x)), fabsf(x[k].y));
    md = fmaxf(fmaxf(md, fabsf(dr)), fabsf(di));
    nan = nan || dr != dr || di != di;   // also for a NaN or two infinities in o and x
  }
  const float lo = 0x1p-40f, hi = 0x1p40f;
  if (mx >= lo && mx <= hi && !nan) {
    Sum3 a{0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < N; ++k) {
      add_square(a, x[k].x);
      add_square(a, x[k].y);
    }
    v[0] += a.value();
  } else if (mx != 0.f || nan) {
#pragma unroll
    for (int k = 0; k < N; ++k) v[0] += (double)x[k].x * x[k].x + (double)x[k].y * x[k].y;
  }
  if (md >= lo && md <= hi && !nan) {
    Sum3 a{0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < N; ++k) {
      float d = o[k].x, e = two_sum(d, -x[k].x);
      add_square(a, d, e);
      d = o[k].y;
      e = two_sum(d, -x[k].y);
      add_square(a, d, e);
    }
    v[1] += a.value();
  } else if (md != 0.f || nan) {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const double er = (double)o[k].x - x[k].x, ei = (double)o[k].y - x[k].y;
      v[1] += er * er + ei * ei;
    }
  }
}

}  // namespace okgb

// Grid reductions whose sums run on the FP32 pipes: the double-float form of ok_reduce.cuh.
#pragma once

#include "ok_reduce.cuh"

namespace okgb {

// ---------------------------------------------------------------------------- FP32-pipe grid sums
// The reductions of the FP32 kernels keep every partial sum as a double-float pair (hi + lo, two
// floats, about 44 significand bits; ok_internal.cuh): each thread adds its chunk sums into pairs,
// each block sums its threads' pairs with a fixed shuffle tree, and the last block sums the block
// partials the same way before the FP64 finalisation.  All of it runs on the FP32 pipes.  FP64
// arithmetic runs at 1/58 of the FP32 rate on this part; done in FP64, the block trees cost more
// than streaming the vectors, and the last block's tree kept one SM busy for about 6 us after the
// others had finished.  The order of every sum is fixed by the launch shape.
template <typename R> struct RedT { using T = double; };
template <> struct RedT<float> { using T = dd; };
__device__ __forceinline__ void red_add(double& a, double c) { a += c; }
__device__ __forceinline__ void red_add(dd& a, float c) { a = a + dd(c, 0.f); }
__device__ __forceinline__ dd shfl_xor_dd(dd a, int o) {
  return dd(__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o));
}

template <int NP, int THREADS>
__device__ __forceinline__ void block_sums_dd(dd (&v)[NP], dd (*sh)[THREADS / 32]) {
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    dd x = v[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = x + shfl_xor_dd(x, o);
    if ((threadIdx.x & 31) == 0) sh[k][threadIdx.x >> 5] = x;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      dd x = sh[k][0];
      for (int w = 1; w < THREADS / 32; ++w) x = x + sh[k][w];
      v[k] = x;
    }
  }
  __syncthreads();
}

// grid_reduce (ok_reduce.cuh) in double-float: block partials stored as pairs of floats in the slots of
// the doubles (no FP64 conversion on the way), the last block sums them and finalises.
template <int NP, int THREADS>
__device__ __forceinline__ void grid_reduce_dd(dd (&v)[NP], const RedArgs& ra, unsigned* ticket) {
  __shared__ dd sh[NP][THREADS / 32];
  __shared__ int last;
  block_sums_dd<NP, THREADS>(v, sh);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < NP; ++k) reinterpret_cast<float2*>(ra.part)[(size_t)blockIdx.x * NP + k] = make_float2(v[k].hi, v[k].lo);
    __threadfence();
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  dd w[NP];
#pragma unroll
  for (int k = 0; k < NP; ++k) w[k] = dd(0.f, 0.f);
  for (unsigned b = threadIdx.x; b < gridDim.x; b += THREADS)
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      const float2 f = __ldcg(reinterpret_cast<const float2*>(ra.part) + (size_t)b * NP + k);
      w[k] = w[k] + dd(f.x, f.y);
    }
  block_sums_dd<NP, THREADS>(w, sh);
  if (threadIdx.x == 0) {
    *ticket = 0u;
    double tot[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < NP && k < 4; ++k) tot[k] = (double)w[k];
    if (ra.out) {
#pragma unroll
      for (int k = 0; k < NP; ++k) ra.out[k] = tot[k];
    }
    finalise(ra.st, ra.fin, tot);
  }
}

}  // namespace okgb

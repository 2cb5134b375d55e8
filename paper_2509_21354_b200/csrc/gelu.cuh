// GELU in its exact form x * Phi(x) for the aggregator MLP kernels (Eq. 2), two values at a time.
//   x Phi(x) = max(x, 0) - |x| Q(|x|),  Q = 1 - Phi the upper tail,  Q(a) = 2^(-g(a)).
// g is so close to a parabola that a polynomial of degree 6 does: fitted here by least squares with weights iterated towards
// the least maximum (Lawson's method) of the resulting error in a Q(a) on 0 <= a <= 6.  Absolute error of the result
// 5.1e-8 in exact arithmetic, 8.1e-8 with every step rounded to fp32 (the erf formula 7.1.26 of Abramowitz and Stegun, used
// before with an exponential and a reciprocal: 2.1e-7).  8 fp32 operations and one exponential per value, in packed
// pairs.  Beyond a = 6 the tail is held at 6 Q(6) = 6e-9 (the min also keeps infinities out of the polynomial); NaN stays NaN.
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

namespace kve {

// nan-propagating max(x, 0)
__device__ __forceinline__ float relu_nan(float x) {
  float y;
  asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(y) : "f"(x));
  return y;
}

// relu: max(x, 0); a: |x|, at most 6; result: the tail Q(a).  x Phi(x) = relu - a * Q
__device__ __forceinline__ float2 gelu_tail2(float2 x, float2& relu, float2& a) {
  a = make_float2(fminf(fabsf(x.x), 6.f), fminf(fabsf(x.y), 6.f));
  relu = make_float2(relu_nan(x.x), relu_nan(x.y));
  constexpr float G[7] = {-0.999993061f, -1.1512017f, -0.458770975f, -0.0534121019f, 0.00808071511f, -0.00076921928f, 3.30927681e-05f};
  float2 p = make_float2(G[6], G[6]);
#pragma unroll
  for (int k = 5; k >= 0; --k) p = fma2(p, a, make_float2(G[k], G[k]));
  return make_float2(ex2_fast(p.x), ex2_fast(p.y));
}

__device__ __forceinline__ float2 gelu2(float2 x) {
  float2 relu, a;
  const float2 q = gelu_tail2(x, relu, a);
  return fma2(make_float2(-a.x, -a.y), q, relu);
}

}  // namespace kve

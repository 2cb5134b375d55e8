// GELU in its exact form x * Phi(x) for the aggregator MLP kernels (Eq. 2), two values at a time.
//   x Phi(x) = max(x, 0) - |x| Q(|x|),  Q = 1 - Phi the upper tail.
// With a = |x| sqrt(log2(e) / 2), so that exp(-x^2 / 2) = 2^(-a^2):  |x| Q(|x|) = 2^(-a^2) a R(a), and a R(a) = |x| Q e^(x^2/2)
// is a smooth bounded function (Mills' ratio times |x|).  R is a polynomial of degree 9, fitted here by least squares
// with weights iterated towards the least maximum (Lawson's method) of the error times 2^(-a^2) on 0 <= a <= 5: absolute error of
// the result 2.0e-7 in exact arithmetic, 2.4e-7 with every step rounded to fp32 (the erf formula 7.1.26 of Abramowitz
// and Stegun, used before with two special-function operations: 2.1e-7).  14 fp32 operations and one exponential per
// value, in packed pairs.  Beyond a = 12 the exponential is 0 (min also keeps infinities out of the polynomial); NaN stays NaN.
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

namespace kve {

constexpr float GELU_SCALE = 0.84932178f;      // sqrt(log2(e) / 2)

// nan-propagating max(x, 0)
__device__ __forceinline__ float relu_nan(float x) {
  float y;
  asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(y) : "f"(x));
  return y;
}

// u = x * GELU_SCALE of two values -> relu: max(u, 0), and the tail 2^(-a^2) a as `ea` with its factor R(a) as the result:
// x Phi(x) = relu / GELU_SCALE - ea * R
__device__ __forceinline__ float2 gelu_tail2(float2 u, float2& relu, float2& ea) {
  const float2 a = make_float2(fminf(fabsf(u.x), 12.f), fminf(fabsf(u.y), 12.f));
  relu = make_float2(relu_nan(u.x), relu_nan(u.y));
  const float2 s = mul2(a, a);
  ea = mul2(make_float2(ex2_fast(-s.x), ex2_fast(-s.y)), a);
  constexpr float R[10] = {0.5886920094f, -0.5527806878f, 0.4061160386f, -0.2486497015f, 0.1271331608f,
                           -0.0520748980f, 0.0159405991f, -0.0033308757f, 0.0004155426f, -2.3050154e-05f};
  float2 p = make_float2(R[9], R[9]);
#pragma unroll
  for (int k = 8; k >= 0; --k) p = fma2(p, a, make_float2(R[k], R[k]));
  return p;
}

__device__ __forceinline__ float2 gelu2(float2 x) {
  float2 relu, ea;
  const float2 p = gelu_tail2(mul2(x, make_float2(GELU_SCALE, GELU_SCALE)), relu, ea);
  return fma2(make_float2(-ea.x, -ea.y), p, make_float2(relu_nan(x.x), relu_nan(x.y)));
}

}  // namespace kve

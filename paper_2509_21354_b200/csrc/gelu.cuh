// GELU in its exact form x * Phi(x) for the aggregator MLP kernels (Eq. 2), two values at a time.
//   x Phi(x) = max(x, 0) - |x| Q(|x|),  Q = 1 - Phi the upper tail,  Q(a) = 2^(-g(a)).
// g is so close to a parabola that a polynomial of low degree does: fitted here by least squares with weights iterated
// towards the least maximum (Lawson's method) of the resulting error in a Q(a) on 0 <= a <= 6.  Error of the result for
// x ~ N(0, 1) with every step rounded to fp32: degree 6: rms 3.7e-8, max 9.4e-8; degree 8: rms 1.0e-8, max 4.9e-8 (the erf
// formula 7.1.26 of Abramowitz and Stegun, used before with an exponential and a reciprocal: rms 4.9e-8, max 2.1e-7).
// Degree 8 where the tensor cores bound the kernel and the activations are free (the chunk means' MLP: 219.8 us a step with
// either on 256 sequences x 4096 tokens); degree 6 where the activations bound it and are averaged over a chunk's tokens anyway
// (the per-token MLP: 381 us a step with 6, 395 with 7, 406 with 8).  Beyond a = 6 the tail is held at 6 Q(6) = 6e-9 (the
// min also keeps infinities out of the polynomial); NaN stays NaN.
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

// coefficients of -g at degree 6, lowest first (the per-token MLP, which has the steps of several values side by side)
#define KVE_GELU_TAIL6 {-0.999993061f, -1.1512017f, -0.458770975f, -0.0534121019f, 0.00808071511f, -0.00076921928f, 3.30927681e-05f}

// x Phi(x) at degree 8
__device__ __forceinline__ float2 gelu2(float2 x) {
  constexpr float G8[9] = {-0.999998868f, -1.15112329f, -0.459115446f, -0.0527141988f, 0.00733338343f, -0.00032334181f, -0.000114462782f,
                           2.50833236e-05f, -1.69040277e-06f};
  const float2 a = make_float2(fminf(fabsf(x.x), 6.f), fminf(fabsf(x.y), 6.f)), relu = make_float2(relu_nan(x.x), relu_nan(x.y));
  float2 p = make_float2(G8[8], G8[8]);
#pragma unroll
  for (int k = 7; k >= 0; --k) p = fma2(p, a, make_float2(G8[k], G8[k]));
  return fma2(make_float2(-a.x, -a.y), make_float2(ex2_fast(p.x), ex2_fast(p.y)), relu);
}

}  // namespace kve

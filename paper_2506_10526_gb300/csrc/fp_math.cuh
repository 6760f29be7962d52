// Elementary functions of the kernels whose time is arithmetic, each with its
// derivation and the error measured over every argument it may get.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

namespace bsi {
namespace fpm {

// Packed FP32 pairs: one instruction for two values.
__device__ __forceinline__ uint64_t pk(float a, float b) {
  return (uint64_t)__float_as_uint(a) | ((uint64_t)__float_as_uint(b) << 32);
}
__device__ __forceinline__ float lo_f(uint64_t v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi_f(uint64_t v) { return __uint_as_float((uint32_t)(v >> 32)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// tanh of two values, about 11 instructions each and no branch.
//  |x| < 0.6875: x + x^3 P(x^2).  P, of degree 4, is the weighted minimax fit (Lawson's
//  iteratively reweighted least squares on Chebyshev nodes, the coefficients rounded to
//  FP32 one after the other, the rest fitted again) of (tanh(x) / x - 1) / x^2; it is
//  off by 1.3e-8 of tanh, the rest is rounding.
//  Above: 1 - 2 e / (1 + e) with e = exp(-2 |x|).  The subtracted part is at most 0.41
//  against 0.59, so the errors of the approximate exponential and reciprocal enter with
//  a weight of 0.7 at the switch, below a quarter from 1.1 on.
// Over every FP32 argument from 2^-13 to 16 the result is within 1.8e-7 relative of tanh
// and its mean over a binade within 1e-8 of that of the rounded tanh (CUDA's tanhf on the
// same device: 2.0e-7, and 3e-8 between 0.25 and 0.55); below 2^-13 tanh(x) = x to
// rounding; zeros keep their sign, NaN stays NaN, infinities give 1.  Inference of
// 1540 x 60^2 rows: 1.86 ms; a switch at 0.875 and degree 5 (1.4e-7) takes 0.04 ms more,
// at 1.125 and degree 7 (8.7e-8) 0.08, the exponential branch in packed operations 0.04.
__device__ __forceinline__ void tanh_pair(float x0, float x1, float &y0, float &y1) {
  const float a0 = fabsf(x0), a1 = fabsf(x1);
  const float e0 = ex2(a0 * -2.88539008f), e1 = ex2(a1 * -2.88539008f);  // 2^(-2 log2(e) |x|)
  const float g0 = fmaf(e0, rcp(fmaf(e0, -0.5f, -0.5f)), 1.f);
  const float g1 = fmaf(e1, rcp(fmaf(e1, -0.5f, -0.5f)), 1.f);
  const uint64_t a = pk(a0, a1), q = mul2(a, a);
  uint64_t p = fma2(q, pk(-0.00523358723f, -0.00523358723f), pk(0.0201927293f, 0.0201927293f));
  p = fma2(q, p, pk(-0.0535953492f, -0.0535953492f));
  p = fma2(q, p, pk(0.133296251f, 0.133296251f));
  p = fma2(q, p, pk(-0.333332121f, -0.333332121f));
  const uint64_t small = fma2(mul2(q, a), p, a);
  y0 = copysignf(a0 < 0.6875f ? lo_f(small) : g0, x0);
  y1 = copysignf(a1 < 0.6875f ? hi_f(small) : g1, x1);
}

}  // namespace fpm
}  // namespace bsi

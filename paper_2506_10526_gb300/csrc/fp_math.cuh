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
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
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

// tanh of two values for the gradient.  |x| >= 0.55: (1 - e) / (1 + e) with one residual
// step on the quotient, so that the reciprocal's error, which has one sign, does not add
// up over the rows in 1 - tanh^2; below: x + x^3 P(x^2) with a least-squares fit of
// degree 4.  Within 2.3e-7 relative over the same arguments, its mean over a binade
// within 2e-8.  The gradient of 20000 rows is off by 3e-8 (RMS, of its largest entry)
// with this, 4e-8 with CUDA's tanhf.  Kept beside tanh_pair, which is closer and
// shorter, because training carries any change of rounding on: after 24 steps the loss
// differs by up to 4e-5 between the two.
__device__ __forceinline__ void tanh_pair_grad(float x0, float x1, float &y0, float &y1) {
  const float a0 = fabsf(x0), a1 = fabsf(x1);
  const uint64_t a = pk(a0, a1), one = pk(1.f, 1.f);
  const uint64_t u = mul2(a, pk(-2.88539008f, -2.88539008f));  // -2 log2(e) |x|
  const uint64_t e = pk(ex2(lo_f(u)), ex2(hi_f(u)));
  const uint64_t den = add2(e, one);
  const uint64_t num = fma2(e, pk(-1.f, -1.f), one), rd = pk(rcp(lo_f(den)), rcp(hi_f(den)));
  uint64_t big = mul2(num, rd);
  big = fma2(fma2(big, pk(-lo_f(den), -hi_f(den)), num), rd, big);
  const uint64_t q = mul2(a, a);
  uint64_t p = fma2(q, pk(-0.00626437f, -0.00626437f), pk(0.02106414f, 0.02106414f));
  p = fma2(q, p, pk(-0.0538503f, -0.0538503f));
  p = fma2(q, p, pk(0.13332564f, 0.13332564f));
  p = fma2(q, p, pk(-0.33333317f, -0.33333317f));
  const uint64_t small = fma2(mul2(q, a), p, a);
  y0 = copysignf(a0 < 0.55f ? lo_f(small) : lo_f(big), x0);
  y1 = copysignf(a1 < 0.55f ? hi_f(small) : hi_f(big), x1);
}

// (x - mu) / sd for many x per column, two columns at a time.  The product with a stored
// reciprocal r has two roundings and overflows where r does; one residual step,
// q + (a - q s) r with the remainder from a fused multiply-add (Markstein, IBM J. Res.
// Dev. 34, 1990), takes the quotient to the rounding of a division at five
// operations.  Inference of 1540 x 60^2 rows: 1.842 ms with the product alone, 1.866
// with the residual step, 0.3 more with divisions.  The deviation is scaled by a power of two (c) into [0.5, 1), so
// that r exists for every deviation.
struct __align__(16) DivPair {
  float2 nmu, c, r, ns;  // -mu, power of two, 1 / (sd c), -(sd c)
};
__device__ __forceinline__ void div_column(float mu, float sd, float &nmu, float &c, float &r,
                                           float &ns) {
  int k = 0;
  frexpf(sd, &k);  // sd = f 2^k, f in [0.5, 1)
  k = max(-126, min(126, k));
  c = __uint_as_float((uint32_t)(127 - k) << 23);
  nmu = -mu;
  ns = isinf(sd) ? 0.f : -(sd * c);  // an infinite deviation: r = 0, quotients 0
  r = 1.f / (sd * c);
}
__device__ __forceinline__ void normalise_pair(float x0, float x1, const DivPair &t, float &u0,
                                               float &u1) {
  const float a0 = (x0 + t.nmu.x) * t.c.x, a1 = (x1 + t.nmu.y) * t.c.y;
  const float q0 = a0 * t.r.x, q1 = a1 * t.r.y;
  u0 = fmaf(fmaf(q0, t.ns.x, a0), t.r.x, q0);
  u1 = fmaf(fmaf(q1, t.ns.y, a1), t.r.y, q1);
}
// The product alone, for the gradient (whose bits in training stay as they are).
__device__ __forceinline__ void scale_pair(float x0, float x1, const DivPair &t, float &u0, float &u1) {
  u0 = (x0 + t.nmu.x) * t.c.x * t.r.x;
  u1 = (x1 + t.nmu.y) * t.c.y * t.r.y;
}

// 1 / sqrt(s) in FP64 for s in FP32's normal range: an FP32 seed (relative error
// below 2^-19: the 20 leading mantissa bits of s, then rsqrtf) and one third-order
// step, y (1 + e / 2 + 3 e^2 / 8) with e = 1 - s y^2 (the start of the binomial series of
// (1 - e)^(-1/2)), whose error 5 e^3 / 16 is below 2^-55; with the roundings of s y and
// of the result less than 2^-52 relative.  Five FP64 operations, against a square root
// and a division.
__device__ __forceinline__ double rsqrt64(double s) {
  const uint32_t h = (uint32_t)__double2hiint(s);
  const uint32_t f = __float_as_uint(rsqrtf(__uint_as_float((h - (896u << 20)) << 3)));
  const double y = __hiloint2double((int)((f >> 3) + (896u << 20)), (int)(f << 29));
  const double e = __fma_rn(-__dmul_rn(s, y), y, 1.0);
  return __fma_rn(__dmul_rn(y, e), __fma_rn(0.375, e, 0.5), y);
}

}  // namespace fpm
}  // namespace bsi

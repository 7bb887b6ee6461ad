// What the two forms of the GLA read on the tensor cores share (fem_gla_tc.cu, fem_gla_par.cu).
#pragma once

#include "fem_common.cuh"

namespace fem {

constexpr int kGC = 128;  // steps per chunk (rows of S, TMEM lanes)
constexpr int kGM = 64;   // feature width
constexpr float kGlaLinBeta = 0.25f;  // channels below it take the linear bank

// expm1(y) / beta for y = beta x: x times the series of expm1(y) / y for |y| < 1/2
// (truncation below 4e-6 relative), (e^y - 1) / beta beyond (ex2.approx: the result
// is rounded to bf16); x itself at beta = 0.
__device__ __forceinline__ float em1_beta_fast(float x, float y, float rb) {
  float p = fmaf(y, 1.f / 720.f, 1.f / 120.f);  // both forms, then a select: no branch per element
  p = fmaf(y, p, 1.f / 24.f);
  p = fmaf(y, p, 1.f / 6.f);
  p = fmaf(y, p, 0.5f);
  p = fmaf(y, p, 1.f);
  const float far = (__expf(y) - 1.f) * rb;
  return fabsf(y) < 0.5f ? x * p : far;
}

// log1p(x) for x > -1: the series to x^5 for |x| < 2^-6 (truncation below 2^-36
// relative), lg2.approx of 1 + x beyond.
__device__ __forceinline__ float log1p_fast(float x) {
  float p = fmaf(x, 0.2f, -0.25f);  // both forms, then a select
  p = fmaf(x, p, 1.f / 3.f);
  p = fmaf(x, p, -0.5f);
  p = fmaf(x, p, 1.f);
  const float far = __logf(1.f + x);
  return fabsf(x) < 0.015625f ? x * p : far;
}

}  // namespace fem

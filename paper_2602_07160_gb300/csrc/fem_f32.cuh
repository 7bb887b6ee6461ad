// Loads and elementary functions shared by the tiled fp32 kernels (the read and its gradients).
#pragma once

#include "fem_common.cuh"

namespace fem {

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16 *p) {
  const uint2 w = *reinterpret_cast<const uint2 *>(p);
  return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                     __uint_as_float(w.y & 0xffff0000u));
}
__device__ __forceinline__ float ld1(const float *p) { return *p; }
__device__ __forceinline__ float ld1(const __nv_bfloat16 *p) { return __bfloat162float(*p); }

// Four consecutive channels j .. j + 3 of a row (zero past d); rows are 16-byte (fp32) or 8-byte
// (bf16) aligned when d is a multiple of four.
template <typename In>
__device__ __forceinline__ float4 ld_row4(const In *row, int j, int d, bool vec) {
  if (vec) return j < d ? ld4(row + j) : make_float4(0.f, 0.f, 0.f, 0.f);
  return make_float4(j < d ? ld1(row + j) : 0.f, j + 1 < d ? ld1(row + j + 1) : 0.f, j + 2 < d ? ld1(row + j + 2) : 0.f,
                     j + 3 < d ? ld1(row + j + 3) : 0.f);
}

// expm1(y) / beta with y = beta x for two linear channels (inv_b = 1 / beta, e = e^y); x at beta = 0.
// The series of expm1(y)/y for |y| < 1/2 (truncation below 2e-7 relative), (e^y - 1) / beta beyond.
__device__ __forceinline__ float2 em1_over_beta2(float2 x, float2 y, float2 e, float2 inv_b) {
  float2 p = __ffma2_rn(y, make_float2(1.f / 5040.f, 1.f / 5040.f), make_float2(1.f / 720.f, 1.f / 720.f));
  p = __ffma2_rn(y, p, make_float2(1.f / 120.f, 1.f / 120.f));
  p = __ffma2_rn(y, p, make_float2(1.f / 24.f, 1.f / 24.f));
  p = __ffma2_rn(y, p, make_float2(1.f / 6.f, 1.f / 6.f));
  p = __ffma2_rn(y, p, make_float2(0.5f, 0.5f));
  p = __ffma2_rn(y, p, make_float2(1.f, 1.f));
  p = __fmul2_rn(x, p);
  return make_float2(fabsf(y.x) < 0.5f ? p.x : (e.x - 1.f) * inv_b.x,
                     fabsf(y.y) < 0.5f ? p.y : (e.y - 1.f) * inv_b.y);
}

// exp(beta (x - c)) with the exponent to twice fp32's precision (the rounding errors of x - c and of
// the product enter to first order): an exponent of -60 costs no more accuracy than one near zero,
// which the gradients need of the read (they take exp(beta (v - o)) of its output).
__device__ __forceinline__ float exp_tilt(float b, float x, float c) {
  const float d = x - c, z = d - x, derr = (x - (d - z)) - (c + z);
  const float y = b * d, ylo = fmaf(b, d, -y) + b * derr, e = expf(y);
  return fabsf(y) < 80.f ? fmaf(e, ylo, e) : e;
}

}  // namespace fem

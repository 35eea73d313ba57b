// Device arithmetic: the BF16 / FP8 conversions of the step executor
// (hiccl_runtime.cu) and the sweep kernels (hiccl_sweep_kernels.cuh), and the executor's
// combine operators (the sweeps combine many sources at a time with their own).
#pragma once

#include <cuda_runtime.h>

#include "hiccl_internal.h"

namespace hiccl {

// one step of a fold on 32-bit lanes: f32 (IEEE RNE add, maxNum, minNum) or
// i32 (wrapping add, max, min, logical or)
__device__ __forceinline__ float comb_f(float a, float b, uint32_t rop) {
  return rop == HICCL_SUM ? __fadd_rn(a, b) : rop == HICCL_MAX ? fmaxf(a, b) : fminf(a, b);
}
__device__ __forceinline__ uint32_t comb32(uint32_t a, uint32_t b, uint32_t dt, uint32_t rop) {
  if (dt == HICCL_F32) return __float_as_uint(comb_f(__uint_as_float(a), __uint_as_float(b), rop));
  const int x = (int)a, y = (int)b;
  switch (rop) {
    case HICCL_SUM: return a + b;
    case HICCL_MAX: return (uint32_t)(x > y ? x : y);
    case HICCL_MIN: return (uint32_t)(x < y ? x : y);
    default: return (x != 0 || y != 0) ? 1u : 0u;
  }
}
__device__ __forceinline__ uint4 add4(uint4 a, uint4 b, uint32_t dt, uint32_t rop = 0) {
  if (rop == HICCL_SUM && dt == HICCL_F32) {
    a.x = __float_as_uint(__fadd_rn(__uint_as_float(a.x), __uint_as_float(b.x)));
    a.y = __float_as_uint(__fadd_rn(__uint_as_float(a.y), __uint_as_float(b.y)));
    a.z = __float_as_uint(__fadd_rn(__uint_as_float(a.z), __uint_as_float(b.z)));
    a.w = __float_as_uint(__fadd_rn(__uint_as_float(a.w), __uint_as_float(b.w)));
  } else if (rop == HICCL_SUM) {   // int32, wrapping
    a.x += b.x;
    a.y += b.y;
    a.z += b.z;
    a.w += b.w;
  } else {
    a.x = comb32(a.x, b.x, dt, rop);
    a.y = comb32(a.y, b.y, dt, rop);
    a.z = comb32(a.z, b.z, dt, rop);
    a.w = comb32(a.w, b.w, dt, rop);
  }
  return a;
}

// ---- reduced-precision payloads -------------------------------------------
// BF16: the upper half of a binary32; rounding to nearest even by cvt.rn.
__device__ __forceinline__ uint32_t f32_to_bf16_rn(float x) {
  unsigned short h;
  asm("cvt.rn.bf16.f32 %0, %1;" : "=h"(h) : "f"(x));
  return h;
}
// two binary32 -> two BF16 (round to nearest even) in one word; the first
// value lands in the low half
__device__ __forceinline__ uint32_t f32x2_to_bf16x2(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}
// FP8 e4m3 (1 sign, 4 exponent bits with bias 7, 3 mantissa bits, no
// infinities, S.1111.111 = NaN): four codes (byte k of w gives component k)
// -> four binary32 values, exactly.  Every e4m3 value is a binary16 value;
// binary16 -> binary32 is a mixed-precision add of -0 (x + -0 = x for every x,
// signed zeros included), measured slightly faster here than cvt.f32.f16.
__device__ __forceinline__ float4 e4m3x4_to_f32x4(uint32_t w) {
  float4 r;
  asm("{\n\t.reg .b16 lo, hi, a, b, c, d;\n\t.reg .b32 h0, h1;\n\t"
      "mov.b32 {lo, hi}, %4;\n\t"
      "cvt.rn.f16x2.e4m3x2 h0, lo;\n\tcvt.rn.f16x2.e4m3x2 h1, hi;\n\t"
      "mov.b32 {a, b}, h0;\n\tmov.b32 {c, d}, h1;\n\t"
      "add.rn.f32.f16 %0, a, 0f80000000;\n\tadd.rn.f32.f16 %1, b, 0f80000000;\n\t"
      "add.rn.f32.f16 %2, c, 0f80000000;\n\tadd.rn.f32.f16 %3, d, 0f80000000;\n\t}"
      : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w)
      : "r"(w));
  return r;
}
// two binary32 -> two e4m3 codes (round to nearest even, saturating at 448);
// the first value lands in the low byte
__device__ __forceinline__ uint32_t f32x2_to_e4m3x2(float lo, float hi) {
  unsigned short d;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(d) : "f"(hi), "f"(lo));
  return d;
}

}  // namespace hiccl

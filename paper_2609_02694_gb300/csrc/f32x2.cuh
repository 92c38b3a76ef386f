// f32x2.cuh -- packed pairs of FP32 values. sm_103a adds, multiplies and multiply-adds two
// FP32 values held in a register pair with one instruction, each half rounded as the scalar
// instruction rounds it. A kernel bound by instruction issue, with its FMA pipe half idle,
// spends half the slots on the same arithmetic.
#pragma once
#include <cuda_runtime.h>

namespace rbe {

using f32x2 = float2;

__device__ __forceinline__ f32x2 pk(float lo, float hi) { return make_float2(lo, hi); }
__device__ __forceinline__ f32x2 pk(float v) { return make_float2(v, v); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) { return __ffma2_rn(a, b, c); }
// Kahan summation of both halves; s - c is formed as fma(c, -1, s), the same rounding.
__device__ __forceinline__ void kahan_add2(f32x2 &s, f32x2 &c, f32x2 x) {
  const f32x2 m1 = pk(-1.f);
  const f32x2 y = fma2(c, m1, x);
  const f32x2 t = add2(s, y);
  c = fma2(y, m1, fma2(s, m1, t));
  s = t;
}

}  // namespace rbe

// Packed pairs of FP32 numbers and of double-floats (unevaluated sums of two
// FP32 numbers, Dekker 1971, Knuth's two-sum): one instruction for two lanes.
#pragma once
#include <cuda_runtime.h>

__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }

// ---------------------------------------------------------------------------
// packed double-float
// ---------------------------------------------------------------------------
struct d2 {
  float2 h, l;
};
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return add2(a, neg2(b)); }
__device__ __forceinline__ d2 dd_neg(d2 a) { return {neg2(a.h), neg2(a.l)}; }
// a + b exactly, |a| >= |b| or a == 0
__device__ __forceinline__ d2 fast_sum(float2 a, float2 b) {
  const float2 s = add2(a, b);
  return {s, sub2(b, sub2(s, a))};
}
__device__ __forceinline__ d2 two_sum(float2 a, float2 b) {
  const float2 s = add2(a, b), v = sub2(s, a);
  return {s, add2(sub2(a, sub2(s, v)), sub2(b, v))};
}
__device__ __forceinline__ d2 dd_add(d2 a, d2 b) {
  const d2 s = two_sum(a.h, b.h);
  return {s.h, add2(s.l, add2(a.l, b.l))};
}
__device__ __forceinline__ d2 dd_norm(d2 a) { return fast_sum(a.h, a.l); }
__device__ __forceinline__ d2 dd_mul(d2 a, d2 b) {
  const float2 p = mul2(a.h, b.h);
  float2 e = fma2(a.h, b.h, neg2(p));
  e = fma2(a.h, b.l, e);
  return {p, fma2(a.l, b.h, e)};
}

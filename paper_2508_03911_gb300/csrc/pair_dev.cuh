// pair_dev.cuh -- numbers as unevaluated sums hi + lo of two float32 (x = hi, y = lo; 48 bits):
// GB300 has 64 float32 units for each float64 one.
#pragma once
#include <cuda_runtime.h>

namespace hv {

// The exact sum of a and b as a pair (Knuth's two-sum).
__device__ __forceinline__ float2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  return make_float2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}

// p + x, renormalised.
__device__ __forceinline__ float2 pair_add(float2 p, float x) {
  const float2 t = two_sum(p.x, x);
  const float lo = p.y + t.y, hi = __fadd_rn(t.x, lo);
  return make_float2(hi, __fsub_rn(lo, __fsub_rn(hi, t.x)));
}

// p + q, renormalised.
__device__ __forceinline__ float2 pair_add(float2 p, float2 q) {
  const float2 s = two_sum(p.x, q.x);
  const float e = __fadd_rn(s.y, __fadd_rn(p.y, q.y)), h = __fadd_rn(s.x, e);
  return make_float2(h, __fsub_rn(e, __fsub_rn(h, s.x)));
}

}  // namespace hv

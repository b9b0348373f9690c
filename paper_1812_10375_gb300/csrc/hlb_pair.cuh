// Two neighbouring columns per thread: packed FP32 arithmetic (one instruction
// for both columns on sm_100 and later) and the exchange of edge columns inside
// a warp.  Every operation is written out (no compiler contraction), so that where a
// cell's update rounds is decided by its source, not by the loop it stands in.
#pragma once
#include "hlb_internal.cuh"

namespace hlb {

__device__ __forceinline__ float2 bc2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b, c - a b (a packed operand's sign turns for free)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 nfma2(float2 a, float2 b, float2 c) {
  return __ffma2_rn(make_float2(-a.x, -a.y), b, c);
}
// Packed operands live in register pairs, so operations with a constant are
// written per column: the constant stays an immediate or in the constant bank.
// Both forms take the FP32 pipe equally long (2.1 cycles for a packed
// instruction, 1.1 for a plain one).
__device__ __forceinline__ float2 cmul2(float2 a, float c) { return make_float2(__fmul_rn(a.x, c), __fmul_rn(a.y, c)); }
__device__ __forceinline__ float2 cfma2(float2 a, float c, float2 b) {
  return make_float2(__fmaf_rn(a.x, c, b.x), __fmaf_rn(a.y, c, b.y));
}
__device__ __forceinline__ float2 cfma2(float2 a, float c, float b) {
  return make_float2(__fmaf_rn(a.x, c, b), __fmaf_rn(a.y, c, b));
}
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float2 rcp2(float2 a) { return make_float2(rcp_approx(a.x), rcp_approx(a.y)); }

// The columns next to a lane's pair: w left of a.x (the previous lane's a.y), e
// right of a.y (the next lane's a.x).  The warp's outermost lanes read their own.
__device__ __forceinline__ void pair_edges(float2 a, float& w, float& e) {
  w = __shfl_up_sync(0xffffffffu, a.y, 1);
  e = __shfl_down_sync(0xffffffffu, a.x, 1);
}

// Compensated sum of both columns (TwoSum, as ff_add).
__device__ __forceinline__ void ff_add2(float2& hi, float2& lo, float2 x) {
  const float2 s = add2(hi, x);
  const float2 bp = sub2(s, hi);
  const float2 e = add2(sub2(hi, sub2(s, bp)), sub2(x, bp));
  hi = s;
  lo = add2(lo, e);
}

}  // namespace hlb

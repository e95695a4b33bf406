// Pairs of floats in one 64-bit register and their packed arithmetic (PTX
// add / mul / fma.rn.f32x2, sm_100 and later): two correctly rounded FP32
// operations per instruction, each the same as the scalar one.
#pragma once

namespace gs2d {

struct F2 {
  unsigned long long v;
};

__device__ __forceinline__ F2 make2(float lo, float hi) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ F2 dup2(float a) { return make2(a, a); }
__device__ __forceinline__ float2 split2(F2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
// two adjacent floats (8-byte aligned)
__device__ __forceinline__ F2 load2(const float* p) {
  return F2{*reinterpret_cast<const unsigned long long*>(p)};
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
// a - b (as a - 1 b: exact product, one rounding)
__device__ __forceinline__ F2 sub2(F2 a, F2 b) { return fma2(b, dup2(-1.f), a); }

// 1 / a.  kTame: a is positive and normal and so is its reciprocal; then the
// hardware approximation and one Newton step y + y (1 - a y) on the pair,
// within 1 ulp.  Otherwise two divisions: the step would make NaN of an infinite
// a, and zero of a reciprocal below the normal range.
template <bool kTame>
__device__ __forceinline__ F2 recip2(F2 a) {
  const float2 s = split2(a);
  if (!kTame) return make2(1.f / s.x, 1.f / s.y);
  const F2 y = make2(__fdividef(1.f, s.x), __fdividef(1.f, s.y));
  const F2 e = fma2(mul2(a, dup2(-1.f)), y, dup2(1.f));
  return fma2(y, e, y);
}

}  // namespace gs2d

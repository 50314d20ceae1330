// FP32 pairs (hi + lo, about 48 significant bits) for short FP64 sequences on
// FP32 data: GB300 executes 64 times as many FP32 as FP64 operations, and a
// pair operation is 5 to 11 of them (Dekker 1971, Knuth's two-sum; products'
// errors from fused multiply-adds).
#pragma once
#include <cuda_runtime.h>

namespace aeth {

struct dfloat {
  float h, l;
  __device__ __forceinline__ dfloat() {}
  __device__ __forceinline__ dfloat(float a) : h(a), l(0.0f) {}
  __device__ __forceinline__ dfloat(float a, float b) : h(a), l(b) {}
  // a double's leading 48 bits
  static __device__ __forceinline__ dfloat of(double a) {
    const float h = (float)a;
    return dfloat(h, (float)(a - (double)h));
  }
  __device__ __forceinline__ explicit operator float() const { return __fadd_rn(h, l); }
};

// a + b with |a| >= |b| or a = 0
__device__ __forceinline__ dfloat quick_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return dfloat(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ dfloat two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  return dfloat(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}
__device__ __forceinline__ dfloat operator-(const dfloat& a) { return dfloat(-a.h, -a.l); }
__device__ __forceinline__ dfloat operator+(const dfloat& a, const dfloat& b) {
  const dfloat s = two_sum(a.h, b.h);
  return quick_two_sum(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ dfloat operator-(const dfloat& a, const dfloat& b) { return a + (-b); }
__device__ __forceinline__ dfloat operator+(const dfloat& a, float b) {
  const dfloat s = two_sum(a.h, b);
  return quick_two_sum(s.h, __fadd_rn(s.l, a.l));
}
__device__ __forceinline__ dfloat operator*(const dfloat& a, const dfloat& b) {
  const float p = __fmul_rn(a.h, b.h);
  const float e = __fmaf_rn(a.h, b.h, -p);
  return quick_two_sum(p, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, e)));
}
__device__ __forceinline__ dfloat operator*(const dfloat& a, float b) {
  const float p = __fmul_rn(a.h, b);
  return quick_two_sum(p, __fmaf_rn(a.l, b, __fmaf_rn(a.h, b, -p)));
}
// 1 / a: the hardware reciprocal and one second-order correction
__device__ __forceinline__ dfloat reciprocal(const dfloat& a) {
  float q;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(q) : "f"(a.h));
  const float r = __fmaf_rn(-a.l, q, __fmaf_rn(-a.h, q, 1.0f));
  return quick_two_sum(q, __fmul_rn(q, __fmaf_rn(r, r, r)));
}

}  // namespace aeth

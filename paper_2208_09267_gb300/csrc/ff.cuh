// ff.cuh -- float-float arithmetic: an unevaluated sum h + l of two floats
// with |l| <= ulp(h)/2, about 48 significant bits.
//
// The FP64 pipe of this chip issues 2 lanes per clock and SM, the FP32 pipe
// 128: a float-float addition (about ten FP32 operations) costs a sixth of an
// FP64 one.  The operations are the error-free transformations of Knuth
// (two-sum), Dekker (fast two-sum, 1971) and, with an FMA, the exact product;
// intrinsics keep the compiler from contracting across them.  Absolute errors
// are a few 2^-48 of the operands; infinities become NaN in the low part and
// are not to be relied on.
#pragma once

namespace lbm {

struct ff {
  float h, l;
};

__device__ __forceinline__ ff ff_of(float a) { return {a, 0.f}; }
__device__ __forceinline__ ff ff_of(double a) {
  const float h = (float)a;
  return {h, (float)(a - (double)h)};
}
// the exact sum of two floats
__device__ __forceinline__ ff two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float t = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
// the exact sum of two floats, |a| >= |b| or a = 0
__device__ __forceinline__ ff fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
// the exact product of two floats
__device__ __forceinline__ ff two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ ff operator-(ff a) { return {-a.h, -a.l}; }
__device__ __forceinline__ ff operator+(ff a, ff b) {
  const ff s = two_sum(a.h, b.h);
  return fast_two_sum(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ ff operator-(ff a, ff b) { return a + (-b); }
__device__ __forceinline__ ff operator+(ff a, float b) {
  const ff s = two_sum(a.h, b);
  return fast_two_sum(s.h, __fadd_rn(s.l, a.l));
}
__device__ __forceinline__ ff operator*(ff a, ff b) {
  const ff p = two_prod(a.h, b.h);
  return fast_two_sum(p.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, p.l)));
}
__device__ __forceinline__ ff operator*(ff a, float b) {
  const ff p = two_prod(a.h, b);
  return fast_two_sum(p.h, __fmaf_rn(a.l, b, p.l));
}
// product with a power of two
__device__ __forceinline__ ff scaled(ff a, float p2) { return {a.h * p2, a.l * p2}; }
__device__ __forceinline__ ff operator/(ff a, ff b) {
  const float r = 1.0f / b.h;
  const float q = __fmul_rn(a.h, r);
  const ff e = a - b * q;
  return fast_two_sum(q, __fmul_rn(e.h, r));
}
__device__ __forceinline__ ff ff_sqrt(ff a) {
  const float y = sqrtf(a.h);
  if (!(y > 0.f)) return ff_of(y);
  const ff e = a - two_prod(y, y);
  return fast_two_sum(y, __fdiv_rn(e.h, 2.0f * y));
}

// Running sum of float-float terms: the high parts are summed without error,
// their errors and the low parts in float; total() renormalises.
struct ff_sum {
  float h = 0.f, l = 0.f;
  __device__ __forceinline__ void add(ff a) {
    const ff s = two_sum(h, a.h);
    h = s.h;
    l = __fadd_rn(l, __fadd_rn(s.l, a.l));
  }
  __device__ __forceinline__ ff total() const { return two_sum(h, l); }
};

}  // namespace lbm

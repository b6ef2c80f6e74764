// tf.cuh - triple-float arithmetic (an unevaluated sum h + m + l of three FP32
// numbers, about 70 bits) for the transforms of FP64 results: the pair sum of
// FP64 plans with the Gaussian envelope and the finish of the whole-lattice solve.
//
// A transform's rounding is relative to the largest values it holds, and the
// factors b_k of the envelopes multiply it by up to e^5 (b_k^2: e^10) at an output;
// in FP64 that was up to seven times the rounding of directly summed pairs (the
// norm of the coefficients' errors), and 30 times on separable tables of Eq. pure.
// Triple-float leaves it below one FP64 rounding.  It is also the cheaper one:
// a sum takes 21 FP32 operations and a product 25, half of them per issue slot as
// pairs (f32x2), where GB300 issues 128 FP32 operations per SM and clock and 2 FP64
// ones.
//
// As in df.cuh: Knuth's two-sum, Dekker's product with a fused multiply-add, parts
// not renormalised after cancellation (the value and its error, relative to the
// operands, stay as they are).  Parts follow Shewchuk's expansions (Discrete
// Comput. Geom. 18, 1997), cut off after the third.
#pragma once

#include "df.cuh"

namespace srm3 {

struct tf {
  float h, m, l;
  tf() = default;
  __host__ __device__ constexpr tf(double v)
      : h((float)v), m((float)(v - (double)h)), l((float)(v - (double)h - (double)m)) {}
  // the sum of two doubles, the second far smaller
  __host__ __device__ constexpr tf(double v, double w)
      : h((float)v), m((float)(v - (double)h)), l((float)((v - (double)h - (double)m) + w)) {}
  __host__ __device__ constexpr tf(float h_, float m_, float l_) : h(h_), m(m_), l(l_) {}
};

// A complex triple-float, the parts of its two components side by side.
struct __align__(8) tf2 {
  float2 h, m, l;
};

__device__ __forceinline__ tf operator+(tf a, tf b) {
  float e1, e2, e3;
  const float h = two_sum(a.h, b.h, e1);
  const float m = two_sum(two_sum(a.m, b.m, e2), e1, e3);
  return tf(h, m, __fadd_rn(__fadd_rn(a.l, b.l), __fadd_rn(e2, e3)));
}
__device__ __forceinline__ tf operator-(tf a) { return tf(-a.h, -a.m, -a.l); }
__device__ __forceinline__ tf operator-(tf a, tf b) { return a + (-b); }
__device__ __forceinline__ tf operator*(tf a, tf b) {
  const float p = __fmul_rn(a.h, b.h), e = __fmaf_rn(a.h, b.h, -p);
  const float p1 = __fmul_rn(a.h, b.m), q1 = __fmaf_rn(a.h, b.m, -p1);
  const float p2 = __fmul_rn(a.m, b.h), q2 = __fmaf_rn(a.m, b.h, -p2);
  float e1, e2;
  const float m = two_sum(e, two_sum(p1, p2, e1), e2);
  float l = __fadd_rn(__fadd_rn(q1, q2), __fadd_rn(e1, e2));
  l = __fmaf_rn(a.l, b.h, l);
  l = __fmaf_rn(a.h, b.l, l);
  return tf(p, m, __fmaf_rn(a.m, b.m, l));
}

// Two triple-floats side by side.
struct tfp {
  pk2 h, m, l;
};
__device__ __forceinline__ pk2 pk_mul(pk2 a, pk2 b) {
  pk2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ pk2 pk_fma(pk2 a, pk2 b, pk2 c) {
  pk2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ pk2 pk_neg(pk2 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ pk2 pk_two_sum(pk2 a, pk2 b, pk2 &e) {
  const pk2 s = pk_add(a, b), v = pk_rsub(a, s);
  e = pk_add(pk_rsub(pk_rsub(v, s), a), pk_rsub(v, b));
  return s;
}
// a - b = s + e exactly
__device__ __forceinline__ pk2 pk_two_diff(pk2 a, pk2 b, pk2 &e) {
  const pk2 s = pk_rsub(b, a), v = pk_rsub(a, s);
  e = pk_rsub(pk_add(b, v), pk_rsub(pk_rsub(v, s), a));
  return s;
}
__device__ __forceinline__ tfp tfp_of(const tf2 &a) { return {pk(a.h), pk(a.m), pk(a.l)}; }
__device__ __forceinline__ tf2 tf2_of(const tfp &a) {
  tf2 r;
  r.h = unpk(a.h);
  r.m = unpk(a.m);
  r.l = unpk(a.l);
  return r;
}
__device__ __forceinline__ tfp tfp_add(const tfp &a, const tfp &b) {
  pk2 e1, e2, e3;
  tfp r;
  r.h = pk_two_sum(a.h, b.h, e1);
  r.m = pk_two_sum(pk_two_sum(a.m, b.m, e2), e1, e3);
  r.l = pk_add(pk_add(a.l, b.l), pk_add(e2, e3));
  return r;
}
__device__ __forceinline__ tfp tfp_sub(const tfp &a, const tfp &b) {
  pk2 e1, e2, e3;
  tfp r;
  r.h = pk_two_diff(a.h, b.h, e1);
  r.m = pk_two_sum(pk_two_diff(a.m, b.m, e2), e1, e3);
  r.l = pk_add(pk_rsub(b.l, a.l), pk_add(e2, e3));
  return r;
}
__device__ __forceinline__ tfp tfp_mul(const tfp &a, const tfp &b) {
  const pk2 p = pk_mul(a.h, b.h), e = pk_fma(a.h, b.h, pk_neg(p));
  const pk2 p1 = pk_mul(a.h, b.m), q1 = pk_fma(a.h, b.m, pk_neg(p1));
  const pk2 p2 = pk_mul(a.m, b.h), q2 = pk_fma(a.m, b.h, pk_neg(p2));
  pk2 e1, e2;
  tfp r;
  r.h = p;
  r.m = pk_two_sum(e, pk_two_sum(p1, p2, e1), e2);
  r.l = pk_add(pk_add(q1, q2), pk_add(e1, e2));
  r.l = pk_fma(a.l, b.h, r.l);
  r.l = pk_fma(a.h, b.l, r.l);
  r.l = pk_fma(a.m, b.m, r.l);
  return r;
}

template <>
struct RealOf<tf2> {
  using type = tf;
};
template <>
__device__ __forceinline__ auto c_re<tf2>(const tf2 &v) {
  return tf(v.h.x, v.m.x, v.l.x);
}
template <>
__device__ __forceinline__ auto c_im<tf2>(const tf2 &v) {
  return tf(v.h.y, v.m.y, v.l.y);
}
template <>
__device__ __forceinline__ tf2 c_make<tf2>(tf re, tf im) {
  tf2 v;
  v.h = make_float2(re.h, im.h);
  v.m = make_float2(re.m, im.m);
  v.l = make_float2(re.l, im.l);
  return v;
}
template <>
__device__ __forceinline__ tf2 c_add<tf2>(const tf2 &a, const tf2 &b) {
  return tf2_of(tfp_add(tfp_of(a), tfp_of(b)));
}
template <>
__device__ __forceinline__ tf2 c_sub<tf2>(const tf2 &a, const tf2 &b) {
  return tf2_of(tfp_sub(tfp_of(a), tfp_of(b)));
}
// both components at once: (ax, ax) (bx, by) + (ay, ay) (-by, bx)
__device__ __forceinline__ tf2 cmul(const tf2 &a, const tf2 &b) {
  const tfp x = {pk(make_float2(a.h.x, a.h.x)), pk(make_float2(a.m.x, a.m.x)),
                 pk(make_float2(a.l.x, a.l.x))};
  const tfp y = {pk(make_float2(a.h.y, a.h.y)), pk(make_float2(a.m.y, a.m.y)),
                 pk(make_float2(a.l.y, a.l.y))};
  const tfp ib = {pk(make_float2(-b.h.y, b.h.x)), pk(make_float2(-b.m.y, b.m.x)),
                  pk(make_float2(-b.l.y, b.l.x))};
  return tf2_of(tfp_add(tfp_mul(x, tfp_of(b)), tfp_mul(y, ib)));
}

}  // namespace srm3

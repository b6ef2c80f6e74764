// df.cuh - double-float arithmetic (an unevaluated sum h + l of two FP32
// numbers, about 46 bits) for the transforms of the FP32 plans' pair sum.
//
// An FFT's rounding is bounded relative to the largest values it holds, not
// to each output; in FP32 that is worse than the directly summed pairs, in
// double-float it is far below FP32 rounding at every output.  GB300 issues
// 128 FP32 operations per SM and clock and 2 FP64 ones, so a double-float
// operation (8 FP32 ones for a sum, 16 for a component of a complex product)
// costs a fourth to an eighth of the native FP64 one.
//
// Sums are Knuth's two-sum (The Art of Computer Programming, vol. 2, 4.2.2)
// with the low parts added to its error; products are Dekker's with the
// fused multiply-add giving the exact error (Numer. Math. 18, 1971).  h and l
// are not renormalised: after cancellation l may exceed an ulp of h, which
// leaves the value h + l and the error bound (relative to the operands, what
// a transform needs) as they are.
#pragma once

#include <cuda_runtime.h>

namespace srm3 {

struct df {
  float h, l;
  df() = default;
  __host__ __device__ constexpr df(double v) : h((float)v), l((float)(v - (double)(float)v)) {}
  __host__ __device__ constexpr df(float h_, float l_) : h(h_), l(l_) {}
};

// A complex double-float: the high parts of its two components side by side,
// then the low parts, so that a sum of two of them is eight packed operations
// on pairs (f32x2: two FP32 operations per lane in one issue slot).
struct __align__(16) df2 {
  float2 h, l;
};

// a + b = s + e exactly
__device__ __forceinline__ float two_sum(float a, float b, float &e) {
  const float s = __fadd_rn(a, b), v = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v));
  return s;
}

__device__ __forceinline__ df operator+(df a, df b) {
  float e;
  const float s = two_sum(a.h, b.h, e);
  return df(s, __fadd_rn(__fadd_rn(a.l, b.l), e));
}
__device__ __forceinline__ df operator-(df a) { return df(-a.h, -a.l); }
__device__ __forceinline__ df operator-(df a, df b) { return a + (-b); }
__device__ __forceinline__ df operator*(df a, df b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  return df(p, e);
}
__device__ __forceinline__ df &operator+=(df &a, df b) { return a = a + b; }
__device__ __forceinline__ df &operator*=(df &a, df b) { return a = a * b; }

// a b + c d, the two products' errors and the low cross terms gathered in
// the low part
__device__ __forceinline__ df dot2(df a, df b, df c, df d) {
  const float p = __fmul_rn(a.h, b.h), q = __fmul_rn(c.h, d.h);
  float ep = __fmaf_rn(a.h, b.h, -p), eq = __fmaf_rn(c.h, d.h, -q);
  ep = __fmaf_rn(a.h, b.l, ep);
  eq = __fmaf_rn(c.h, d.l, eq);
  ep = __fmaf_rn(a.l, b.h, ep);
  eq = __fmaf_rn(c.l, d.h, eq);
  float e;
  const float s = two_sum(p, q, e);
  return df(s, __fadd_rn(e, __fadd_rn(ep, eq)));
}

// Packed FP32 pairs.
typedef unsigned long long pk2;
__device__ __forceinline__ pk2 pk(float2 v) {
  pk2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(v.x), "f"(v.y));
  return r;
}
__device__ __forceinline__ float2 unpk(pk2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ pk2 pk_add(pk2 a, pk2 b) {
  pk2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// b - a, as a * (-1) + b: one rounding either way
__device__ __forceinline__ pk2 pk_rsub(pk2 a, pk2 b) {
  pk2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(0xbf800000bf800000ull), "l"(b));
  return r;
}

// The complex operations of the transforms, by type.
template <typename T2>
struct RealOf;
template <>
struct RealOf<float2> {
  using type = float;
};
template <>
struct RealOf<double2> {
  using type = double;
};
template <>
struct RealOf<df2> {
  using type = df;
};
template <typename T2>
__device__ __forceinline__ auto c_re(const T2 &v) {
  return v.x;
}
template <typename T2>
__device__ __forceinline__ auto c_im(const T2 &v) {
  return v.y;
}
template <>
__device__ __forceinline__ auto c_re<df2>(const df2 &v) {
  return df(v.h.x, v.l.x);
}
template <>
__device__ __forceinline__ auto c_im<df2>(const df2 &v) {
  return df(v.h.y, v.l.y);
}
template <typename T2>
__device__ __forceinline__ T2 c_make(typename RealOf<T2>::type re, typename RealOf<T2>::type im) {
  T2 v;
  v.x = re;
  v.y = im;
  return v;
}
template <>
__device__ __forceinline__ df2 c_make<df2>(df re, df im) {
  df2 v;
  v.h = make_float2(re.h, im.h);
  v.l = make_float2(re.l, im.l);
  return v;
}
template <typename T2>
__device__ __forceinline__ T2 c_zero() {
  using F = typename RealOf<T2>::type;
  return c_make<T2>(F(0), F(0));
}
template <typename T2>
__device__ __forceinline__ T2 c_conj(const T2 &v) {
  return c_make<T2>(c_re(v), -c_im(v));
}
template <typename T2>
__device__ __forceinline__ T2 c_add(const T2 &a, const T2 &b) {
  return c_make<T2>(c_re(a) + c_re(b), c_im(a) + c_im(b));
}
template <typename T2>
__device__ __forceinline__ T2 c_sub(const T2 &a, const T2 &b) {
  return c_make<T2>(c_re(a) - c_re(b), c_im(a) - c_im(b));
}
template <>
__device__ __forceinline__ df2 c_add<df2>(const df2 &a, const df2 &b) {
  const pk2 ah = pk(a.h), bh = pk(b.h);
  const pk2 s = pk_add(ah, bh), v = pk_rsub(ah, s);
  const pk2 e = pk_add(pk_rsub(pk_rsub(v, s), ah), pk_rsub(v, bh));
  df2 r;
  r.h = unpk(s);
  r.l = unpk(pk_add(pk_add(pk(a.l), pk(b.l)), e));
  return r;
}
template <>
__device__ __forceinline__ df2 c_sub<df2>(const df2 &a, const df2 &b) {
  const pk2 ah = pk(a.h), bh = pk(b.h);
  const pk2 s = pk_rsub(bh, ah), v = pk_rsub(ah, s);
  const pk2 e = pk_rsub(pk_add(bh, v), pk_rsub(pk_rsub(v, s), ah));
  df2 r;
  r.h = unpk(s);
  r.l = unpk(pk_add(pk_rsub(pk(b.l), pk(a.l)), e));
  return r;
}

__device__ __forceinline__ df2 cmul(df2 a, df2 b) {
  const df ax = c_re(a), ay = c_im(a), bx = c_re(b), by = c_im(b);
  return c_make<df2>(dot2(ax, bx, -ay, by), dot2(ax, by, ay, bx));
}

}  // namespace srm3

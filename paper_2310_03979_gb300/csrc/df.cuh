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

struct __align__(16) df2 {
  df x, y;
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

__device__ __forceinline__ df2 cmul(df2 a, df2 b) {
  df2 r;
  r.x = dot2(a.x, b.x, -a.y, b.y);
  r.y = dot2(a.x, b.y, a.y, b.x);
  return r;
}

}  // namespace srm3

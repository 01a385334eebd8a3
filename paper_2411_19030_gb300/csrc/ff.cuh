// ff.cuh -- float-float arithmetic: a value is the unevaluated sum h + l of two floats, 48 bits.
//
// GB300 executes one FP64 instruction of a warp in 64 cycles per SM sub-partition (measured, 2 FP64
// FMAs per clock and SM) and one FP32 instruction per cycle.  The CG of the FP64 kinds therefore
// keeps its vectors and scalars as float pairs: a fused multiply-add of pairs takes 15 FP32
// instructions, a product of a pair weight with a float accumulated into a pair 11.  The FP64
// residual loop around the CG decides the accuracy of a solve; the CG only has to reduce its start
// residual, and 48 bits reduce it by up to 1e-14 in one go.
//
// The algorithms are Knuth's two-sum, Dekker's fast two-sum and the FMA two-product; every
// operation uses an _rn intrinsic, which the compiler neither contracts nor reorders.
#pragma once
#include <cuda_runtime.h>

namespace ptg {

struct ff {
  float h, l;
};

__device__ __forceinline__ ff make_ff(float h, float l = 0.f) {
  ff r;
  r.h = h;
  r.l = l;
  return r;
}
// a + b = s + e exactly
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float t = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
}
// the same for |a| >= |b|
__device__ __forceinline__ ff fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return make_ff(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ ff operator+(const ff& x, const ff& y) {
  float s, e;
  two_sum(x.h, y.h, s, e);
  return fast_two_sum(s, __fadd_rn(e, __fadd_rn(x.l, y.l)));
}
// x y as an unnormalised pair
__device__ __forceinline__ void ff_prod(const ff& x, const ff& y, float& p, float& e) {
  p = __fmul_rn(x.h, y.h);
  e = __fmaf_rn(x.h, y.h, -p);
  e = __fmaf_rn(x.h, y.l, e);
  e = __fmaf_rn(x.l, y.h, e);
}
__device__ __forceinline__ void ff_prod(const ff& x, float y, float& p, float& e) {
  p = __fmul_rn(x.h, y);
  e = __fmaf_rn(x.h, y, -p);
  e = __fmaf_rn(x.l, y, e);
}
// acc + x y, the low part of acc left unnormalised (sums of products)
template <class Y>
__device__ __forceinline__ ff ff_acc(const ff& acc, const ff& x, const Y& y) {
  float p, e, s, t;
  ff_prod(x, y, p, e);
  two_sum(acc.h, p, s, t);
  return make_ff(s, __fadd_rn(acc.l, __fadd_rn(t, e)));
}
__device__ __forceinline__ ff ff_div(const ff& a, const ff& b) {
  const float q = __fdiv_rn(a.h, b.h);
  float p, e;
  ff_prod(b, q, p, e);
  const float r = __fadd_rn(__fsub_rn(__fsub_rn(a.h, p), e), a.l);
  return fast_two_sum(q, __fdiv_rn(r, b.h));
}

// The CG's vector and scalar operations in float and in float pairs.
__device__ __forceinline__ float f32(float x) { return x; }
__device__ __forceinline__ float f32(const ff& x) { return x.h; }
// y + a x
__device__ __forceinline__ float vfma(float a, float x, float y) { return fmaf(a, x, y); }
__device__ __forceinline__ ff vfma(const ff& a, const ff& x, const ff& y) {
  float p, e, s, t;
  ff_prod(a, x, p, e);
  two_sum(y.h, p, s, t);
  return fast_two_sum(s, __fadd_rn(__fadd_rn(t, y.l), e));
}
__device__ __forceinline__ ff vfma(const ff& a, const ff& x, float y) { return vfma(a, x, make_ff(y)); }
// acc + x y
__device__ __forceinline__ float vdot(float acc, float x, float y) { return fmaf(x, y, acc); }
__device__ __forceinline__ ff vdot(const ff& acc, const ff& x, const ff& y) { return ff_acc(acc, x, y); }
__device__ __forceinline__ ff vdot(const ff& acc, const ff& x, float y) { return ff_acc(acc, x, y); }
__device__ __forceinline__ float vmul(float a, float b) { return a * b; }
__device__ __forceinline__ ff vmul(const ff& a, const ff& b) {
  float p, e;
  ff_prod(a, b, p, e);
  return fast_two_sum(p, e);
}
__device__ __forceinline__ float vdiv(float a, float b) { return a / b; }
__device__ __forceinline__ ff vdiv(const ff& a, const ff& b) { return ff_div(a, b); }
// a float as one of the CG's scalars
template <class V> __device__ __forceinline__ V vfloat(float a);
template <> __device__ __forceinline__ float vfloat<float>(float a) { return a; }
template <> __device__ __forceinline__ ff vfloat<ff>(float a) { return make_ff(a); }
__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ ff vneg(const ff& a) { return make_ff(-a.h, -a.l); }

// 2^k as a double (|k| <= 1022)
__device__ __forceinline__ double exp2_int(int k) { return __hiloint2double((k + 1023) << 20, 0); }
// v 2^k as a float pair, by integer operations (no FP64 instruction).  Meant for |v 2^k| of order
// one: below 2^-126 the result is 0, and below 2^-74 it has the first 24 bits only.
__device__ __forceinline__ ff split_scaled(double v, int k) {
  const int hi = __double2hiint(v);
  const unsigned lo = (unsigned)__double2loint(v);
  const int e = (hi >> 20) & 0x7ff;
  const int ef = e + k - 896;                       // float exponent field
  if (e == 0x7ff || ef > 254) return make_ff(__int_as_float(0x7fffffff), 0.f);
  if (e == 0 || ef <= 0) return make_ff(0.f, 0.f);
  const unsigned sign = (unsigned)hi & 0x80000000u;
  ff r;
  r.h = __uint_as_float(sign | ((unsigned)ef << 23) | (((unsigned)hi & 0xfffffu) << 3) | (lo >> 29));
  r.l = ef > 52 ? __uint2float_rn(lo & 0x1fffffffu) * __uint_as_float(sign | ((unsigned)(ef - 52) << 23)) : 0.f;
  return r;
}
// a float as a double by integer operations; 0 below the normal range
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f), m = u & 0x7fffffffu;
  if (m < 0x00800000u) return 0.0;
  const unsigned hi = m >= 0x7f800000u ? (m >> 3) | 0x7ff00000u : (m >> 3) + (896u << 20);
  return __hiloint2double((int)((u & 0x80000000u) | hi), (int)(u << 29));
}

}  // namespace ptg

// pairs.cuh -- arithmetic on unevaluated sums of two floats (Dekker 1971; Knuth; Shewchuk 1997),
// on one value (V = float) or on two at once (V = float2, the packed FP32 instructions).
//
// This GPU runs FP64 at 1/64 of its FP32 rate.  Quantities that reach an FP64 value only through a
// small factor (dt R of a Runge-Kutta stage: the time step keeps it far below the state) are formed
// as pairs of floats: h carries 24 bits, l the next 24.  Every operation uses round-to-nearest
// intrinsics, which the compiler neither contracts nor reorders.  Results of add and mul are not
// normalised: l may reach a few units in the last place of h (more after cancellation), and their
// errors are a few 2^-48 of the operands' magnitudes; norm brings l back below half a unit.
#pragma once

#include <cuda_runtime.h>

#include "device_common.cuh"

namespace cfs {

__device__ __forceinline__ float v_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float v_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float v_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float v_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float v_neg(float a) { return -a; }
__device__ __forceinline__ float2 v_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 v_sub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 v_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 v_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 v_neg(float2 a) { return make_float2(-a.x, -a.y); }
template <class V>
__device__ __forceinline__ V v_bc(float a);
template <>
__device__ __forceinline__ float v_bc<float>(float a) { return a; }
template <>
__device__ __forceinline__ float2 v_bc<float2>(float a) { return make_float2(a, a); }

template <class V>
struct Pr {
  V h, l;
};
using P1 = Pr<float>;
using P2 = Pr<float2>;

// s + e = a + b exactly (|a| >= |b| or a = 0; otherwise e is off by a rounding of itself)
template <class V>
__device__ __forceinline__ Pr<V> p_fast2sum(V a, V b) {
  const V s = v_add(a, b);
  return {s, v_sub(b, v_sub(s, a))};
}
// s + e = a + b, a - b exactly
template <class V>
__device__ __forceinline__ Pr<V> p_2sum(V a, V b) {
  const V s = v_add(a, b), t = v_sub(s, a);
  return {s, v_add(v_sub(a, v_sub(s, t)), v_sub(b, t))};
}
template <class V>
__device__ __forceinline__ Pr<V> p_2diff(V a, V b) {
  const V s = v_sub(a, b), t = v_sub(s, a);
  return {s, v_sub(v_sub(a, v_sub(s, t)), v_add(b, t))};
}
template <class V>
__device__ __forceinline__ Pr<V> p_norm(Pr<V> a) { return p_fast2sum(a.h, a.l); }
template <class V>
__device__ __forceinline__ Pr<V> p_neg(Pr<V> a) { return {v_neg(a.h), v_neg(a.l)}; }
template <class V>
__device__ __forceinline__ Pr<V> p_add(Pr<V> a, Pr<V> b) {
  const Pr<V> s = p_2sum(a.h, b.h);
  return {s.h, v_add(s.l, v_add(a.l, b.l))};
}
template <class V>
__device__ __forceinline__ Pr<V> p_sub(Pr<V> a, Pr<V> b) {
  const Pr<V> s = p_2diff(a.h, b.h);
  return {s.h, v_add(s.l, v_sub(a.l, b.l))};
}
template <class V>
__device__ __forceinline__ Pr<V> p_mul(Pr<V> a, Pr<V> b) {
  const V p = v_mul(a.h, b.h);
  V e = v_fma(a.h, b.h, v_neg(p));
  e = v_fma(a.h, b.l, e);
  return {p, v_fma(a.l, b.h, e)};
}
// a * b + c
template <class V>
__device__ __forceinline__ Pr<V> p_fma(Pr<V> a, Pr<V> b, Pr<V> c) {
  const V p = v_mul(a.h, b.h);
  V e = v_fma(a.h, b.h, v_neg(p));
  e = v_fma(a.h, b.l, e);
  e = v_fma(a.l, b.h, e);
  const Pr<V> s = p_2sum(p, c.h);
  return {s.h, v_add(s.l, v_add(e, c.l))};
}
// times a power of two
template <class V>
__device__ __forceinline__ Pr<V> p_scale(Pr<V> a, float f) {
  return {v_mul(a.h, v_bc<V>(f)), v_mul(a.l, v_bc<V>(f))};
}

__device__ __forceinline__ P2 p_bc(P1 a) { return {make_float2(a.h, a.h), make_float2(a.l, a.l)}; }
__device__ __forceinline__ P2 p_pair(P1 a, P1 b) { return {make_float2(a.h, b.h), make_float2(a.l, b.l)}; }
__device__ __forceinline__ P1 p_x(P2 a) { return {a.h.x, a.l.x}; }
__device__ __forceinline__ P1 p_y(P2 a) { return {a.h.y, a.l.y}; }
__device__ __forceinline__ P1 p_of(float2 a) { return {a.x, a.y}; }
__device__ __forceinline__ float2 p_store(P1 a) { return make_float2(a.h, a.l); }
// memory form of two pairs: (h of both, l of both)
__device__ __forceinline__ P2 p_of(float4 a) { return {make_float2(a.x, a.y), make_float2(a.z, a.w)}; }
__device__ __forceinline__ float4 p_store(P2 a) { return make_float4(a.h.x, a.h.y, a.l.x, a.l.y); }

// 1 / a for a normalised pair: the FP32 reciprocal refined by r (1 + e + e^2), e = 1 - a r
__device__ __forceinline__ P1 p_recip(P1 a) {
  const float r = __frcp_rn(a.h);
  float e = __fmaf_rn(-a.h, r, 1.f);
  e = __fmaf_rn(-a.l, r, e);
  return p_fast2sum(r, __fmul_rn(r, __fmaf_rn(e, e, e)));
}

// FP64 -> pair on the integer pipe: x is the exact sum of three floats, its FP32 truncation t and
// the remaining 29 mantissa bits as 23 + 6 (split_fast's construction); h = t + q1 rounded, l the
// rest, rounded once (2^-49 |x|).  |x| < 2^-126 gives zero, |x| >= 2^128, infinities and NaN give
// NaN; below 2^-97 the remaining bits are dropped.
__device__ __forceinline__ P1 p_split(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned ahi = hi & 0x7fffffffu, e = ahi >> 20, sg = hi & 0x80000000u;
  unsigned t = (__funnelshift_l(lo, hi, 3) & 0x7fffffffu) ^ 0x40000000u;
  t = (ahi < 0x38100000u) ? 0u : t;
  t = (ahi >= 0x47f00000u) ? 0x7fc00000u : t;
  const unsigned m = lo & 0x1fffffffu;
  const unsigned eb1 = (e - 919u) << 23, eb2 = (e - 925u) << 23;  // 2^(E-1046), 2^(E-1052)
  const float q1 = __uint_as_float(eb1 | (m >> 6)) - __uint_as_float(eb1);
  const float q2 = __uint_as_float(eb2 | (m & 63u)) - __uint_as_float(eb2);
  const bool ok = e >= 926u;
  const P1 s = p_fast2sum(__uint_as_float(t), ok ? q1 : 0.f);
  const float l = __fadd_rn(s.l, ok ? q2 : 0.f);
  return {__uint_as_float(__float_as_uint(s.h) ^ sg), __uint_as_float(__float_as_uint(l) ^ sg)};
}
// pair -> FP64: one FP64 addition
__device__ __forceinline__ double p_double(P1 a) { return f2d_fast(a.h) + f2d_fast(a.l); }

}  // namespace cfs

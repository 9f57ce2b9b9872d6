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

#include <cmath>

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
// The same two values as plain FP32 instructions: twice as many, but the operands need not be brought
// into register pairs
struct F2 {
  float x, y;
};
__device__ __forceinline__ F2 v_add(F2 a, F2 b) { return {__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y)}; }
__device__ __forceinline__ F2 v_sub(F2 a, F2 b) { return {__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y)}; }
__device__ __forceinline__ F2 v_mul(F2 a, F2 b) { return {__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y)}; }
__device__ __forceinline__ F2 v_fma(F2 a, F2 b, F2 c) { return {__fmaf_rn(a.x, b.x, c.x), __fmaf_rn(a.y, b.y, c.y)}; }
__device__ __forceinline__ F2 v_neg(F2 a) { return {-a.x, -a.y}; }
template <class V>
__device__ __forceinline__ V v_bc(float a);
template <>
__device__ __forceinline__ F2 v_bc<F2>(float a) { return {a, a}; }
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

// (W: float2, or F2 for two values by plain instructions)
template <class W = float2>
__device__ __forceinline__ Pr<W> p_bc(P1 a) { return {W{a.h, a.h}, W{a.l, a.l}}; }
template <class W = float2>
__device__ __forceinline__ Pr<W> p_pair(P1 a, P1 b) { return {W{a.h, b.h}, W{a.l, b.l}}; }
template <class W>
__device__ __forceinline__ P1 p_x(Pr<W> a) { return {a.h.x, a.l.x}; }
template <class W>
__device__ __forceinline__ P1 p_y(Pr<W> a) { return {a.h.y, a.l.y}; }
__device__ __forceinline__ P1 p_of(float2 a) { return {a.x, a.y}; }
__device__ __forceinline__ float2 p_store(P1 a) { return make_float2(a.h, a.l); }
// memory form of two pairs: (h of both, l of both)
template <class W = float2>
__device__ __forceinline__ Pr<W> p_of(float4 a) { return {W{a.x, a.y}, W{a.z, a.w}}; }
template <class W>
__device__ __forceinline__ float4 p_store(Pr<W> a) { return make_float4(a.h.x, a.h.y, a.l.x, a.l.y); }

// 1 / a for a normalised pair: the FP32 reciprocal refined by r (1 + e + e^2), e = 1 - a r
__device__ __forceinline__ P1 p_recip(P1 a) {
  const float r = __frcp_rn(a.h);
  float e = __fmaf_rn(-a.h, r, 1.f);
  e = __fmaf_rn(-a.l, r, e);
  return p_fast2sum(r, __fmul_rn(r, __fmaf_rn(e, e, e)));
}

// FP64 -> the exact sum of three floats on the integer pipe: the FP32 truncation t and the remaining 29
// mantissa bits as 23 + 6, q1 and q2 (split_fast's construction).  |x| < 2^-126 gives zero, |x| >=
// 2^128, infinities and NaN give NaN; below 2^-97 the remaining bits are dropped.
struct Triple {
  float t, q1, q2;
};
__device__ __forceinline__ Triple p_split3(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned ahi = hi & 0x7fffffffu, e = ahi >> 20, sg = hi & 0x80000000u;
  unsigned t = (__funnelshift_l(lo, hi, 3) & 0x7fffffffu) ^ 0x40000000u;
  t = (ahi < 0x38100000u) ? 0u : t;
  t = (ahi >= 0x47f00000u) ? 0x7fc00000u : t;
  const unsigned m = lo & 0x1fffffffu;
  const unsigned eb1 = ((e - 919u) << 23) | sg, eb2 = ((e - 925u) << 23) | sg;  // +-2^(E-1046), 2^(E-1052)
  const float q1 = __uint_as_float(eb1 | (m >> 6)) - __uint_as_float(eb1);
  const float q2 = __uint_as_float(eb2 | (m & 63u)) - __uint_as_float(eb2);
  const bool ok = e >= 926u;
  return {__uint_as_float(t | sg), ok ? q1 : 0.f, ok ? q2 : 0.f};
}
// FP64 -> pair: h = t + q1 rounded, l the rest, rounded once (2^-49 |x|)
__device__ __forceinline__ P1 p_pair_of(Triple x) {
  const P1 s = p_fast2sum(x.t, x.q1);
  return {s.h, __fadd_rn(s.l, x.q2)};
}
__device__ __forceinline__ P1 p_split(double x) { return p_pair_of(p_split3(x)); }
// x - c for a float c, the difference taken before anything is rounded: 2^-48 of the difference, not of x
__device__ __forceinline__ P1 p_less(Triple x, float c) {
  const P1 s = p_2diff(x.t, c);
  const P1 r = p_2sum(s.h, x.q1);
  return p_norm(P1{r.h, __fadd_rn(r.l, __fadd_rn(s.l, x.q2))});
}
// Two FP64 values as triples, and the difference of two such as pairs: exact but for the last rounding
// (2^-48 of the difference, however small it is against the values)
struct Triple2 {
  float2 t, q1, q2;
};
__device__ __forceinline__ Triple2 p_triples(double a, double b) {
  const Triple x = p_split3(a), y = p_split3(b);
  return {make_float2(x.t, y.t), make_float2(x.q1, y.q1), make_float2(x.q2, y.q2)};
}
__device__ __forceinline__ P2 p_pair_of(Triple2 x) {
  const P2 s = p_fast2sum(x.t, x.q1);
  return {s.h, v_add(s.l, x.q2)};
}
__device__ __forceinline__ P2 p_diff(Triple2 a, Triple2 b) {
  const P2 s = p_2diff(a.t, b.t);
  const P2 r = p_2sum(s.h, v_sub(a.q1, b.q1));
  return p_norm(P2{r.h, v_add(r.l, v_add(s.l, v_sub(a.q2, b.q2)))});
}
// pair -> FP64: one FP64 addition
__device__ __forceinline__ double p_double(P1 a) { return f2d_fast(a.h) + f2d_fast(a.l); }
// The same of a normalised pair on the integer pipe, in a third of the issue slots of the addition: l as a
// multiple L of the last place of h as FP64 (below a power of two, of half of it), added to the bit
// pattern.  l is left out where |h| < 2^-66.
__device__ __forceinline__ double p_double_int(P1 a) {
  const unsigned hb = __float_as_uint(a.h), e = (hb >> 23) & 255u;
  float l = __fmul_rn(a.l, __uint_as_float((306u - e) << 23));  // 2^(52 - E)
  l = __uint_as_float(__float_as_uint(l) ^ (hb & 0x80000000u));
  if ((hb & 0x7fffffu) == 0 && l < 0.f) l = __fadd_rn(l, l);
  const int L = e > 60u && e < 255u ? __float2int_rn(l) : 0;
  return __longlong_as_double(__double_as_longlong(f2d_fast(a.h)) + L);
}

// x^a = exp(a ln x) for positive x, table-driven after Tang (ACM TOMS 1989, 1990) as the FP64 power
// of kernels.cu, on pairs.  ln x: x = m 2^e with m in [1, 2); the top six mantissa bits pick a
// float rc_j near 1 / c_j, c_j = 1 + (j + 1/2)/64; u = m rc_j - 1 (|u| < 1/128, the product split
// exactly), ln m = -ln rc_j + log1p(u): u, u^2/2 and u^3/3 as pairs, u^4 to u^7 in FP32.  exp y: y =
// (64 k' + j') ln2/64 + r, |r| <= ln2/128, exp r with r and r^2/2 as pairs and r^3 to r^5 in FP32,
// times the tabulated 2^(j'/64), times 2^k'.  Relative error below 2^-44 (1 + |a ln x|).  About 120
// FP32 operations, where the FP64 power's 20 take the time of 1,280.  Other x, or |a ln x| >= 60, go to
// the library's pow.  tab: [5][64]: rc_j, -ln rc_j (h, l), 2^(j/64) (h, l).
#define POW_PAIR_TAB (5 * 64)
__device__ __forceinline__ P1 p_pow(P1 x, P1 a, const float* __restrict__ tab) {
  const unsigned b = __float_as_uint(x.h);
  if (b - 0x08000000u < 0x6f000000u) {  // 2^-111 <= x.h < 2^111
    const int e = (int)(b >> 23) - 127;
    const int j = (int)(b >> 17) & 63;
    const float m = __uint_as_float((b & 0x007fffffu) | 0x3f800000u);
    const float ml = __fmul_rn(x.l, __uint_as_float((unsigned)(127 - e) << 23));
    const float rc = __ldg(tab + j);
    const float p = __fmul_rn(m, rc);
    const P1 u = p_fast2sum(__fsub_rn(p, 1.f), __fmaf_rn(ml, rc, __fmaf_rn(m, rc, -p)));
    const P1 u2 = p_norm(p_mul(u, u));
    const P1 u3 = p_mul(p_norm(p_mul(u2, u)), P1{0.33333334f, -9.934108e-09f});
    float t = 1.f / 7.f;
    t = __fmaf_rn(t, u.h, -1.f / 6.f);
    t = __fmaf_rn(t, u.h, 1.f / 5.f);
    t = __fmaf_rn(t, u.h, -1.f / 4.f);
    t = __fmul_rn(t, __fmul_rn(u2.h, u2.h));
    // ln 2 = 0.693145751953125 (16 bits, e times it is exact) + the rest as a pair
    const float ef = (float)e;
    P1 L = p_add(P1{__fmul_rn(ef, 0.693145751953125f), 0.f}, P1{__ldg(tab + 64 + j), __ldg(tab + 128 + j)});
    L = p_add(L, p_mul(P1{ef, 0.f}, P1{1.4286068e-06f, 5.497923e-14f}));
    P1 s = p_add(p_add(u, p_scale(u2, -0.5f)), u3);
    s.l = __fadd_rn(s.l, t);
    const P1 y = p_norm(p_mul(p_norm(p_add(L, s)), a));
    if (fabsf(y.h) < 60.f) {
      const float kf = rintf(__fmul_rn(y.h, 92.332482f));  // 64 / ln 2
      // ln2/64 = 0.01082611083984375 (11 bits, k times it is exact) + the rest as a pair
      P1 r = p_add(y, P1{__fmul_rn(kf, -0.01082611083984375f), 0.f});
      r = p_norm(p_add(r, p_mul(P1{kf, 0.f}, P1{-4.3138566e-06f, 2.0164563e-13f})));
      const P1 r2 = p_mul(r, r);
      float q = 1.f / 120.f;
      q = __fmaf_rn(q, r.h, 1.f / 24.f);
      q = __fmaf_rn(q, r.h, 1.f / 6.f);
      q = __fmul_rn(q, __fmul_rn(r2.h, r.h));
      P1 w = p_add(r, p_scale(r2, 0.5f));
      w.l = __fadd_rn(w.l, q);
      w = p_norm(p_add(P1{1.f, 0.f}, w));
      const int k = (int)kf;
      w = p_norm(p_mul(w, P1{__ldg(tab + 192 + (k & 63)), __ldg(tab + 256 + (k & 63))}));
      return p_scale(w, __uint_as_float((unsigned)((k >> 6) + 127) << 23));
    }
  }
  return p_split(pow((double)x.h + (double)x.l, (double)a.h + (double)a.l));
}

// The tables of p_pow (host).
inline void pow_pair_table(float* t) {
  auto put = [&](int at, int j, long double x) {
    t[at + j] = (float)x;
    t[at + 64 + j] = (float)(x - (long double)t[at + j]);
  };
  for (int j = 0; j < 64; ++j) {
    t[j] = (float)(128.0 / (129.0 + 2.0 * j));
    put(64, j, -logl((long double)t[j]));
    put(192, j, exp2l((long double)j / 64.0L));
  }
}

}  // namespace cfs

// level_sums.cuh -- weighted sums over the delayed time levels of a point in FP32 arithmetic, compensated
// to about the accuracy of FP64 sums (the FP32 form's AT halo values and filter halos).
#pragma once

#include <cuda_runtime.h>

#include "cfs_internal.h"
#include "device_common.cuh"
#include "pairs.cuh"

namespace cfs {

// The delayed levels of one point as the AT sums take them: U_0 = h0 + l0 (to 48 bits) and the
// differences U_l - U_0 = ah + al (to 2^-48 of the levels); rho and rho u, rho v and rho w as packed
// pairs, rho E alone.  U_l = h + q, h its FP32 truncation.  h - h0 is exact when the levels are within a
// factor of two; where they are not (a momentum that changes sign) its rounding goes to al, since
// the weights would multiply it by up to 1,500.
struct LevelDiffs {
  float2 h0[2], l0[2], ah[CFS_MAX_LEVELS][2], al[CFS_MAX_LEVELS][2];
  float h4, l4, ah4[CFS_MAX_LEVELS], al4[CFS_MAX_LEVELS];
};
__device__ __forceinline__ void level_diffs(const double (*r)[5], int C, LevelDiffs& d) {
  float h0[5], l0[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    h0[v] = d2f_fast(r[0][v]);
    l0[v] = dev_fast(r[0][v], h0[v], 0.f);
  }
  d.h0[0] = make_float2(h0[0], h0[1]);
  d.h0[1] = make_float2(h0[2], h0[3]);
  d.l0[0] = make_float2(l0[0], l0[1]);
  d.l0[1] = make_float2(l0[2], l0[3]);
  d.h4 = h0[4];
  d.l4 = l0[4];
#pragma unroll
  for (int l = 1; l < CFS_MAX_LEVELS; ++l)
    if (l < C) {
      float h[5], q[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) split_fast(r[l][v], h[v], q[v]);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const P2 s = p_2diff(make_float2(h[2 * k], h[2 * k + 1]), d.h0[k]);
        d.ah[l][k] = s.h;
        d.al[l][k] = v_add(s.l, v_sub(make_float2(q[2 * k], q[2 * k + 1]), d.l0[k]));
      }
      const P1 s = p_2diff(h[4], d.h4);
      d.ah4[l] = s.h;
      d.al4[l] = v_add(s.l, v_sub(q[4], d.l4));
    }
}

// (S - 1) U_0 + sum_{l >= 1} W_l (U_l - U_0) with the weights c[0 .. C-1] = pairs of S - 1, W_1, ...:
// products of the high parts split exactly with an FMA and summed with TwoSum.
template <class V, class A, class L>
__device__ __forceinline__ V at_sum(V h0, A ah, L al, const float2* c, int C) {
  V sh = v_bc<V>(0.f), st = v_mul(v_bc<V>(c[0].x), h0);  // running sum and its error terms
#pragma unroll
  for (int l = 1; l < CFS_MAX_LEVELS; ++l)
    if (l < C) {
      const V wx = v_bc<V>(c[l].x), a = ah(l);
      const V p = v_mul(wx, a);
      const V pe = v_fma(wx, a, v_neg(p));  // exact: p + pe = c.x * ah
      const V s2 = v_add(sh, p);            // TwoSum(sh, p)
      const V bv = v_sub(s2, sh);
      const V se = v_add(v_sub(sh, v_sub(s2, bv)), v_sub(p, bv));
      sh = s2;
      st = v_add(st, v_add(se, pe));
      st = v_fma(wx, al(l), st);
      st = v_fma(v_bc<V>(c[l].y), a, st);
    }
  return v_add(sh, st);
}
// the five variables' sums
__device__ __forceinline__ void at_sums(const LevelDiffs& d, const float2* c, int C, float* out) {
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float2 x = at_sum(d.h0[k], [&](int l) { return d.ah[l][k]; }, [&](int l) { return d.al[l][k]; }, c, C);
    out[2 * k] = x.x;
    out[2 * k + 1] = x.y;
  }
  out[4] = at_sum(d.h4, [&](int l) { return d.ah4[l]; }, [&](int l) { return d.al4[l]; }, c, C);
}

}  // namespace cfs

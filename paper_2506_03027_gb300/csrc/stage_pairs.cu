// stage_pairs.cu -- the Runge-Kutta stage of the FP64 form for 3-D Navier-Stokes: FP64 state, FP64
// low-storage update, and the right-hand side between them on pairs of floats (pairs.cuh).
//
// In FP64 the stage is bound by the FP64 pipe: about 215 FP64 operations per point and stage at 2
// per clock and SM, while the FP32 pipe (64 times as fast) and memory idle.  dt R is a small
// correction of the state (the time step keeps it below about 1e-2 of it), so a right-hand side that
// is good to a few 2^-48 leaves the error of U + B Q where it was, at the FP64 rounding of the sum.
// Pressure and total energy are carried as deviations from the reference state (p_ref =
// 1/(gamma M^2) is 70 times the dynamic pressure at M = 0.1), taken before anything is rounded to a
// pair, so that the pressure gradient does not lose what rho E rounds at: the momentum after one step at
// a CFL number of 0.5 is off by 1.5e-16 rms at M = 0.1, 1.4e-15 at 0.01 (FP64 sums over the full
// pressure: 3.1e-16, 2.8e-15; rho E as a pair before its deviation: 1.5e-15, 2.1e-14).
//
// The kernels are those of kernels.cu (view, flux, update) with pairs in the scratch arrays, two
// values interleaved where the same operation acts on both, so that one 16-byte load and the
// packed FP32 instructions serve (u, v) and (w, kappa T) together:
//   W    A (u, v), B (w, kappa T), C (rho, p - p_ref): float4 {h, h, l, l}; D (rho E + p - H_ref): float2
//   Phi  per direction a: M (x, y momentum), E (z momentum, energy): float4; N (mass): FP64
// The mass flux is the momentum itself: the update differences it in FP64, from the state inside a Cartesian
// sub-domain and from N elsewhere (the strips beyond its faces; curvilinear blocks, times the metric row),
// which the view stores.  The energy flux is H_ref times it plus a remainder, -((rho E + p -
// H_ref) - H_ref (rho - 1)) u, which alone is a pair: pairs of the whole, 250 u at M = 0.1, would
// raise the energy's error of a step from the 1.8e-14 of its rounding to 3.2e-14, pairs of the mass flux
// the density's from 1.1e-16 to 1.5e-16.
// and one more, once per asynchronous step: k_at_halo forms the AT halo values of all stages from
// one read of the delayed levels (they would be read once per stage otherwise).
//
// 128^3 in 64 sub-domains, us per launch, FP64 -> pairs: view 150 -> 84 (DRAM at 52 % of its rate and
// issue at 51 %), flux 384 -> 110 (49 %, 72 %), update 290 -> 135 (60 %, 44 %); the halo values, once per
// step instead of inside the view, 223 (52 %, 55 %).
#include <cuda_runtime.h>

#include <mutex>
#include <type_traits>

#include "cfs_internal.h"
#include "device_common.cuh"
#include "launch_common.cuh"
#include "pairs.cuh"

namespace cfs {

namespace {

struct WView {
  float4 *A, *B, *C;
  float2* D;
};
__device__ __forceinline__ WView w_view(void* W, long long P) {
  float4* a = (float4*)W;
  return {a, a + P, a + 2 * P, (float2*)(a + 3 * P)};
}

__device__ __forceinline__ P1 cst(float2 c) { return {c.x, c.y}; }

// Primitives of a conserved state (rho E as its deviation from E_ref): velocities, p - p_ref, kappa T and
// rho E + p - H_ref.
struct PrimsP {
  P1 rho, mz, w, p, kT, et;
  P2 mxy, uv;
};
__device__ __forceinline__ PrimsP prims_p(const PairPhysics& ph, P1 rho, P2 mxy, P1 mz, P1 rE) {
  PrimsP r;
  const P1 ir = p_recip(rho);
  r.rho = rho;
  r.mxy = mxy;
  r.mz = mz;
  r.uv = p_norm(p_mul(mxy, p_bc(ir)));
  r.w = p_norm(p_mul(mz, ir));
  const P2 k2 = p_mul(mxy, r.uv);
  const P1 ke = p_scale(p_fma(mz, r.w, p_add(p_x(k2), p_y(k2))), 0.5f);
  r.p = p_norm(p_mul(cst(ph.gm1), p_norm(p_sub(rE, ke))));
  r.kT = p_norm(p_mul(p_norm(p_fma(cst(ph.kgM2), r.p, cst(ph.kT0))), ir));
  r.et = p_norm(p_add(rE, r.p));
  return r;
}
__device__ __forceinline__ PrimsP prims_of(const PairPhysics& ph, const double* u) {
  return prims_p(ph, p_split(u[0]), p_pair(p_split(u[1]), p_split(u[2])), p_split(u[3]), p_less(p_split3(u[4]), ph.Eref));
}
__device__ __forceinline__ void store_prims(const WView& W, long long o, const PrimsP& r) {
  W.A[o] = p_store(r.uv);
  W.B[o] = p_store(p_pair(r.w, r.kT));
  W.C[o] = p_store(p_pair(r.rho, r.p));
  W.D[o] = p_store(r.et);
}

// What the energy flux carries beside H_ref times the mass flux, per unit velocity: -((rho E + p - H_ref) -
// H_ref (rho - 1))
__device__ __forceinline__ P1 rest_enthalpy(const PairPhysics& ph, P1 et, P1 rho) {
  return p_norm(p_neg(p_fma(cst(ph.H), p_norm(p_sub(P1{1.f, 0.f}, rho)), et)));
}

// Mass fluxes rho U_a of a point from its FP64 momentum m(0 .. 2), times the metric row on a
// curvilinear block, along axis `as` or (as < 0) every axis; stored at scratch index o.
template <class F>
__device__ __forceinline__ void store_mass_flux(const Geometry& g, const SubDev& d, void* Phi, long long o, F m, int ci, int cj,
                                                int as) {
  const double* __restrict__ M = nullptr;
  if (d.mbase >= 0) M = g.metric + d.mbase + (long long)(d.ox + ci + g.G) + (long long)d.mx * (d.oy + cj + g.G);
  double* __restrict__ N = (double*)((float4*)Phi + 6 * g.Ptot) + o;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (as >= 0 && as != a) continue;
    double f = m(a);
    if (M) f = a < 2 ? fma(M[(2 * a + 1) * d.mpl], m(1), M[2 * a * d.mpl] * m(0)) : M[4 * d.mpl] * f;
    N[a * g.Ptot] = f;
  }
}

// Inviscid combined fluxes -F_a (Eq. A2) at scratch index o, along axis `as` or (as < 0) every axis;
// M: the metric terms of the point on a curvilinear block, or null.  The mass flux is stored apart.
__device__ __forceinline__ void store_euler_flux(const PairPhysics& ph, void* Phi, long long P, long long o, const PrimsP& r,
                                                 int as, const float2* M, long long pl) {
  float4* __restrict__ F4 = (float4*)Phi;
  const P1 rest = rest_enthalpy(ph, r.et, r.rho), zero = {0.f, 0.f};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (as >= 0 && as != a) continue;
    P1 U = a == 0 ? p_x(r.uv) : (a == 1 ? p_y(r.uv) : r.w);
    P1 n = p_neg(a == 0 ? p_x(r.mxy) : (a == 1 ? p_y(r.mxy) : r.mz));
    P2 pxy = {make_float2(a == 0 ? r.p.h : 0.f, a == 1 ? r.p.h : 0.f), make_float2(a == 0 ? r.p.l : 0.f, a == 1 ? r.p.l : 0.f)};
    P1 pz = a == 2 ? r.p : zero;
    if (M) {
      if (a < 2) {
        const P2 row = p_pair(p_of(M[2 * a * pl]), p_of(M[(2 * a + 1) * pl])), x = p_mul(row, r.uv);
        U = p_norm(p_add(p_x(x), p_y(x)));
        pxy = p_mul(p_bc(r.p), row);
      } else {
        const P1 zz = p_of(M[4 * pl]);
        U = p_norm(p_mul(zz, r.w));
        pz = p_mul(zz, r.p);
      }
      n = p_norm(p_neg(p_mul(r.rho, U)));
    }
    F4[(long long)(2 * a) * P + o] = p_store(p_norm(p_sub(p_mul(p_bc(n), r.uv), pxy)));
    F4[(long long)(2 * a + 1) * P + o] = p_store(p_norm(p_sub(p_mul(p_pair(n, rest), p_pair(r.w, U)), p_pair(pz, zero))));
  }
}

// Delay of a halo point: the largest of the faces it lies beyond; faces on a physical boundary of
// the block carry none for points beyond the block.
__device__ __forceinline__ int point_delay(const StepSched& sc, const SubDev& d, int sid, int ci, int cj, int ck, bool beyond) {
  int kd = 0;
  if ((ci < 0 || ci >= d.sx) && !(beyond && ((d.phys >> (ci < 0 ? 0 : 1)) & 1))) kd = max(kd, face_delay(sc, sid, ci < 0 ? 0 : 1));
  if ((cj < 0 || cj >= d.sy) && !(beyond && ((d.phys >> (cj < 0 ? 2 : 3)) & 1))) kd = max(kd, face_delay(sc, sid, cj < 0 ? 2 : 3));
  if ((ck < 0 || ck >= d.sz) && !(beyond && ((d.phys >> (ck < 0 ? 4 : 5)) & 1))) kd = max(kd, face_delay(sc, sid, ck < 0 ? 4 : 5));
  return kd;
}

struct HaloPoint {
  int sid, q, ci, cj, ck;
  long long gi;   // state offset of the wrapped point
  bool beyond;    // beyond a non-periodic block face: ent is its gather entry
  const GatherEntry* ent;
};

__device__ __forceinline__ HaloPoint halo_point(const Geometry& g, const SubDev& d, int2 e) {
  HaloPoint h;
  h.sid = e.x;
  h.q = e.y;
  const int exy = d.ex * d.ey;
  const int k = h.q / exy, r2 = h.q - k * exy, j = r2 / d.ex, i = r2 - j * d.ex;
  h.ci = i - g.G;
  h.cj = j - g.G;
  h.ck = k - g.Gz;
  auto wrap1 = [](int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); };
  const int ux = d.ox + h.ci, uy = d.oy + h.cj;
  const int gx = wrap1(ux, d.bnx), gy = wrap1(uy, d.bny), gz = wrap1(d.oz + h.ck, d.bnz);
  h.gi = d.bbase + (long long)gx + (long long)d.bnx * ((long long)gy + (long long)d.bny * gz);
  h.beyond = d.ebase >= 0 && (ux < 0 || ux >= d.bnx || uy < 0 || uy >= d.bny);
  h.ent = nullptr;
  if (h.beyond) h.ent = &g.gent[g.emap[d.ebase + (ux + g.GE) + (long long)d.gmx * ((uy + g.GE) + (long long)d.gmy * gz)]];
  return h;
}

// Whether source t of the entry is the sub-domain's own current value (a wall mirror or an outflow
// copy, for points inside the sub-domain in z; beyond a z face the source is a neighbouring PE's)
__device__ __forceinline__ bool own_source(const HaloPoint& h, const SubDev& d, int t) {
  return h.ck >= 0 && h.ck < d.sz && !(h.ent->flags[t] & 2) && h.ent->sid[t] == h.sid;
}
__device__ __forceinline__ bool any_own_source(const HaloPoint& h, const SubDev& d) {
  bool own = false;
  for (int t = 0; t < h.ent->nt; ++t) own = own || own_source(h, d, t);
  return own;
}

// The value of a gather entry with an own source at stage `stage`: own sources from the stage input, a
// neighbouring PE's by the mode (live, latest delayed level, or the AT weights), far-field constants; FP64.
__device__ __forceinline__ void gather_value(const Geometry& g, const StepSched& sc, const HaloPoint& h, const SubDev& d, int kd,
                                             const double* __restrict__ Uin, const double* __restrict__ ring, int stage,
                                             int s, double* u) {
  const GatherEntry& E = *h.ent;
  const int nR = mod_ring(sc.n, sc.R);
  const long long lvN = 5 * g.N;
  auto slot = [&](int l) { const int q = nR - kd - l; return (long long)(q < 0 ? q + sc.R : q) * lvN; };
#pragma unroll
  for (int v = 0; v < 5; ++v) u[v] = E.cst[v];
  for (int t = 0; t < E.nt; ++t) {
    const double wt = E.w[t], wf = (E.flags[t] & 1) ? -wt : wt;
    const long long o = E.off[t], bN = E.bN[t];
    double x[5];
    if (sc.mode == 0 || own_source(h, d, t)) {
#pragma unroll
      for (int v = 0; v < 5; ++v) x[v] = Uin[o + v * bN];
    } else if (sc.mode == 2) {
#pragma unroll
      for (int v = 0; v < 5; ++v) x[v] = ring[slot(0) + o + v * bN];
    } else {
#pragma unroll
      for (int v = 0; v < 5; ++v) x[v] = 0.0;
      for (int l = 0; l < sc.C; ++l) {
        const double wl = __ldg(sc.W + (kd * s + stage) * sc.C + l);
#pragma unroll
        for (int v = 0; v < 5; ++v) x[v] = fma(wl, ring[slot(l) + o + v * bN], x[v]);
      }
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) u[v] = fma((v >= 1 && v <= 3) ? wf : wt, x[v], u[v]);
  }
}

}  // namespace

// ------------------------------------------------------------------------------- k_at_halo

// Once per asynchronous step: for every entry of the halo list the conserved state of all S stages,
// U^(m) = sum_l W^(m)_l(k) U^{n-k-l} (Eq. 14-15 and the buffer updates of Eq. 8 collapsed into
// weights), as U_0 + (S_m - 1) U_0 + sum_{l>=1} W^(m)_l (U_l - U_0) with U_l = U^{n-k-l} and S_m the
// sum of the weights: the levels differ by a step's change, so the products of pairs keep the sum
// at the accuracy of the FP64 one.  With the learned halo, face points start from the network's
// stage-0 value and add the sums with W^(m) - W^(0).  Stored [stage][entry]: (rho, rho u), (rho v,
// rho w) and rho E - E_ref; or (only >= 0) of that stage alone.  Bound by its reads: C x 40 bytes per entry at the sub-domains' faces.
template <int S>
__global__ void __launch_bounds__(256, 3) k_at_halo(Geometry g, PairPhysics ph, StepSched sc, const double* __restrict__ ring,
                                                 const SubDev* __restrict__ subs, const int2* __restrict__ halo,
                                                 long long nhalo, int only, float4* __restrict__ H4,
                                                 float2* __restrict__ H2) {
  pdl_enter();
  sc = resolve(sc);
  if (sc.mode == 0) return;
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nhalo) return;
  const int2 hv = halo[e];
  const SubDev d = subs[hv.x];
  const HaloPoint h = halo_point(g, d, hv);
  const int kd = point_delay(sc, d, h.sid, h.ci, h.cj, h.ck, h.beyond);
  // (entries with an own source are formed from the live stage input by k_view_p)
  if (h.beyond && any_own_source(h, d)) return;
  const long long lvN = 5 * g.N;
  const int nR = mod_ring(sc.n, sc.R);
  auto slot = [&](int l) { const int q = nR - kd - l; return (long long)(q < 0 ? q + sc.R : q) * lvN; };
  const int C = sc.mode == 2 ? 1 : sc.C;
  long long lev[CFS_MAX_LEVELS];
#pragma unroll
  for (int l = 0; l < CFS_MAX_LEVELS; ++l) lev[l] = l < C ? slot(l) : 0;
  const bool learned = sc.LH && sc.mode == 1 && ((int)(h.ci < 0 || h.ci >= d.sx) + (int)(h.cj < 0 || h.cj >= d.sy) + (int)(h.ck < 0 || h.ck >= d.sz) == 1);
  // (AS, mode 2: the latest visible level, the same for every stage -- stage 0 alone is stored)
  const int one = sc.mode == 2 ? 0 : only;
  const float2* __restrict__ wt = (const float2*)(learned ? sc.W32d : sc.W32) + (long long)kd * S * sc.C;
  const long long lh = d.pbase + h.q;
  // two components at a time (rho and rho u, rho v and rho w, rho E alone): few registers, so that
  // several warps per scheduler keep the levels' loads in flight
#pragma unroll
  for (int grp = 0; grp < 3; ++grp) {
    const int v0 = 2 * grp, v1 = grp < 2 ? v0 + 1 : v0;
    double x[CFS_MAX_LEVELS], y[CFS_MAX_LEVELS];
    if (!h.beyond) {
#pragma unroll
      for (int l = 0; l < CFS_MAX_LEVELS; ++l)
        if (l < C) {
          x[l] = ring[lev[l] + h.gi + v0 * d.bN];
          if (grp < 2) y[l] = ring[lev[l] + h.gi + v1 * d.bN];
        }
    } else {
      // beyond a non-periodic block face: the weighted sources of the gather entry and the far-field
      // constant, level by level (FP64)
      const GatherEntry& E = *h.ent;
#pragma unroll
      for (int l = 0; l < CFS_MAX_LEVELS; ++l) {
        x[l] = E.cst[v0];
        y[l] = E.cst[v1];
      }
      for (int t = 0; t < E.nt; ++t) {
        const double w = E.w[t], wf = (E.flags[t] & 1) ? -w : w;
        const double w0 = grp == 1 ? wf : w, w1 = wf;  // (components 0, 1 | 2, 3 | 4)
        const double* src = ring + E.off[t];
        const long long sN = E.bN[t];
#pragma unroll
        for (int l = 0; l < CFS_MAX_LEVELS; ++l)
          if (l < C) {
            x[l] = fma(w0, src[lev[l] + v0 * sN], x[l]);
            if (grp < 2) y[l] = fma(w1, src[lev[l] + v1 * sN], y[l]);
          }
      }
    }
    // what the sums are added to: U_0, or the network's stage-0 value
    const Triple2 t0 = p_triples(x[0], grp < 2 ? y[0] : 0.0);
    const P2 u0 = p_pair_of(t0);
    P1 bx = p_x(u0), by = p_y(u0);
    if (learned) {
      bx = p_split(sc.LH[(long long)v0 * g.Ptot + lh]);
      if (grp < 2) by = p_split(sc.LH[(long long)v1 * g.Ptot + lh]);
    }
    if (grp == 2) bx = p_less(p_split3(learned ? sc.LH[4LL * g.Ptot + lh] : x[0]), ph.Eref);
    P2 acc[S];
#pragma unroll
    for (int m = 0; m < S; ++m) {
      // (with the network, stage 0 is its value: the weights W^(0) - W^(0) are zero)
      const float2 c = sc.mode == 2 ? make_float2(0.f, 0.f) : __ldg(wt + m * C);
      acc[m] = p_fma(p_bc(P1{c.x, c.y}), u0, p_pair(bx, by));
    }
#pragma unroll
    for (int l = 1; l < CFS_MAX_LEVELS; ++l)
      if (l < C) {
        // (the weights of long delays sum to hundreds in magnitude: the differences are taken before
        // anything is rounded to a pair)
        const P2 dl = p_diff(p_triples(x[l], grp < 2 ? y[l] : 0.0), t0);
#pragma unroll
        for (int m = 0; m < S; ++m) {
          const float2 w = __ldg(wt + m * C + l);
          acc[m] = p_fma(p_bc(P1{w.x, w.y}), dl, acc[m]);
        }
      }
#pragma unroll
    for (int m = 0; m < S; ++m) {
      if (one >= 0 && m != one) continue;
      const P2 a = p_norm(acc[m]);
      const int row = one >= 0 ? 0 : m;
      if (grp < 2) H4[(long long)(2 * row + grp) * nhalo + e] = p_store(a);
      else H2[(long long)row * nhalo + e] = p_store(p_x(a));
    }
  }
}

// ------------------------------------------------------------------------------- k_view_p

// The stage input as primitives, own points and halo points in one launch (as k_view).  EULER: the
// inviscid fluxes, which need no more than the point itself, instead of the primitives -- along
// every axis at own points, along the axis of the face a halo point lies beyond.  Both store the mass
// fluxes that the state does not hold: beyond a face to the depth that is differenced, and on
// curvilinear blocks.
template <bool EULER>
__global__ void __launch_bounds__(256, EULER ? 3 : 4) k_view_p(Geometry g, PairPhysics ph, StepSched sc, const double* __restrict__ Uin0,
                                                const double* __restrict__ ring, int in_ring, const SubDev* __restrict__ subs,
                                                const int2* __restrict__ halo, long long nhalo, const float4* __restrict__ H4,
                                                const float2* __restrict__ H2, void* Wp, void* Phi, int stage, int s, int one_stage, int own_blocks, int rev) {
  pdl_enter();
  sc = resolve(sc);
  const double* __restrict__ Uin = ring_or(Uin0, in_ring, ring, sc, 0);
  // (m: the FP64 momentum; as 3: no flux)
  auto put = [&](const SubDev& d, const PrimsP& r, auto m, long long o, int ci, int cj, int as) {
    if (as < 3 && (as >= 0 || d.mbase >= 0)) store_mass_flux(g, d, Phi, o, m, ci, cj, as);
    if (EULER) {
      const float2* M = nullptr;
      if (d.mbase >= 0) M = g.metric_p + d.mbase + (long long)(d.ox + ci + g.G) + (long long)d.mx * (d.oy + cj + g.G);
      store_euler_flux(ph, Phi, g.Ptot, o, r, as, M, d.mpl);
    } else {
      store_prims(w_view(Wp, g.Ptot), o, r);
    }
  };
  const long long b = rev ? gridDim.x - 1 - blockIdx.x : blockIdx.x, nown = (long long)own_blocks * g.nsub;
  if (b < nown) {
    const int sid = (int)(b / own_blocks);
    const SubDev& d = subs[sid];
    if (!d.own) return;  // another process's sub-domain
    const int t = (int)(b - (long long)sid * own_blocks) * blockDim.x + threadIdx.x;
    if (t >= d.sx * d.sy * d.sz) return;
    const int sxy = d.sx * d.sy, ck = t / sxy, r2 = t - ck * sxy, cj = r2 / d.sx, ci = r2 - cj * d.sx;
    const long long gi = (long long)(d.ox + ci) + (long long)d.bnx * ((long long)(d.oy + cj) + (long long)d.bny * (d.oz + ck));
    const long long q = (long long)(ci + g.G) + (long long)d.ex * ((long long)(cj + g.G) + (long long)d.ey * (ck + g.Gz));
    double u[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) u[v] = Uin[d.bbase + v * d.bN + gi];
    put(d, prims_of(ph, u), [&](int a) { return u[1 + a]; }, d.pbase + q, ci, cj, -1);
    return;
  }
  const long long e = (b - nown) * blockDim.x + threadIdx.x;
  if (e >= nhalo) return;
  const int2 hv = halo[e];
  const SubDev& d = subs[hv.x];
  const long long o = d.pbase + hv.y;
  const HaloPoint h = halo_point(g, d, hv);
  // the axis along which the point's flux is differenced: that of the one face it lies beyond
  const int dx = h.ci < 0 ? -h.ci : h.ci - d.sx + 1, dy = h.cj < 0 ? -h.cj : h.cj - d.sy + 1,
            dz = h.ck < 0 ? -h.ck : h.ck - d.sz + 1;
  int as = dx > 0 ? 0 : (dy > 0 ? 1 : 2);
  if (max(dx, max(dy, dz)) > g.fs || (dx > 0) + (dy > 0) + (dz > 0) > 1) as = 3;
  if (sc.mode == 0 || (d.ebase >= 0 && h.beyond && any_own_source(h, d))) {
    double u[5];
    if (h.beyond) {
      const int kd = sc.mode == 0 ? 0 : point_delay(sc, d, h.sid, h.ci, h.cj, h.ck, true);
      gather_value(g, sc, h, d, kd, Uin, ring, stage, s, u);
    } else {
#pragma unroll
      for (int v = 0; v < 5; ++v) u[v] = Uin[v * d.bN + h.gi];
    }
    put(d, prims_of(ph, u), [&](int a) { return u[1 + a]; }, o, h.ci, h.cj, as);
    return;
  }
  const int m = sc.mode == 2 || one_stage ? 0 : stage;
  const P2 a = p_of(H4[(long long)(2 * m) * nhalo + e]), c = p_of(H4[(long long)(2 * m + 1) * nhalo + e]);
  put(d, prims_p(ph, p_x(a), p_pair(p_y(a), p_x(c)), p_y(c), p_of(H2[(long long)m * nhalo + e])),
      [&](int i) { return p_double(i == 0 ? p_y(a) : (i == 1 ? p_x(c) : p_y(c))); }, o, h.ci, h.cj, as);
}

// ------------------------------------------------------------------------------- k_flux_p

namespace {

// Central difference without its factor (times c2 for CD4, c1 for CD2), of two values
template <int R, class W = float2>
__device__ __forceinline__ Pr<W> diff2(const float4* __restrict__ f, long long q, long long st) {
  const Pr<W> c = p_of<W>(f[q + st]), d = p_of<W>(f[q - st]);
  if (R == 1) return p_norm(p_sub(c, d));
  const Pr<W> a = p_of<W>(f[q + 2 * st]), b = p_of<W>(f[q - 2 * st]);
  const W m8 = {-8.f, -8.f};
  const Pr<W> x = p_2diff(a.h, b.h), y = p_2diff(c.h, d.h);
  const Pr<W> s = p_2sum(x.h, v_mul(m8, y.h));
  const W lo = v_add(v_fma(m8, y.l, x.l), v_fma(m8, v_sub(c.l, d.l), v_sub(a.l, b.l)));
  return p_norm(Pr<W>{s.h, v_add(s.l, lo)});
}

}  // namespace

__device__ float g_pow_pair[POW_PAIR_TAB];  // tables of p_pow

// Combined fluxes (but the mass flux, which is the momentum) at the owned points and the strips of r
// points beyond each face (the flux along that face's axis only), thread by thread as in k_flux.
// CURV: the context has curvilinear blocks.  R: stencil radius (CD4: 2).  LAW: the viscosity is the power law.  Bound by instruction issue
// and memory about equally (128^3: half of each).  A Cartesian point forms most of its pairs of values from
// components of others, and bringing those into register pairs for the packed instructions costs more than
// they save: two plain instructions each are faster (121 -> 114 us at 128^3); on curvilinear blocks,
// whose metric products take whole rows, the packed ones are.
template <int R, bool CURV, bool LAW>
__global__ void __launch_bounds__(256, CURV ? 3 : 4) k_flux_p(Geometry g, PairPhysics ph, const SubDev* __restrict__ subs,
                                                const void* __restrict__ Wp, void* __restrict__ Phi, int rev) {
  using V2 = std::conditional_t<CURV, float2, F2>;
  using P2 = Pr<V2>;
  pdl_enter();
  const int sid = rev ? gridDim.y - 1 - blockIdx.y : blockIdx.y;
  const SubDev& d = subs[sid];
  if (!d.own) return;  // another process's sub-domain
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  int ci, cj, ck, kind;
  if (!flux_point<3>(d, R, t, ci, cj, ck, kind)) return;
  const int as = kind - 1;  // strip axis (-1: owned point, every axis)
  const long long P = g.Ptot;
  const long long st[3] = {1, d.ex, (long long)d.ex * d.ey};
  const long long q = d.pbase + (long long)(ci + g.G) + st[1] * (cj + g.G) + st[2] * (ck + g.Gz);
  const float4* __restrict__ A = (const float4*)Wp;
  const float4* __restrict__ B = A + P;
  const float4* __restrict__ Cc = A + 2 * P;
  const float2* __restrict__ D = (const float2*)(A + 3 * P);
  float4* __restrict__ F4 = (float4*)Phi;

  const P2 uv = p_of<V2>(A[q]), wT = p_of<V2>(B[q]), rp = p_of<V2>(Cc[q]);
  const P1 w = p_x(wT), rho = p_x(rp), pr = p_y(rp);
  const P1 rest = rest_enthalpy(ph, p_of(D[q]), rho);
  P1 iv = cst(ph.ivT);  // the factor of the viscous terms: 1/Re x (units of the differences) x mu
  // differences of (u, v) and (w, kappa T) along each axis
  P2 Gx = diff2<R, V2>(A, q, st[0]), Gy = diff2<R, V2>(A, q, st[1]), Gz = diff2<R, V2>(A, q, st[2]);
  P2 Hz = diff2<R, V2>(B, q, st[2]);
  P2 Hx = {V2{0.f, 0.f}, V2{0.f, 0.f}}, Hy = Hx;
  if (as != 1) Hx = diff2<R, V2>(B, q, st[0]);
  if (as != 0) Hy = diff2<R, V2>(B, q, st[1]);
  const bool curv = CURV && d.mbase >= 0;
  P2 xi = {V2{0.f, 0.f}, V2{0.f, 0.f}}, et = xi;  // metric rows (xi_x, xi_y), (eta_x, eta_y)
  P1 zz = {0.f, 0.f};
  if (curv) {
    // index-space differences to physical gradients / J: x: xi_x, eta_x; y: xi_y, eta_y; z: zeta_z
    const float2* M = g.metric_p + d.mbase + (long long)(d.ox + ci + g.G) + (long long)d.mx * (d.oy + cj + g.G);
    const long long pl = d.mpl;
    xi = p_pair<V2>(p_of(M[0]), p_of(M[pl]));
    et = p_pair<V2>(p_of(M[2 * pl]), p_of(M[3 * pl]));
    zz = p_of(M[4 * pl]);
    if (as == 1) Hx = diff2<R, V2>(B, q, st[0]);  // (the rows mix the two in-plane differences)
    if (as == 0) Hy = diff2<R, V2>(B, q, st[1]);
    const P2 g0 = Gx, h0 = Hx;
    Gx = p_norm(p_fma(p_bc<V2>(p_x(et)), Gy, p_mul(p_bc<V2>(p_x(xi)), g0)));
    Hx = p_norm(p_fma(p_bc<V2>(p_x(et)), Hy, p_mul(p_bc<V2>(p_x(xi)), h0)));
    Gy = p_norm(p_fma(p_bc<V2>(p_y(et)), Gy, p_mul(p_bc<V2>(p_y(xi)), g0)));
    Hy = p_norm(p_fma(p_bc<V2>(p_y(et)), Hy, p_mul(p_bc<V2>(p_y(xi)), h0)));
    Gz = p_norm(p_mul(p_bc<V2>(zz), Gz));
    Hz = p_norm(p_mul(p_bc<V2>(zz), Hz));
    iv = p_norm(p_mul(iv, p_norm(p_mul(cst(d.cg[0]), p_of(M[6 * pl])))));
  } else if (d.iso) {
    iv = p_norm(p_mul(iv, cst(d.cg[0])));
  } else {
    const P2 kx = p_bc<V2>(cst(d.cg[0])), ky = p_bc<V2>(cst(d.cg[1])), kz = p_bc<V2>(cst(d.cg[2]));
    Gx = p_norm(p_mul(kx, Gx));
    Hx = p_norm(p_mul(kx, Hx));
    Gy = p_norm(p_mul(ky, Gy));
    Hy = p_norm(p_mul(ky, Hy));
    Gz = p_norm(p_mul(kz, Gz));
    Hz = p_norm(p_mul(kz, Hz));
  }
  if (LAW) iv = p_norm(p_mul(iv, p_pow(p_y(wT), cst(ph.visc_exp), g_pow_pair)));
  // tau / (mu gs): diagonal (t00, t11), t22, t01, and (t02, t12)
  const P2 dia = p_pair<V2>(p_x(Gx), p_y(Gy));
  const P1 div = p_norm(p_mul(P1{-0.6666667f, 1.9868216e-08f}, p_norm(p_add(p_add(p_x(dia), p_y(dia)), p_x(Hz)))));
  const P2 td = p_norm(p_add(p_scale(dia, 2.f), p_bc<V2>(div)));
  const P1 t22 = p_norm(p_add(p_scale(p_x(Hz), 2.f), div));
  const P1 t01 = p_norm(p_add(p_x(Gy), p_y(Gx)));
  const P2 t2 = p_norm(p_add(Gz, p_pair<V2>(p_x(Hx), p_x(Hy))));
  // b_a = u_i tau_ai + kappa mu dT/dx_a of row (ra, rc) = ((tau_a0, tau_a1), tau_a2)
  auto heat = [&](P2 ra, P1 rc, P1 dT) {
    const P2 x = p_mul(uv, ra);
    return p_norm(p_fma(w, rc, p_add(p_add(p_x(x), p_y(x)), dT)));
  };
  auto put = [&](int a, P2 m, P2 e) {
    F4[(long long)(2 * a) * P + q] = p_store(p_norm(m));
    F4[(long long)(2 * a + 1) * P + q] = p_store(p_norm(e));
  };
  const P1 zero = {0.f, 0.f};
  if (curv) {
    const P1 b0 = heat(p_pair<V2>(p_x(td), t01), p_x(t2), p_y(Hx)), b1 = heat(p_pair<V2>(t01, p_y(td)), p_y(t2), p_y(Hy)),
             b2 = heat(t2, t22, p_y(Hz));
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      if (as >= 0 && as != a) continue;
      const P2 row = a == 0 ? xi : et;
      const P2 x = p_mul(row, uv);
      const P1 Uc = p_norm(p_add(p_x(x), p_y(x)));  // contravariant velocity
      const P1 n = p_norm(p_neg(p_mul(rho, Uc)));
      const P2 r0 = p_bc<V2>(p_x(row)), r1 = p_bc<V2>(p_y(row));
      P2 m = p_sub(p_mul(p_bc<V2>(n), uv), p_mul(p_bc<V2>(pr), row));
      m = p_fma(p_bc<V2>(iv), p_norm(p_fma(r0, p_pair<V2>(p_x(td), t01), p_mul(r1, p_pair<V2>(t01, p_y(td))))), m);
      P2 e = p_mul(p_pair<V2>(n, rest), p_pair<V2>(w, Uc));
      e = p_fma(p_bc<V2>(iv), p_norm(p_fma(r0, p_pair<V2>(p_x(t2), b0), p_mul(r1, p_pair<V2>(p_y(t2), b1)))), e);
      put(a, m, e);
    }
    if (as < 0 || as == 2) {
      const P1 Uc = p_norm(p_mul(zz, w)), n = p_norm(p_neg(p_mul(rho, Uc)));
      const P2 iz = p_bc<V2>(p_norm(p_mul(iv, zz)));
      const P2 m = p_fma(iz, t2, p_mul(p_bc<V2>(n), uv));
      P2 e = p_mul(p_pair<V2>(n, rest), p_pair<V2>(w, Uc));
      e = p_sub(e, p_pair<V2>(p_mul(zz, pr), zero));
      put(2, m, p_fma(iz, p_pair<V2>(t22, b2), e));
    }
    return;
  }
  const P2 nuv = p_norm(p_neg(p_mul(p_bc<V2>(rho), uv)));  // -rho u, -rho v
  if (as < 0 || as == 0) {
    const P2 ra = p_pair<V2>(p_x(td), t01);
    P2 m = p_sub(p_mul(p_bc<V2>(p_x(nuv)), uv), p_pair<V2>(pr, zero));
    P2 e = p_mul(p_pair<V2>(p_x(nuv), rest), p_pair<V2>(w, p_x(uv)));
    put(0, p_fma(p_bc<V2>(iv), ra, m), p_fma(p_bc<V2>(iv), p_pair<V2>(p_x(t2), heat(ra, p_x(t2), p_y(Hx))), e));
  }
  if (as < 0 || as == 1) {
    const P2 ra = p_pair<V2>(t01, p_y(td));
    P2 m = p_sub(p_mul(p_bc<V2>(p_y(nuv)), uv), p_pair<V2>(zero, pr));
    P2 e = p_mul(p_pair<V2>(p_y(nuv), rest), p_pair<V2>(w, p_y(uv)));
    put(1, p_fma(p_bc<V2>(iv), ra, m), p_fma(p_bc<V2>(iv), p_pair<V2>(p_y(t2), heat(ra, p_y(t2), p_y(Hy))), e));
  }
  if (as < 0 || as == 2) {
    const P1 n = p_norm(p_neg(p_mul(rho, w)));
    const P2 m = p_mul(p_bc<V2>(n), uv);
    P2 e = p_sub(p_mul(p_pair<V2>(n, rest), p_pair<V2>(w, w)), p_pair<V2>(pr, zero));
    put(2, p_fma(p_bc<V2>(iv), t2, m), p_fma(p_bc<V2>(iv), p_pair<V2>(t22, heat(t2, t22, p_y(Hz))), e));
  }
}

// ------------------------------------------------------------------------------- k_rk_p

// dt R = sum_a dt D_a Phi_a (times J on a curvilinear block), of the mass flux in FP64, of the others on
// pairs, the energy taking H_ref times the mass's; then the low-storage update Q = A Q + dt R, U^(m) =
// U^(m-1) + B Q in FP64.  Bound by memory latency (310 B of traffic per point at half the DRAM rate, 64
// registers) and by the FP64 pipe, on which 24 operations per point take as long as 1,500 others: the
// pairs are converted on the integer pipe (154 -> 135 us at 128^3).  Q, density and energy, not read again
// before they would be evicted anyway, pass by the caches as streaming accesses and leave the L2
// to what neighbouring points share.
template <int R>
__global__ void __launch_bounds__(256, 4) k_rk_p(Geometry g, StepSched sc, const SubDev* __restrict__ subs,
                                              const void* __restrict__ Phi, const double* __restrict__ Uin0,
                                              double* __restrict__ Uout0, const double* __restrict__ ring, int in_ring,
                                              int out_ring, double* __restrict__ Q, double A, double B, float2 dt, double dtd,
                                              double H, int first, int last, int rev) {
  pdl_enter();
  sc = resolve(sc);
  const double* Uin = ring_or(Uin0, in_ring, ring, sc, 0);
  double* Uout = const_cast<double*>(ring_or(Uout0, out_ring, ring, sc, 1));
  const int sid = rev ? gridDim.y - 1 - blockIdx.y : blockIdx.y;
  const SubDev& d = subs[sid];
  if (!d.own) return;  // another process's sub-domain
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= d.sx * d.sy * d.sz) return;
  const int sxy = d.sx * d.sy, ck = t / sxy, r2 = t - ck * sxy, cj = r2 / d.sx, ci = r2 - cj * d.sx;
  const long long st[3] = {1, d.ex, (long long)d.ex * d.ey};
  const long long q = d.pbase + (long long)(ci + g.G) + st[1] * (cj + g.G) + st[2] * (ck + g.Gz);
  const long long gi = d.bbase + (long long)(d.ox + ci) + (long long)d.bnx * ((long long)(d.oy + cj) + (long long)d.bny * (d.oz + ck));
  const long long P = g.Ptot;
  const float4* __restrict__ F4 = (const float4*)Phi;
  const double* __restrict__ N = (const double*)(F4 + 6 * P);
  double qv[5], uv[5];
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    qv[c] = first ? 0.0 : __ldcs(Q + c * d.bN + gi);
    uv[c] = c >= 1 && c <= 3 ? Uin[c * d.bN + gi] : __ldcs(Uin + c * d.bN + gi);
  }
  P2 m = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)}, e = m;
  double n = 0.0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const P1 k = p_norm(p_mul(cst(dt), cst(d.cg[a])));
    m = p_fma(p_bc(k), diff2<R>(F4 + (long long)(2 * a) * P, q, st[a]), m);
    e = p_fma(p_bc(k), diff2<R>(F4 + (long long)(2 * a + 1) * P, q, st[a]), e);
    const int ca = a == 0 ? ci : (a == 1 ? cj : ck), sa = a == 0 ? d.sx : (a == 1 ? d.sy : d.sz);
    const long long gst = a == 0 ? 1 : (a == 1 ? (long long)d.bnx : (long long)d.bnx * d.bny);
    const double *pu = Uin + (1 + a) * d.bN + gi, *pn = N + a * P + q;
    const bool cart = d.mbase < 0;
    auto mass = [&](int o) { return cart && (unsigned)(ca + o) < (unsigned)sa ? __ldg(pu + o * gst) : __ldg(pn + o * st[a]); };
    const double d1 = mass(1) - mass(-1);
    n = R == 1 ? fma(d.c1[a], d1, n) : fma(d.c2[a], fma(-8.0, d1, mass(2) - mass(-2)), n);
  }
  n *= -dtd;
  if (d.mbase >= 0) {
    const long long mq = d.mbase + 6 * d.mpl + (long long)(d.ox + ci + g.G) + (long long)d.mx * (d.oy + cj + g.G);
    const P1 J = p_of(g.metric_p[mq]);
    m = p_mul(p_bc(J), p_norm(m));
    e = p_mul(p_bc(J), p_norm(e));
    n *= g.metric[mq];
  }
  m = p_norm(m);
  e = p_norm(e);
  const double dtR[5] = {n, p_double_int(p_x(m)), p_double_int(p_y(m)), p_double_int(p_x(e)), fma(H, n, p_double_int(p_y(e)))};
  const bool wallpt = d.wall && ((((d.wall >> 0) & 1) && ci == 0) || (((d.wall >> 1) & 1) && ci == d.sx - 1) ||
                                 (((d.wall >> 2) & 1) && cj == 0) || (((d.wall >> 3) & 1) && cj == d.sy - 1));
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    double qn = first ? dtR[c] : fma(A, qv[c], dtR[c]);
    double un = fma(B, qn, uv[c]);
    if (wallpt && c >= 1 && c <= 3) qn = un = 0.0;  // no-slip wall points keep zero momentum
    if (!last) __stcs(Q + c * d.bN + gi, qn);
    Uout[c * d.bN + gi] = un;
  }
}

// ------------------------------------------------------------------------------- compact scheme

// Sixth-order compact derivative (Eq. 2, alpha = 1/3; closure as k_compact_div) of the fluxes along
// `axis`, one thread per line and group of components: M (x, y momentum) and E (z momentum, what the
// energy flux carries beside H_ref times the mass flux) on pairs, N (mass) into FP64.  In units
// of b/(4h) the right side is (f_{i+2} - f_{i-2}) + 28 (f_{i+1} - f_{i-1}); the sweeps z_i = rhs_i -
// c_{i-1} z_{i-1}, x_i = z_i / m_i - c_i x_{i+1} keep z_i in shared memory ([n][CL], CL lines per CTA),
// where every line is staged first with all its loads in flight (x: a warp along a line, y and z: a warp
// across 32 lines).  dt R gathers in R over the x and y passes; the z pass adds its part and takes the
// low-storage update, so the divergence is neither written nor read a third time.  The energy's dt R takes
// H_ref times the whole of the mass's, so the y launch solves N along z as well (into the
// scratch of its x flux, which the launch before consumed) and the z launch's E group updates the density
// too.  In FP64 the three passes were bound by their eight operations per value (190 us each at 128^3).
constexpr int CL = 64;  // lines per CTA

// The lines of a CTA along `axis` of sub-domain d
template <int axis>
struct LineSet {
  static constexpr int LD = axis == 0 ? CL + 1 : CL;
  static constexpr int a1 = axis == 0 ? 1 : 0, a2 = axis == 2 ? 1 : 2;
  int n, nlines, l0, s1;
  long long st[3], gst[3], q0, r0;
  __device__ __forceinline__ LineSet(const Geometry& g, const SubDev& d) {
    const int sz[3] = {d.sx, d.sy, d.sz};
    n = sz[axis];
    s1 = sz[a1];
    l0 = blockIdx.x * CL;
    nlines = min(CL, s1 * sz[a2] - l0);
    st[0] = gst[0] = 1;
    st[1] = d.ex;
    st[2] = (long long)d.ex * d.ey;
    gst[1] = d.bnx;
    gst[2] = (long long)d.bnx * d.bny;
    q0 = d.pbase + g.G + st[1] * g.G + st[2] * g.Gz;
    r0 = d.bbase / 5 + (long long)d.ox + gst[1] * d.oy + gst[2] * d.oz;
  }
  // line l of the CTA: its first point in the padded box and in the state's point order
  __device__ __forceinline__ void at(int l, long long& q, long long& r) const {
    const int t = l0 + l, t1 = t % s1, t2 = t / s1;
    q = q0 + t1 * st[a1] + t2 * st[a2];
    r = r0 + t1 * gst[a1] + t2 * gst[a2];
  }
  // the lines and 4 points beyond each end to shared memory
  __device__ __forceinline__ void stage(float4* sm, const float4* __restrict__ F) const {
    const int tid = threadIdx.x;
    long long q, r;
    if (axis == 0) {
      const int lane = tid & 31;
      for (int l = tid >> 5; l < nlines; l += CL / 32) {
        at(l, q, r);
        for (int i = lane; i < n + 8; i += 32) cp_async16(sm + i * LD + l, F + q + i - 4);
      }
    } else if (tid < nlines) {
      at(tid, q, r);
      for (int i = 0; i < n + 8; ++i) cp_async16(sm + i * LD + tid, F + q + (i - 4) * st[axis]);
    }
    cp_async_commit();
    cp_async_wait_all();
    __syncthreads();
  }
  // the solved lines along x from shared memory to R
  __device__ __forceinline__ void unstage(const float4* sm, float4* __restrict__ R) const {
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int l = threadIdx.x >> 5; l < nlines; l += CL / 32) {
      long long q, r;
      at(l, q, r);
      for (int i = lane; i < n; i += 32) R[r + i] = sm[i * LD + l];
    }
  }
};

// What the z launch's update takes beside the group's own dt R
struct CompactUpdate {
  const double* Uin;
  double *Uout, *Q;
  const double *RN, *NZ;  // the mass's dt R: of the x and y passes in point order, of the z pass in scratch order
  double A, B, H;
  int first, last;
};

// grp 0: M, 1: E
template <int axis, int grp>
__device__ __forceinline__ void compact_group(const Geometry& g, const SubDev& d, const float4* __restrict__ F,
                                              float4* __restrict__ R, const float2* __restrict__ cth, int Lmax, float2 dt,
                                              unsigned char* raw, const CompactUpdate& up) {
  float4* sm = reinterpret_cast<float4*>(raw);
  const LineSet<axis> ls(g, d);
  constexpr int LD = LineSet<axis>::LD;
  const int n = ls.n, tid = threadIdx.x;
  ls.stage(sm, F);
  if (tid < ls.nlines) {
    long long q, r;
    ls.at(tid, q, r);
    const float2* __restrict__ cp = cth;
    const float2* __restrict__ im = cp + Lmax;
    auto f = [&](int i) -> P2 { return p_of(sm[(i + 4) * LD + tid]); };
    // closures at the first halo points, 0.6 (45 (f_1 - f_-1) - 9 (f_2 - f_-2) + (f_3 - f_-3)), times alpha
    auto cst1 = [](float h, float l) { return P2{v_bc<float2>(h), v_bc<float2>(l)}; };
    auto closure = [&](P2 d1, P2 d2, P2 d3) {
      P2 x = p_fma(cst1(45.f, 0.f), d1, d3);
      x = p_norm(p_fma(cst1(-9.f, 0.f), d2, x));
      return p_norm(p_mul(cst1(0.2f, -2.9802323e-09f), x));  // 0.6 / 3
    };
    P2 w[5];  // f(i - 2) .. f(i + 2)
    const P2 m4 = f(-4), m3 = f(-3);
    w[0] = f(-2);
    w[1] = f(-1);
    w[2] = f(0);
    w[3] = f(1);
    w[4] = f(2);
    const P2 dl = closure(p_norm(p_sub(w[2], w[0])), p_norm(p_sub(w[3], m3)), p_sub(w[4], m4));
    P2 z = {v_bc<float2>(0.f), v_bc<float2>(0.f)};
    float2 cm = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int i = 0; i < n; ++i) {
      P2 rhs = p_fma(cst1(28.f, 0.f), p_norm(p_sub(w[3], w[1])), p_sub(w[4], w[0]));
      if (i == 0) rhs = p_sub(rhs, dl);
      if (i == n - 1)
        rhs = p_sub(rhs, closure(p_norm(p_sub(w[4], w[2])), p_norm(p_sub(f(n + 2), w[1])), p_sub(f(n + 3), w[0])));
      z = p_norm(p_fma(cst1(-cm.x, -cm.y), z, rhs));
      // (slot i held f(i - 4), no longer read)
      sm[i * LD + tid] = p_store(z);
      cm = __ldg(cp + i);
#pragma unroll
      for (int k = 0; k < 4; ++k) w[k] = w[k + 1];
      if (i + 1 < n) w[4] = f(i + 3);
    }
    // k = dt b / (4h): the difference coefficient of the block is -1 / (12 h)
    const P1 k1 = p_norm(p_mul(p_norm(p_mul(P1{dt.x, dt.y}, cst(d.cg[axis]))), P1{-0.33333334f, 9.934108e-09f}));
    const P2 kk = cst1(k1.h, k1.l);
    P2 x = {v_bc<float2>(0.f), v_bc<float2>(0.f)};
    constexpr int NU = grp == 0 ? 2 : 3;  // variables that the z launch updates: 1, 2 or 3, 4, 0
    auto comp = [](int v) { return grp == 0 ? 1 + v : (v < 2 ? 3 + v : 0); };
    // four points at a time, what they read from memory in flight before the first is solved
    for (int i0 = n - 1; i0 >= 0; i0 -= 4) {
      float4 rv[4];
      double qv[4][NU], uv[4][NU], nv[4];
      if (axis > 0) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (i0 - k >= 0) {
            const long long ri = r + (long long)(i0 - k) * ls.gst[axis], pt = ri - d.bbase / 5;
            rv[k] = R[ri];
            if (axis == 2) {
#pragma unroll
              for (int v = 0; v < NU; ++v) {
                const long long gi = d.bbase + (long long)comp(v) * d.bN + pt;
                qv[k][v] = up.first ? 0.0 : __ldcs(up.Q + gi);
                uv[k][v] = __ldcs(up.Uin + gi);
              }
              if (grp == 1) nv[k] = up.RN[ri] + up.NZ[q + (i0 - k) * ls.st[2]];
            }
          }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int i = i0 - k;
        if (i < 0) break;
        const float2 c = __ldg(cp + i), m = __ldg(im + i);
        x = p_norm(p_fma(cst1(-c.x, -c.y), x, p_mul(cst1(m.x, m.y), p_of(sm[i * LD + tid]))));
        const P2 kx = p_mul(kk, x);
        if (axis == 0) {
          sm[i * LD + tid] = p_store(p_norm(kx));
          continue;
        }
        const long long ri = r + (long long)i * ls.gst[axis];
        const P2 sum = p_norm(p_add(kx, p_of(rv[k])));
        if (axis == 1) {
          R[ri] = p_store(sum);
          continue;
        }
        const long long pt = ri - d.bbase / 5;
        double dtR[3] = {p_double(p_x(sum)), p_double(p_y(sum)), 0.0};
        if (grp == 1) {
          dtR[1] = fma(up.H, nv[k], dtR[1]);
          dtR[2] = nv[k];
        }
#pragma unroll
        for (int v = 0; v < NU; ++v) {
          const long long gi = d.bbase + (long long)comp(v) * d.bN + pt;
          const double qn = up.first ? dtR[v] : fma(up.A, qv[k][v], dtR[v]);
          if (!up.last) __stcs(up.Q + gi, qn);
          up.Uout[gi] = fma(up.B, qn, uv[k][v]);
        }
      }
    }
  }
  if (axis == 0) ls.unstage(sm, R);
}

// N along one axis: x into R, y added to it, z into the scratch array NZ, in FP64.  The line's right side is
// differenced in FP64; the system is solved on pairs for what the solution x has beside 3/5 of it (the
// system's row sum is 5/3), (1/3, 1, 1/3) y = -1/5 delta^2 rhs, which is small for smooth fluxes, so
// that the sweeps' rounding is small against that of x.
template <int axis>
__device__ __forceinline__ void compact_mass(const Geometry& g, const SubDev& d, const double* __restrict__ Uin,
                                             const double* __restrict__ F, double* __restrict__ R, double* __restrict__ NZ,
                                             const float2* __restrict__ cth, int Lmax, double dt, unsigned char* raw) {
  const LineSet<axis> ls(g, d);
  constexpr int LD = LineSet<axis>::LD;
  const int n = ls.n, tid = threadIdx.x;
  float4* sm = reinterpret_cast<float4*>(raw);  // a slot: the FP64 flux in its first half, later the pairs z and rhs
  auto val = [&](int i, int l) -> double& { return *reinterpret_cast<double*>(sm + i * LD + l); };
  // the lines and 4 points beyond each end: inside the sub-domain from the momentum (indexed as R is, in point
  // order over all blocks), beyond its faces from the scratch array
  const double* __restrict__ U = Uin + d.bbase + (1 + axis) * d.bN - d.bbase / 5;
  auto copy = [&](int l, int i, long long q, long long r) {
    const int k = i - 4;
    cp_async8(&val(i, l), (unsigned)k < (unsigned)n ? U + r + k * ls.gst[axis] : F + q + k * ls.st[axis]);
  };
  long long q, r;
  if (axis == 0) {
    for (int l = tid >> 5; l < ls.nlines; l += CL / 32) {
      ls.at(l, q, r);
      for (int i = tid & 31; i < n + 8; i += 32) copy(l, i, q, r);
    }
  } else if (tid < ls.nlines) {
    ls.at(tid, q, r);
    for (int i = 0; i < n + 8; ++i) copy(tid, i, q, r);
  }
  cp_async_commit();
  cp_async_wait_all();
  __syncthreads();
  if (tid < ls.nlines) {
    ls.at(tid, q, r);
    auto f = [&](int i) { return val(i + 4, tid); };
    const P1 fifth = {0.2f, -2.9802323e-09f};
    // 1/3 of the closure at the first halo point, 0.6 (45 (f_1 - f_-1) - 9 (f_2 - f_-2) + (f_3 - f_-3))
    auto closure = [&](double d1, double d2, double d3) { return p_mul(fifth, p_split(fma(45.0, d1, fma(-9.0, d2, d3)))); };
    auto right = [](const double* w) { return p_split(fma(28.0, w[3] - w[1], w[4] - w[0])); };
    double w[5] = {f(-3), f(-2), f(-1), f(0), f(1)};  // f(i - 2) .. f(i + 2)
    auto next = [&](double v) {
#pragma unroll
      for (int k = 0; k < 4; ++k) w[k] = w[k + 1];
      w[4] = v;
    };
    P1 rm = right(w);  // right sides of points i - 1, i, i + 1
    next(f(2));
    P1 rc = right(w);
    const P1 yl = p_norm(p_sub(closure(w[2] - w[0], w[3] - f(-3), w[4] - f(-4)), p_mul(fifth, rm)));
    P1 z = {0.f, 0.f};
    float2 cm = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int i = 0; i < n; ++i) {
      next(f(i + 3));
      const P1 rn = right(w);
      P1 h = p_norm(p_mul(fifth, p_norm(p_sub(p_sub(rc, rm), p_sub(rn, rc)))));
      if (i == 0) h = p_sub(h, yl);
      if (i == n - 1)
        h = p_sub(h, p_norm(p_sub(closure(w[3] - w[1], w[4] - w[0], f(n + 3) - f(n - 3)), p_mul(fifth, rn))));
      z = p_norm(p_fma(P1{-cm.x, -cm.y}, z, h));
      // (slot i held f(i - 4), no longer read)
      sm[i * LD + tid] = make_float4(z.h, z.l, rc.h, rc.l);
      cm = __ldg(cth + i);
      rm = rc;
      rc = rn;
    }
    const double kk = dt * d.c2[axis] / 3.0;  // -dt b / (4h)
    P1 y = {0.f, 0.f};
    for (int i0 = n - 1; i0 >= 0; i0 -= 4) {
      double rv[4];
      if (axis == 1)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (i0 - k >= 0) rv[k] = R[r + (long long)(i0 - k) * ls.gst[1]];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int i = i0 - k;
        if (i < 0) break;
        const float2 c = __ldg(cth + i), m = __ldg(cth + Lmax + i);
        const float4 v = sm[i * LD + tid];
        y = p_norm(p_fma(P1{-c.x, -c.y}, y, p_mul(P1{m.x, m.y}, P1{v.x, v.y})));
        const double x = p_double_int(p_norm(p_fma(P1{0.6f, -2.3841858e-08f}, P1{v.z, v.w}, y)));
        if (axis == 0) val(i, tid) = kk * x;
        else if (axis == 1) R[r + (long long)i * ls.gst[1]] = fma(kk, x, rv[k]);
        else NZ[q + i * ls.st[2]] = kk * x;
      }
    }
  }
  if (axis == 0) {
    __syncthreads();
    for (int l = tid >> 5; l < ls.nlines; l += CL / 32) {
      ls.at(l, q, r);
      for (int i = tid & 31; i < n; i += 32) R[r + i] = val(i, l);
    }
  }
}

// blockIdx.y: M, E and, in the x and y launches, N along that axis, in the y launch N along z
template <int axis>
__global__ void __launch_bounds__(CL) k_compact_p(Geometry g, StepSched sc, const SubDev* __restrict__ subs, void* Phi,
                                                  void* __restrict__ Rv, const float2* __restrict__ cth, int Lmax,
                                                  const double* __restrict__ Uin0, double* __restrict__ Uout0,
                                                  const double* __restrict__ ring, int in_ring, int out_ring,
                                                  double* __restrict__ Q, double A, double B, double H, float2 dt, double dtd,
                                                  int first, int last, int rev) {
  extern __shared__ __align__(16) unsigned char craw[];
  pdl_enter();
  const SubDev& d = subs[rev ? gridDim.z - 1 - blockIdx.z : blockIdx.z];
  const int grp = blockIdx.y;
  const int lines = grp == 3 || axis == 2 ? d.sx * d.sy : (axis == 0 ? d.sy * d.sz : d.sx * d.sz);
  if (!d.own || (int)blockIdx.x * CL >= lines) return;
  const long long P = g.Ptot, N = g.N;
  const float4* F4 = (const float4*)Phi;
  double* FN = (double*)((float4*)Phi + 6 * P);
  float4* R4 = (float4*)Rv;
  double* RN = (double*)(R4 + 2 * N);
  sc = resolve(sc);
  const double* Uin = ring_or(Uin0, in_ring, ring, sc, 0);
  CompactUpdate up{};
  if (axis == 2) up = {Uin, const_cast<double*>(ring_or(Uout0, out_ring, ring, sc, 1)), Q, RN, FN, A, B, H, first, last};
  if (grp == 0) compact_group<axis, 0>(g, d, F4 + 2 * axis * P, R4, cth, Lmax, dt, craw, up);
  else if (grp == 1) compact_group<axis, 1>(g, d, F4 + (2 * axis + 1) * P, R4 + N, cth, Lmax, dt, craw, up);
  else if (axis < 2 && grp == 2) compact_mass<axis>(g, d, Uin, FN + axis * P, RN, nullptr, cth, Lmax, dtd, craw);
  else if (axis == 1) compact_mass<2>(g, d, Uin, FN + 2 * P, nullptr, FN, cth, Lmax, dtd, craw);
}

// ------------------------------------------------------------------------------- launchers

// The tables of p_pow in the current device's copy of the array, once per device (as
// pow_tables_init).
int pow_pair_tables_init() {
  constexpr int kMaxDev = 64;
  static std::mutex mu;
  static bool done[kMaxDev] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return (int)e;
  if (dev < 0 || dev >= kMaxDev) return (int)cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(mu);
  if (done[dev]) return 0;
  float t[POW_PAIR_TAB];
  pow_pair_table(t);
  e = cudaMemcpyToSymbol(g_pow_pair, t, sizeof(t));
  if (e != cudaSuccess) return (int)e;
  done[dev] = true;
  return 0;
}

int launch_at_halo(const Geometry& g, const PairPhysics& ph, const StepSched& sc, const double* ring, const SubDev* subs,
                   const int* halo, long long nhalo, void* H, int s, int only, void* stream, long long* launches,
                   const Timer* tm) {
  if (nhalo <= 0) return 0;
  float4* H4 = (float4*)H;
  float2* H2 = (float2*)(H4 + 2LL * (only >= 0 ? 1 : s) * nhalo);
  TIMED(tm, 0, (launch_pdl(s == 2 ? k_at_halo<2> : k_at_halo<5>, dim3(nblk(nhalo, 256)), dim3(256), 0, (cudaStream_t)stream, g,
                           ph, sc, ring, subs, (const int2*)halo, nhalo, only, H4, H2)));
  if (launches) *launches += 1;
  return (int)cudaGetLastError();
}

int launch_stage_pairs(const Geometry& g, const PairPhysics& ph, const StepSched& sc, const StageLaunch& a, const void* H,
                       void* stream, long long* launches, const Timer* tm) {
  const cudaStream_t st = (cudaStream_t)stream;
  const int B = a.threads == 128 ? 128 : 256;
  const float4* H4 = (const float4*)H;
  const float2* H2 = (const float2*)(H4 + 2LL * (a.one_stage ? 1 : a.s) * a.nhalo);
  const unsigned own_blocks = nblk(a.max_own, B);
  const unsigned nb = own_blocks * (unsigned)g.nsub + nblk(a.nhalo, B);
  const dim3 gf(nblk(a.max_flux, B), g.nsub), gr(nblk(a.max_own, B), g.nsub);
  const float dth = (float)a.dt;
  const float2 dt = make_float2(dth, (float)(a.dt - (double)dth));
  // Each kernel takes the sub-domains in the opposite order of the one before it, so that it starts on
  // what that one wrote last and the L2 still holds (a step of 128^3 in 64 sub-domains: 2450 -> 2417 us;
  // 100^3 in 27: 1117 -> 1089)
  const int per_stage = a.compact ? 4 : (g.viscous ? 3 : 2);
  auto rev = [&](int k) { return (a.stage * per_stage + k) & 1; };
  // (inviscid: the fluxes come straight from the view)
  TIMED(tm, 0, (launch_pdl(g.viscous ? k_view_p<false> : k_view_p<true>, dim3(nb), dim3(B), 0, st, g, ph, sc, a.Uin, a.ring, a.in_ring, a.subs, (const int2*)a.halo,
                           a.nhalo, H4, H2, a.Wp, a.Phi, a.stage, a.s, a.one_stage, (int)own_blocks, rev(0))));
  if (launches) *launches += 1;
  if (a.compact) {
    // x and y passes gather dt R, the z pass takes the update
    const size_t slots = (size_t)(a.Lmax + 8) * CL, staged = (size_t)(a.Lmax + 8) * (CL + 1);
    const float2* cth = (const float2*)a.cthomas;
    auto run = [&](auto kernel, size_t smem, unsigned groups, int k) {
      const dim3 gc(nblk((long long)a.Lmax * a.Lmax, CL), groups, g.nsub);
      TIMED(tm, 2, (launch_pdl(kernel, gc, dim3(CL), smem * sizeof(float4), st, g, sc, a.subs, a.Phi, (void*)a.R, cth, a.Lmax,
                               a.Uin, a.Uout, a.ring, a.in_ring, a.out_ring, a.Q, a.A, a.B, ph.Hd, dt, a.dt, a.first, a.last, rev(k))));
    };
    run(k_compact_p<0>, staged, 3, 1);
    run(k_compact_p<1>, slots, 4, 2);
    run(k_compact_p<2>, slots, 2, 3);
    if (launches) *launches += 3;
    return (int)cudaGetLastError();
  }
  if (g.viscous) {
    auto pick = [&](auto r) {
      constexpr int R = decltype(r)::value;
      if (ph.visc_law == 1) return g.metric ? k_flux_p<R, true, true> : k_flux_p<R, false, true>;
      return g.metric ? k_flux_p<R, true, false> : k_flux_p<R, false, false>;
    };
    const auto flux = g.r == 2 ? pick(std::integral_constant<int, 2>{}) : pick(std::integral_constant<int, 1>{});
    TIMED(tm, 1, (launch_pdl(flux, gf, dim3(B), 0, st, g, ph, a.subs, (const void*)a.Wp, a.Phi, rev(1))));
    if (launches) *launches += 1;
  }
  auto rk = g.r == 2 ? k_rk_p<2> : k_rk_p<1>;
  TIMED(tm, 2, (launch_pdl(rk, gr, dim3(B), 0, st, g, sc, a.subs, (const void*)a.Phi, a.Uin, a.Uout, a.ring, a.in_ring,
                           a.out_ring, a.Q, a.A, a.B, dt, a.dt, ph.Hd, a.first, a.last, rev(g.viscous ? 2 : 1))));
  if (launches) *launches += 1;
  return (int)cudaGetLastError();
}

// The shared-memory opt-in of the compact passes for lines of up to Lmax points: a per-device attribute
// shared by every context, so it only ever rises (as filter_prepare).
int compact_pairs_prepare(int Lmax) {
  const size_t sm = (size_t)(Lmax + 8) * (CL + 1) * sizeof(float4);
  if (sm > 227 * 1024) return (int)cudaErrorInvalidValue;
  static std::mutex mu;
  static int set_to[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return (int)e;
  if (dev < 0 || dev >= 64) return (int)cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(mu);
  if ((int)sm <= set_to[dev]) return 0;
  e = cudaFuncSetAttribute(k_compact_p<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_compact_p<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_compact_p<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e == cudaSuccess) set_to[dev] = (int)sm;
  return (int)e;
}

}  // namespace cfs

// euler2d.cu -- the Runge-Kutta stage of the FP64 form for two-dimensional inviscid runs on periodic
// Cartesian blocks in one launch (view, flux and update of kernels.cu in one).
//
// Small grids (64 x 64) are bound by launches: three kernels per stage take 14 us whatever they do.
// Large ones (1024 x 1024) are bound by the FP64 pipe, 2 operations per clock and SM, and by the
// scratch arrays between the kernels.  A CTA takes a tile of one sub-domain: its threads form the
// primitives and fluxes of the tile's points and of its rim (R columns and rows
// beyond it, halo points by the schedule), the fluxes go through shared memory, and each thread
// updates its points.  The mass flux is the momentum itself, the off-diagonal momentum flux is
// shared by the axes, the differences are taken without their factor where the spacings are equal,
// and a tile without z momentum and with finite velocities leaves that component out (it stays zero).  Five fourth-order steps of
// 64^2: 359 -> 171 us; a second-order step of 1024^2: 348 -> 303 us (131 us per stage, 81 of them at
// the FP64 rate).
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "cfs_internal.h"
#include "device_common.cuh"
#include "launch_common.cuh"

namespace cfs {

template <int R, int TX, int TY>
struct E2Smem {
  static constexpr int FW = TX + 2 * R;
  // fluxes of the tile extended along their axis: x, y, z momentum, energy, mass
  double x[5][TY * FW], y[5][(TY + 2 * R) * TX];
};

// NT threads: points of the tile first, then of its rim, NT at a time (small tiles: one point per
// thread, so that the rim's chain of FP64 operations runs beside the tile's).
template <int R, int TX, int TY, int NT>
__global__ void __launch_bounds__(NT, NT >= 256 ? 3 : 1) k_euler2d(Geometry g, Physics ph, StepSched sc,
                                                                   const double* __restrict__ Uin0, double* __restrict__ Uout0,
                                                                   const double* __restrict__ ring, int in_ring, int out_ring,
                                                                   const SubDev* __restrict__ subs, double* __restrict__ Q,
                                                                   int stage, int s, double A, double B, double dt, int first,
                                                                   int last) {
  using S = E2Smem<R, TX, TY>;
  constexpr int FW = S::FW, OWN = TX * TY, NX = 2 * R * TY, NXY = NX + 2 * R * TX;
  constexpr int KO = (OWN + NT - 1) / NT, KP = (OWN + NXY + NT - 1) / NT;
  extern __shared__ __align__(16) unsigned char e2raw[];
  S& sm = *reinterpret_cast<S*>(e2raw);
  const int sid = blockIdx.y, tid = threadIdx.x;
  const SubDev d = subs[sid];
  const int tiles_x = (d.sx + TX - 1) / TX, tile = blockIdx.x;
  const int i0 = (tile % tiles_x) * TX, j0 = (tile / tiles_x) * TY;
  const bool work = d.own && j0 < d.sy;
  // (what does not depend on the previous kernel is above)
  pdl_enter();
  if (!work) return;
  sc = resolve(sc);
  const double* __restrict__ Uin = ring_or(Uin0, in_ring, ring, sc, 0);
  double* __restrict__ Uout = const_cast<double*>(ring_or(Uout0, out_ring, ring, sc, 1));
  const int wa = min(TX, d.sx - i0), ha = min(TY, d.sy - j0);  // the tile's own extent
  const long long N = d.bN;
  const long long g0 = d.bbase + (long long)(d.ox + i0) + (long long)d.bnx * (d.oy + j0);
  auto wrap1 = [](int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); };

  // the state at point (pi, pj) of the sub-domain, up to R beyond it along one axis
  auto load = [&](int pi, int pj, double* u) {
    const int f = pi < 0 ? 0 : (pi >= d.sx ? 1 : (pj < 0 ? 2 : (pj >= d.sy ? 3 : -1)));
    const long long o = d.bbase + (long long)wrap1(d.ox + pi, d.bnx) + (long long)d.bnx * wrap1(d.oy + pj, d.bny);
    if (f < 0 || sc.mode == 0) {
#pragma unroll
      for (int v = 0; v < 5; ++v) u[v] = Uin[o + v * N];
      return;
    }
    // halo point of an asynchronous step: AT weights over the delayed levels, or the latest one
    const int kd = face_delay(sc, sid, f), nR = mod_ring(sc.n, sc.R);
    const long long lvN = 5 * g.N;
    const int C = sc.mode == 2 ? 1 : sc.C;
    double r[CFS_MAX_LEVELS][5];
#pragma unroll
    for (int l = 0; l < CFS_MAX_LEVELS; ++l)
      if (l < C) {
        const int q = nR - kd - l;
        const double* src = ring + (long long)(q < 0 ? q + sc.R : q) * lvN + o;
#pragma unroll
        for (int v = 0; v < 5; ++v) r[l][v] = src[v * N];
      }
    const double* w = sc.W + (kd * s + stage) * sc.C;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      double x = sc.mode == 2 ? r[0][v] : __ldg(w) * r[0][v];
#pragma unroll
      for (int l = 1; l < CFS_MAX_LEVELS; ++l)
        if (l < C) x = fma(__ldg(w + l), r[l][v], x);
      u[v] = x;
    }
  };
  // velocities, p and rho E + p (App. A)
  auto prims = [&](const double* u, double& vx, double& vy, double& p, double& et) {
    const double ir = recip(u[0]);
    vx = u[1] * ir;
    vy = u[2] * ir;
    double k2 = fma(u[2], vy, u[1] * vx);
    if (__double_as_longlong(u[3]) << 1) k2 = fma(u[3], u[3] * ir, k2);
    p = ph.gm1 * fma(-0.5, k2, u[4]);
    et = u[4] + p;
  };

  // ---- the tile's points and its rim: loads first
  // point e of the tile (kind 3) or its rim: the R columns beyond it in x (kind 1), then the R rows
  // beyond it in y (2); 0: none
  auto point = [&](int e, int& pi, int& pj) -> int {
    if (e < OWN) {
      pi = e % TX;
      pj = e / TX;
      return pi < wa && pj < ha ? 3 : 0;
    }
    e -= OWN;
    if (e < NX) {
      const int c = e % (2 * R);
      pj = e / (2 * R);
      pi = c < R ? c - R : wa + c - R;
      return pj < ha ? 1 : 0;
    }
    e -= NX;
    const int r = e / TX;
    pi = e % TX;
    pj = r < R ? r - R : ha + r - R;
    return r < 2 * R && pi < wa ? 2 : 0;
  };
  // (bit patterns: FP64 compares would occupy the FP64 pipe)
  auto nonzero = [](double x) { return (__double_as_longlong(x) << 1) != 0; };
  double u[KP][5];
  bool zm = false;
#pragma unroll
  for (int k = 0; k < KP; ++k) {
    int pi, pj;
    const int kind = point(tid + k * NT, pi, pj);
    if (kind == 3) {
#pragma unroll
      for (int v = 0; v < 5; ++v) u[k][v] = Uin[g0 + pi + (long long)d.bnx * pj + v * N];
    } else if (kind) {
      load(i0 + pi, j0 + pj, u[k]);
    }
    zm = zm || (kind && nonzero(u[k][3]));
  }
  // whether the z momentum is anything but zero on the tile and its rim
  const bool zmom = __syncthreads_or(zm);
  bool bad = false;  // a velocity that is not finite: its product with zero is not zero

#pragma unroll
  for (int k = 0; k < KP; ++k) {
    int pi, pj;
    const int kind = point(tid + k * NT, pi, pj);
    if (!kind) continue;
    const double* w = u[k];
    double vx, vy, p, et;
    prims(w, vx, vy, p, et);
    bad = bad || max(__double2hiint(vx) & 0x7fffffff, __double2hiint(vy) & 0x7fffffff) >= 0x7ff00000;
    const int ox = pj * FW + pi + R, oy = (pj + R) * TX + pi;
    const double uv = w[1] * vy;
    if (kind & 1) {  // fluxes along x: the tile and its columns
      sm.x[0][ox] = fma(w[1], vx, p);
      sm.x[1][ox] = uv;
      if (zmom) sm.x[2][ox] = w[3] * vx;
      sm.x[3][ox] = et * vx;
      sm.x[4][ox] = w[1];
    }
    if (kind & 2) {  // along y: the tile and its rows
      sm.y[0][oy] = uv;
      sm.y[1][oy] = fma(w[2], vy, p);
      if (zmom) sm.y[2][oy] = w[3] * vy;
      sm.y[3][oy] = et * vy;
      sm.y[4][oy] = w[2];
    }
  }
  // the first point's low-storage register in flight over the barrier
  double q[5];
  auto load_q = [&](int k) {
    int pi, pj;
    const int e = tid + k * NT;
    const bool own = e < OWN && point(e, pi, pj) == 3 && !first;
#pragma unroll
    for (int v = 0; v < 5; ++v) q[v] = own ? Q[g0 + pi + (long long)d.bnx * pj + v * N] : 0.0;
  };
  load_q(0);
  bool zflux = zmom;
  if (__syncthreads_or(bad) && !zmom) {
    zflux = true;
#pragma unroll
    for (int k = 0; k < KP; ++k) {
      int pi, pj;
      const int kind = point(tid + k * NT, pi, pj);
      if (!kind) continue;
      double vx, vy, p, et;
      prims(u[k], vx, vy, p, et);
      if (kind & 1) sm.x[2][pj * FW + pi + R] = u[k][3] * vx;
      if (kind & 2) sm.y[2][(pj + R) * TX + pi] = u[k][3] * vy;
    }
    __syncthreads();
  }

  // ---- - dt (D_x F + D_y G) in units of the difference factor, and the low-storage update
  const double cx = R == 2 ? d.c2[0] : d.c1[0], cy = R == 2 ? d.c2[1] : d.c1[1];
  const bool iso = __double_as_longlong(cx) == __double_as_longlong(cy);
  const double kx = -dt * cx, ky = iso ? kx : -dt * cy;
  auto diff = [&](const double* f, int o, int st) {
    const double d1 = f[o + st] - f[o - st];
    return R == 2 ? fma(-8.0, d1, f[o + 2 * st] - f[o - 2 * st]) : d1;
  };
#pragma unroll
  for (int k = 0; k < KO; ++k) {
    int pi, pj;
    if (k > 0) load_q(k);
    if (tid + k * NT >= OWN || point(tid + k * NT, pi, pj) != 3) continue;
    const int ox = pj * FW + pi + R, oy = (pj + R) * TX + pi;
    const long long gi = g0 + pi + (long long)d.bnx * pj;
    auto update = [&](int v, int comp) {
      const double dx = diff(sm.x[comp], ox, 1), dy = diff(sm.y[comp], oy, TX);
      double qn = first ? 0.0 : A * q[v];
      if (iso) qn = fma(kx, dx + dy, qn);
      else qn = fma(ky, dy, fma(kx, dx, qn));
      if (!last) Q[gi + v * N] = qn;
      Uout[gi + v * N] = fma(B, qn, u[k][v]);
    };
    update(0, 4);
    update(1, 0);
    update(2, 1);
    if (zflux || nonzero(q[3])) {
      if (!zflux) {
        const double qn = A * q[3];
        if (!last) Q[gi + 3 * N] = qn;
        Uout[gi + 3 * N] = fma(B, qn, u[k][3]);
      } else {
        update(3, 2);
      }
    } else {
      if (!last) Q[gi + 3 * N] = 0.0;
      Uout[gi + 3 * N] = u[k][3];
    }
    update(4, 3);
  }
}

namespace {

// The tile shapes: large grids 32 x 16 points on 256 threads (a rim of a fifth of the tile at R = 1),
// small ones 8 x 8 on 128 threads, half of them on the rim.  The small tile's rim costs as much as
// the tile (at R = 2 twice as much), but on a small grid the FP64 pipes of 152 SMs are idle and what
// counts is how many SMs and warps a stage spreads over: 64 x 64 points take 64 CTAs instead of 8.
// A step with large / small tiles, us (square grids, sub-domains of 64 x 64):
//          64^2         128^2        192^2        256^2         320^2        384^2        512^2
//   R = 2  69.7 / 26.7  69.7 / 38.9  71.7 / 45.1  92.3 / 82.9  147.5 / 119   170 / 158    236 / 265
//   R = 1  24.7 / 12.4  24.7 / 14.4  25.8 / 18.5  26.7 / 30.8  41.0 / 45.1   49.2 / 57.4  75.6 / 96.3
// so the line lies between 384^2 and 512^2 (2304 and 4096 small tiles), and between 192^2 and 240^2
// (576 and 1024).
//
// A row of a large tile is a warp, so sub-domains whose width is not near a multiple of 32 leave lanes idle, and
// the kernels of kernels.cu, three launches over the points of a sub-domain in a row, are faster.  A step,
// us, three launches / large tiles, by the part of the lanes that have a point:
//          33 wide: 0.52      40: 0.63    48: 0.75      60: 0.94   64: 1
//   R = 2  1097 / 1724        293 / 382   1310 / 1411              881 / 758
//   R = 1  361 / 576          99 / 129    439 / 459                348 / 303
// (1056^2, 520^2, 1200^2, 1024^2 points).  The line is 0.8; below it small tiles are compared with the three
// launches: 330^2 in 100 sub-domains (2500 tiles) 168 against 200 and 62 against 60.
constexpr long long small_tiles(int r, bool full) { return r == 1 ? 152 * (full ? 4 : 16) : 152 * 18; }

template <int R, int TX, int TY, int NT>
int launch_tile(const Geometry& g, const Physics& ph, const StepSched& sc, const StageLaunch& a, int tiles, cudaStream_t st) {
  using S = E2Smem<R, TX, TY>;
  // the shared-memory opt-in is a per-device attribute of the kernel
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return (int)e;
  if (dev < 0 || dev >= 64) return (int)cudaErrorInvalidDevice;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (!done[dev]) {
      e = cudaFuncSetAttribute(k_euler2d<R, TX, TY, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(S));
      if (e != cudaSuccess) return (int)e;
      done[dev] = true;
    }
  }
  launch_pdl(k_euler2d<R, TX, TY, NT>, dim3(tiles, g.nsub), dim3(NT), sizeof(S), st, g, ph, sc, a.Uin, a.Uout, a.ring,
             a.in_ring, a.out_ring, a.subs, a.Q, a.stage, a.s, a.A, a.B, a.dt, a.first, a.last);
  return (int)cudaGetLastError();
}

int tiles_of(int sx, int sy, int tx, int ty) { return ((sx + tx - 1) / tx) * ((sy + ty - 1) / ty); }

}  // namespace

Euler2dShape euler2d_shape(const SubDev* subs, int nsub, int r) {
  Euler2dShape e{0, 0};
  long long small = 0, points = 0, lanes = 0;
  int most_small = 0, most_large = 0;
  for (int i = 0; i < nsub; ++i) {
    const int t = tiles_of(subs[i].sx, subs[i].sy, 8, 8);
    small += t;
    points += (long long)subs[i].sx * subs[i].sy;
    lanes += (long long)((subs[i].sx + 31) / 32) * 32 * subs[i].sy;
    most_small = std::max(most_small, t);
    most_large = std::max(most_large, tiles_of(subs[i].sx, subs[i].sy, 32, 16));
  }
  const bool full = 10 * points >= 8 * lanes;
  e.small = small <= small_tiles(r, full);
  e.tiles = e.small ? most_small : (full ? most_large : 0);
  return e;
}

int launch_euler2d(const Geometry& g, const Physics& ph, const StepSched& sc, const StageLaunch& a, Euler2dShape e,
                   void* stream, long long* launches, const Timer* tm) {
  const cudaStream_t st = (cudaStream_t)stream;
  int rc;
  TIMED(tm, 2, (rc = e.small ? (g.r == 2 ? launch_tile<2, 8, 8, 128>(g, ph, sc, a, e.tiles, st)
                                         : launch_tile<1, 8, 8, 128>(g, ph, sc, a, e.tiles, st))
                             : (g.r == 2 ? launch_tile<2, 32, 16, 256>(g, ph, sc, a, e.tiles, st)
                                         : launch_tile<1, 32, 16, 256>(g, ph, sc, a, e.tiles, st))));
  if (launches) *launches += 1;
  return rc;
}

}  // namespace cfs

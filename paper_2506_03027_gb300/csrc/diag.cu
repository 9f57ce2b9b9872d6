// diag.cu -- diagnostics of a state: kinetic energy, enstrophy, totals and the non-finite flag.
//
// Per block of points one CTA (256 points at a time, or, where that is faster, a tile of 32 x 8 columns marching
// through a chunk of z planes) writes one row of partial sums; a last CTA adds the rows in a fixed order.  In FP64 the sums are bound by
// the FP64 pipe: a reciprocal of the density and six differences per point are about 110 FP64
// operations at 2 per clock and SM.  Only the five totals need FP64 accumulation point by point; the
// velocities, their differences and the two squares are formed on pairs of floats (pairs.cuh), a
// column's few values per chunk added as pairs and the columns in FP64.  A 128^3 state: 1.52 ms per
// call (one thread per point, FP64) -> 0.16 ms, of which the tile kernel takes 113 us at about the
// rate the pairs' instructions issue (the state's 84 MB take 12) and the last CTA 11.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "cfs_internal.h"
#include "device_common.cuh"
#include "pairs.cuh"

namespace cfs {

namespace {

constexpr int DTX = 32, DTY = 8;

// The five totals, the kinetic energy (x 2) and the enstrophy (x 2, and the volume it covers) of one
// point in FP64: any block (curvilinear, two-dimensional, not periodic, partitioned), any finite or
// non-finite value.
template <bool CURV>
__device__ __forceinline__ void diag_point(const DiagBlock& b, const double* __restrict__ U, int x, int y, int z, double* acc) {
  const int ndim = b.nz > 1 ? 3 : 2;
  const long long i = (long long)x + (long long)b.nx * ((long long)y + (long long)b.ny * z);
  const long long mq = (long long)(x + b.G) + (long long)b.mx * (y + b.G);  // metric plane index
  const double dV = CURV ? b.M[5 * b.mpl + mq] : b.dV;  // cell volume (J^-1 on a curvilinear grid)
  double u[5];
  for (int v = 0; v < 5; ++v) {
    u[v] = U[b.bbase + v * b.bN + i];
    if (!isfinite(u[v])) acc[7] = 1.0;
    acc[2 + v] += u[v] * dV;
  }
  const double rho = u[0], ir = recip(rho);
  acc[0] += 0.5 * ir * (u[1] * u[1] + u[2] * u[2] + u[3] * u[3]) * dV;
  // enstrophy only where the CD stencils stay in the block or cross periodic faces
  if (b.nonper) {
    const int c3[3] = {x, y, z}, n3[3] = {b.nx, b.ny, b.nz};
    for (int a = 0; a < ndim; ++a) {
      if (((b.nonper >> (2 * a)) & 1) && c3[a] < b.rs) return;
      if (((b.nonper >> (2 * a + 1)) & 1) && c3[a] > n3[a] - 1 - b.rs) return;
    }
  }
  acc[8] += dV;
  // velocity differences by the CD scheme, one reciprocal of the density per stencil point
  double dv[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
  const bool far = b.c2[0] != 0.0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (a >= ndim) continue;
    // the axis's four (CD2: two) stencil points, all loads before the first division
    const int n = a == 0 ? b.nx : (a == 1 ? b.ny : b.nz), c0 = a == 0 ? x : (a == 1 ? y : z);
    const long long st = a == 0 ? 1 : (a == 1 ? (long long)b.nx : (long long)b.nx * b.ny);
    double q[4][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int o = k < 2 ? 2 * k - 1 : 4 * k - 10;  // -1, 1, -2, 2
      if (k >= 2 && !far) continue;
      const double* src = U + b.bbase + i + (long long)(wrapc(c0 + o, n) - c0) * st;
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (CURV || c != 1 + a) q[k][c] = src[c * b.bN];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (k >= 2 && !far) continue;
      const double w = ((k & 1) ? recip(q[k][0]) : -recip(q[k][0])) * (k < 2 ? b.c1[a] : b.c2[a]);
#pragma unroll
      for (int c = 0; c < 3; ++c)
        if (CURV || c != a) dv[c][a] = fma(w, q[k][1 + c], dv[c][a]);  // (the vorticity takes c != a)
    }
  }
  if (CURV) {  // index-space derivatives -> physical: d/dx_j = J sum_k (metric row k)_j d/dxi_k
    const double J = b.M[6 * b.mpl + mq];
    const double m[3][3] = {{b.M[mq], b.M[b.mpl + mq], 0.0}, {b.M[2 * b.mpl + mq], b.M[3 * b.mpl + mq], 0.0},
                            {0.0, 0.0, b.M[4 * b.mpl + mq]}};
    double dp[3][3];
    for (int c = 0; c < 3; ++c)
      for (int j = 0; j < 3; ++j) dp[c][j] = J * (m[0][j] * dv[c][0] + m[1][j] * dv[c][1] + m[2][j] * dv[c][2]);
    for (int c = 0; c < 3; ++c)
      for (int j = 0; j < 3; ++j) dv[c][j] = dp[c][j];
  }
  const double wx = dv[2][1] - dv[1][2], wy = dv[0][2] - dv[2][0], wz = dv[1][0] - dv[0][1];
  acc[1] += 0.5 * rho * (wx * wx + wy * wy + wz * wz) * dV;
}

// The column of a marching CTA that cannot use the pairs (rare: out of line, so that the march keeps its registers)
__device__ __noinline__ void diag_column(const DiagBlock& b, const double* __restrict__ U, int x, int y, int z0, int z1, double* acc) {
  for (int z = z0; z < z1; ++z) diag_point<false>(b, U, x, y, z, acc);
}

// acc of 256 threads -> one row: through shared memory, a warp per quantity (each lane eight threads'
// values, then a shuffle tree): a third of the FP64 additions of a tree per warp and quantity.
// buf: DIAG_NQ x 256 doubles.
__device__ __forceinline__ void diag_row(const double* acc, double* __restrict__ row, double* buf) {
  const int tid = threadIdx.x + blockDim.x * threadIdx.y, lane = tid & 31, wid = tid >> 5;
  __syncthreads();  // (buf may hold what the march read)
#pragma unroll
  for (int c = 0; c < DIAG_NQ; ++c) buf[c * 256 + tid] = acc[c];
  __syncthreads();
  for (int c = wid; c < DIAG_NQ; c += 8) {
    double v = buf[c * 256 + lane];
#pragma unroll
    for (int k = 1; k < 8; ++k) {
      const double o = buf[c * 256 + lane + 32 * k];
      v = (c == 7) ? fmax(v, o) : v + o;
    }
    for (int o = 16; o > 0; o >>= 1) {
      const double other = __shfl_down_sync(0xffffffffu, v, o);
      v = (c == 7) ? fmax(v, other) : v + other;
    }
    if (lane == 0) row[c] = v;
  }
}

template <bool CURV>
__global__ void __launch_bounds__(256) k_diag(DiagBlock b, const double* __restrict__ U, double* __restrict__ partial) {
  double acc[DIAG_NQ] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < b.bN; i += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(i % b.nx), y = (int)((i / b.nx) % b.ny), z = (int)(i / ((long long)b.nx * b.ny));
    if (b.subs && !b.subs[b.sid0 + b.owner[0][x] + b.P[0] * (b.owner[1][y] + b.P[1] * b.owner[2][z])].own) continue;
    diag_point<CURV>(b, U, x, y, z, acc);
  }
  __shared__ double buf[DIAG_NQ * 256];
  diag_row(acc, partial + (long long)blockIdx.x * DIAG_NQ, buf);
}

// One differenced pair of values from points -2, -1, 1, 2 (or -1, 1), without its factor.
template <int R, class V>
__device__ __forceinline__ Pr<V> diff_pts(Pr<V> m2, Pr<V> m1, Pr<V> p1, Pr<V> p2) {
  if (R == 1) return p_norm(p_sub(p1, m1));
  const V m8 = v_bc<V>(-8.f);
  const Pr<V> x = p_2diff(p2.h, m2.h), y = p_2diff(p1.h, m1.h);
  const Pr<V> s = p_2sum(x.h, v_mul(m8, y.h));
  const V lo = v_add(v_fma(m8, y.l, x.l), v_fma(m8, v_sub(p1.l, m1.l), v_sub(p2.l, m2.l)));
  return p_norm(Pr<V>{s.h, v_add(s.l, lo)});
}

// Cartesian 3-D block: a CTA marches its tile of columns through planes [z0, z1).  Per plane the
// velocities of the tile and of R points beyond it in x and y go to one of four shared-memory planes
// (one barrier per plane), the column's own (u, v) stay in registers for the z differences; plane
// L - R is finished when plane L has arrived.  A CTA takes its points in FP64 instead when it meets a value
// outside the pairs' range (a density, a momentum; also NaN and infinity), when what it forms from
// them leaves that range (a sum of squares of 2^100 and more), and when the largest sum of squares of its
// columns is below 2^-60 but not zero, so that the squares' low words may be lost.
template <int R>
__global__ void __launch_bounds__(DTX * DTY, 3) k_diag_tile(DiagBlock b, const double* __restrict__ U, double* __restrict__ partial,
                                                         int tiles_x, int tiles, int zc, int rows) {
  if ((int)blockIdx.x >= rows) {  // beyond the block's work: a row of zeros
    const int t = threadIdx.x + DTX * threadIdx.y;
    if (t < DIAG_NQ) partial[(long long)blockIdx.x * DIAG_NQ + t] = 0.0;
    return;
  }
  constexpr int BX = DTX + 2 * R, BY = DTY + 2 * R, XS = BX + 1;
  __shared__ float4 sUV[4][BY * XS];
  __shared__ float2 sW[4][BY * XS];
  const int tx = threadIdx.x, ty = threadIdx.y, tid = tx + DTX * ty;
  const int tile = blockIdx.x % tiles, chunk = blockIdx.x / tiles;
  const int x0 = (tile % tiles_x) * DTX, y0 = (tile / tiles_x) * DTY, z0 = chunk * zc, z1 = min(b.nz, z0 + zc);
  const int x = x0 + tx, y = y0 + ty;
  const bool own = x < b.nx && y < b.ny;
  const long long plane = (long long)b.nx * b.ny;
  const double* __restrict__ base = U + b.bbase;
  const long long col = (long long)wrapc(x, b.nx) + (long long)b.nx * wrapc(y, b.ny);
  // a second point: the R columns beyond the tile in x, the R rows beyond it in y
  constexpr int NX = 2 * R * DTY, NXY = NX + 2 * R * DTX;
  int hx = 0, hy = 0;
  if (tid < NX) {
    const int c = tid % (2 * R);
    hx = c < R ? c - R : DTX + c - R;
    hy = tid / (2 * R);
  } else if (tid < NXY) {
    const int r = (tid - NX) / DTX;
    hx = (tid - NX) % DTX;
    hy = r < R ? r - R : DTY + r - R;
  }
  const long long hcol = (long long)wrapc(x0 + hx, b.nx) + (long long)b.nx * wrapc(y0 + hy, b.ny);
  const int so = (ty + R) * XS + tx + R, sh = (hy + R) * XS + hx + R;
  bool bad = false;
  auto outside = [](double v, int lo) {  // |v| >= 2^60, or below 2^(lo - 1023) (lo > 0)
    const int e = (__double2hiint(v) >> 20) & 0x7ff;
    return e >= 1023 + 60 || e < lo;
  };
  double acc[DIAG_NQ] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  P2 uv[2 * R + 1];     // (u, v) of the column, planes L - 2R .. L
  P1 rh[R + 1];         // density, planes L - R .. L
  P1 kin = {0.f, 0.f}, ens = {0.f, 0.f};
  const P1 cx = {b.cg[0].x, b.cg[0].y}, cy = {b.cg[1].x, b.cg[1].y}, cz = {b.cg[2].x, b.cg[2].y};
#pragma unroll
  for (int k = 0; k <= 2 * R; ++k) uv[k] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
  for (int k = 0; k <= R; ++k) rh[k] = {0.f, 0.f};
  int nens = 0;
  unsigned moving = 0;  // bits of the column's momenta, without the sign
  for (int L = z0 - R; L < z1 + R; ++L) {
    const bool inner = L >= z0 && L < z1;
    const double* __restrict__ pl = base + plane * wrapc(L, b.nz);
    double u[5], hu[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) u[v] = pl[v * b.bN + col];
    if (inner) {
      u[4] = pl[4 * b.bN + col];
      if (tid < NXY) {
#pragma unroll
        for (int v = 0; v < 4; ++v) hu[v] = pl[v * b.bN + hcol];
      }
    }
#pragma unroll
    for (int k = 0; k < 2 * R; ++k) uv[k] = uv[k + 1];
#pragma unroll
    for (int k = 0; k < R; ++k) rh[k] = rh[k + 1];
    bad = bad || outside(u[0], 1023 - 60) || outside(u[1], 0) || outside(u[2], 0) || outside(u[3], 0);
    const P1 rho = p_split(u[0]), ir = p_recip(rho);
    const P2 mxy = p_pair(p_split(u[1]), p_split(u[2]));
    uv[2 * R] = p_norm(p_mul(mxy, p_bc(ir)));
    rh[R] = rho;
    if (inner) {
      const P1 mz = p_split(u[3]), w = p_norm(p_mul(mz, ir));
      sUV[L & 3][so] = p_store(uv[2 * R]);
      sW[L & 3][so] = p_store(w);
      if (tid < NXY) {
        bad = bad || outside(hu[0], 1023 - 60) || outside(hu[1], 0) || outside(hu[2], 0) || outside(hu[3], 0);
        const P1 hi = p_recip(p_split(hu[0]));
        sUV[L & 3][sh] = p_store(p_norm(p_mul(p_pair(p_split(hu[1]), p_split(hu[2])), p_bc(hi))));
        sW[L & 3][sh] = p_store(p_norm(p_mul(p_split(hu[3]), hi)));
      }
      if (own) {
#pragma unroll
        for (int v = 0; v < 5; ++v) acc[2 + v] += u[v];
        bad = bad || outside(u[4], 0);
#pragma unroll
        for (int v = 1; v < 4; ++v) moving |= (unsigned)(__double2hiint(u[v]) << 1) | (unsigned)__double2loint(u[v]);
        const P2 k2 = p_mul(mxy, uv[2 * R]);
        kin = p_norm(p_add(kin, p_norm(p_fma(mz, w, p_add(p_x(k2), p_y(k2))))));
      }
    }
    __syncthreads();
    const int z = L - R;
    if (z < z0 || !own) continue;
    if (b.nonper) {
      const int c3[3] = {x, y, z}, n3[3] = {b.nx, b.ny, b.nz};
      bool in = true;
#pragma unroll
      for (int a = 0; a < 3; ++a)
        in = in && !(((b.nonper >> (2 * a)) & 1) && c3[a] < R) && !(((b.nonper >> (2 * a + 1)) & 1) && c3[a] > n3[a] - 1 - R);
      if (!in) continue;
    }
    ++nens;
    const float4* A = sUV[z & 3] + so;
    const float2* W = sW[z & 3] + so;
    auto vw = [&](int o) { const float4 t = A[o]; const float2 w = W[o]; return P2{make_float2(t.y, w.x), make_float2(t.w, w.y)}; };
    auto uw = [&](int o) { const float4 t = A[o]; const float2 w = W[o]; return P2{make_float2(t.x, w.x), make_float2(t.z, w.y)}; };
    constexpr int T = R == 2 ? 2 : 1;
    const P2 dx = p_mul(p_bc(cx), diff_pts<R>(vw(-T), vw(-1), vw(1), vw(T)));                          // d(v, w)/dx
    const P2 dy = p_mul(p_bc(cy), diff_pts<R>(uw(-T * XS), uw(-XS), uw(XS), uw(T * XS)));              // d(u, w)/dy
    const P2 dz = p_mul(p_bc(cz), diff_pts<R>(uv[0], uv[R - 1], uv[R + 1], uv[2 * R]));                // d(u, v)/dz
    const P2 a = p_norm(p_sub(p_pair(p_y(dy), p_x(dz)), p_pair(p_y(dz), p_y(dx))));                    // w_x, w_y
    const P1 c = p_norm(p_sub(p_x(dx), p_x(dy)));                                                      // w_z
    const P2 a2 = p_mul(a, a);
    const P1 w2 = p_norm(p_fma(c, c, p_add(p_x(a2), p_y(a2))));
    ens = p_norm(p_add(ens, p_norm(p_mul(rh[0], w2))));
  }
  bad = bad || !(kin.h < 0x1p100f) || !(ens.h < 0x1p100f);
  const bool lost = (!__syncthreads_or(kin.h >= 0x1p-60f) && __syncthreads_or(moving != 0)) ||
                    (!__syncthreads_or(ens.h >= 0x1p-60f) && __syncthreads_or(ens.h != 0.f));
  if (__syncthreads_or(bad) || lost) {
    for (int c = 0; c < DIAG_NQ; ++c) acc[c] = 0.0;
    if (own) diag_column(b, U, x, y, z0, z1, acc);
  } else {
#pragma unroll
    for (int v = 0; v < 5; ++v) acc[2 + v] *= b.dV;
    acc[0] = 0.5 * b.dV * ((double)kin.h + (double)kin.l);
    acc[1] = 0.5 * b.dV * ((double)ens.h + (double)ens.l);
    acc[8] = nens * b.dV;
  }
  static_assert(sizeof(sUV) >= sizeof(double) * DIAG_NQ * 256, "the reduction reuses the planes");
  diag_row(acc, partial + (long long)blockIdx.x * DIAG_NQ, reinterpret_cast<double*>(&sUV[0][0]));
}

// The rows in a fixed order, a warp per quantity: lane l adds rows l, l + 32, ..., the lanes combine
// in a fixed tree.  K is a volume average (sum of value x cell volume over the total volume), the
// enstrophy an average over the volume of the points it covers.
__global__ void __launch_bounds__(32 * DIAG_NQ) k_diag_final(const double* __restrict__ partial, int nrows,
                                                            double* __restrict__ out, double volume) {
  __shared__ double tot[DIAG_NQ];
  const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double v = 0.0;
#pragma unroll 8
  for (int r = lane; r < nrows; r += 32) {
    const double x = partial[(long long)r * DIAG_NQ + c];
    v = (c == 7) ? fmax(v, x) : v + x;
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double other = __shfl_down_sync(0xffffffffu, v, o);
    v = (c == 7) ? fmax(v, other) : v + other;
  }
  if (lane == 0) tot[c] = v;
  __syncthreads();
  if (threadIdx.x >= 8) return;
  const int q = threadIdx.x;
  double r = tot[q];
  if (q == 0) r /= volume;
  if (q == 1) r = tot[8] > 0.0 ? r / tot[8] : 0.0;
  out[q] = r;
}

struct TileShape {
  int tiles_x, tiles, zc;
  long long rows;
};

// Planes per CTA: the chunk count that takes the least time, waves of 3 CTAs on 152 SMs times the
// planes a CTA marches (its own and four beyond), a last wave that is nearly empty included.
TileShape tile_shape(int nx, int ny, int nz) {
  TileShape s;
  s.tiles_x = (nx + DTX - 1) / DTX;
  const long long t = (long long)s.tiles_x * ((ny + DTY - 1) / DTY);
  s.tiles = (int)std::min<long long>(t, 1 << 30);
  s.zc = nz;
  long long best = -1;
  for (int c = 1; c <= std::min(nz, 64); ++c) {
    const int zc = (nz + c - 1) / c;
    const long long rows = t * ((nz + zc - 1) / zc), cost = ((rows + 455) / 456) * (zc + 4);
    if (best < 0 || cost < best) {
      best = cost;
      s.zc = zc;
    }
  }
  s.rows = t * ((nz + s.zc - 1) / s.zc);
  return s;
}

// CTAs of the kernel by points: one per 256 points up to eight per SM.  (No more than have work: the first CTAs of
// a larger grid share SMs.  32^3 points in 304 CTAs: 41 us, in 128: 21.)
int point_rows(int nx, int ny, int nz) { return (int)std::min<long long>(((long long)nx * ny * nz + 255) / 256, 8 * 152); }

// Whether a block's shape suits the marching kernel.  us it takes: per wave of 456 CTAs and plane 1.4 (the
// latency of a plane) and up to 3.5 more as the SMs fill; the kernel by points 7.7 per 152 CTAs of 256 points.
// Slender blocks leave most of a tile's columns or of the SMs without work, small ones are one
// wave of either.  us per call, marching / by points: 4 x 4 x 16384 364 / 83, 8 x 8 x 4096 130 / 83,
// 2 x 1024^2 952 / 421, 32^3 25 / 21, 12^2 x 2000 97 / 73, 20^2 x 800 54 / 80, 64^3 35 / 66, 256^3 800 / 3300.
bool march(int nx, int ny, int nz, const TileShape& s) {
  const double waves = (double)((s.rows + 455) / 456), fill = std::min(1.0, s.rows / 456.0);
  const long long ctas = ((long long)nx * ny * nz + 255) / 256;
  return nz > 1 && waves * (s.zc + 4) * (1.4 + 3.5 * fill) < 7.7 * (double)((ctas + 151) / 152);
}

// the marching kernel: 3-D Cartesian blocks computed here as a whole, of spacings within the pairs' range
bool tiled(const DiagBlock& b, const TileShape& s) {
  if (b.M || b.subs || !march(b.nx, b.ny, b.nz, s)) return false;
  for (int a = 0; a < 3; ++a)
    if (!(std::fabs(b.c1[a]) > 1e-12 && std::fabs(b.c1[a]) < 1e12)) return false;
  return true;
}

}  // namespace

int diag_rows(int nx, int ny, int nz, int most) {
  const TileShape s = tile_shape(nx, ny, nz);
  return march(nx, ny, nz, s) && s.rows <= most ? (int)s.rows : point_rows(nx, ny, nz);
}

int launch_diagnostics_block(const DiagBlock& b, const double* U, double* partial, int row0, int rows, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  double* p = partial + (long long)row0 * DIAG_NQ;
  const TileShape s = tile_shape(b.nx, b.ny, b.nz);
  if (tiled(b, s) && s.rows <= rows) {
    if (b.rs == 2) k_diag_tile<2><<<rows, dim3(DTX, DTY), 0, st>>>(b, U, p, s.tiles_x, s.tiles, s.zc, (int)s.rows);
    else k_diag_tile<1><<<rows, dim3(DTX, DTY), 0, st>>>(b, U, p, s.tiles_x, s.tiles, s.zc, (int)s.rows);
  } else {
    (b.M ? k_diag<true> : k_diag<false>)<<<rows, 256, 0, st>>>(b, U, p);
  }
  return (int)cudaGetLastError();
}

int launch_diagnostics_final(const double* partial, int nrows, double* out, double volume, void* stream) {
  k_diag_final<<<1, 32 * DIAG_NQ, 0, (cudaStream_t)stream>>>(partial, nrows, out, volume);
  return (int)cudaGetLastError();
}

}  // namespace cfs

// launch_common.cuh -- launch helpers and device code shared by the stage kernels (kernels.cu,
// stage_pairs.cu).
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "cfs_internal.h"
#include "device_common.cuh"

namespace cfs {

// Programmatic dependent launch: the kernels of the FP64 stage sequence (view, flux, stage update,
// filter passes, step counter) are launched with programmatic stream serialization, so the next
// kernel's CTAs are scheduled while this one drains.  Every such kernel first lets its successor
// launch, then waits for its predecessor to complete (and its memory to be visible) before it
// reads anything the predecessor wrote; launched without the attribute both are no-ops.
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
}

template <typename... KArgs, typename... Args>
static inline void launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// Flux points of a sub-domain, in warp-uniform groups: first the owned points (x fastest), then
// the strips of 2r points beyond each face where only the flux along that axis is needed (x
// strips: the 2r columns fastest, then y and z; y strips: x fastest; z strips: x fastest).  A warp
// of strip points evaluates one flux direction and only the gradients it needs.
template <int ND>
__device__ __forceinline__ bool flux_point(const SubDev& d, int r, int t, int& ci, int& cj, int& ck, int& kind) {
  const int sxy = d.sx * d.sy, nown = sxy * d.sz;
  if (t < nown) {
    ck = t / sxy;
    const int r2 = t - ck * sxy;
    cj = r2 / d.sx;
    ci = r2 - cj * d.sx;
    kind = 0;
    return true;
  }
  t -= nown;
  const int w = 2 * r;
  const int nx = w * d.sy * d.sz;
  if (t < nx) {  // x strips
    const int s = t % w, rest = t / w;
    cj = rest % d.sy;
    ck = rest / d.sy;
    ci = s < r ? s - r : d.sx + s - r;
    kind = 1;
    return true;
  }
  t -= nx;
  const int ny = w * d.sx * d.sz;
  if (t < ny) {  // y strips
    ci = t % d.sx;
    const int rest = t / d.sx, s = rest % w;
    ck = rest / w;
    cj = s < r ? s - r : d.sy + s - r;
    kind = 2;
    return true;
  }
  t -= ny;
  if (ND == 3 && t < w * sxy) {  // z strips
    ci = t % d.sx;
    const int rest = t / d.sx;
    cj = rest % d.sy;
    const int s = rest / d.sy;
    ck = s < r ? s - r : d.sz + s - r;
    kind = 3;
    return true;
  }
  return false;
}

static inline unsigned nblk(long long n, int b) { return (unsigned)((n + b - 1) / b); }

#define TIMED(tm, kind, launch)              \
  do {                                       \
    if (tm) tm->rec(tm->self, kind, 1);      \
    launch;                                  \
    if (tm) tm->rec(tm->self, kind, 0);      \
  } while (0)


// x^a = exp(a ln x) in FP64 for positive normal x (the viscosity law mu = T^a), table-driven
// after Tang (ACM TOMS 1989, 1990), about 20 FP64 operations.  ln x: x = m 2^e with m in [1, 2)
// from the bit fields; the top six mantissa bits pick c_j = 1 + (j + 1/2)/64, u = m / c_j - 1
// (|u| <= 1/129) from a table of 1/c_j, ln m = ln c_j + log1p(u) with the series of log1p to u^7.
// exp y: y = (64 k' + j') ln2/64 + r with |r| <= ln2/128 (ln 2 / 64 split into a 32-bit head and
// its tail: k ln2_head is exact), exp r by its Taylor series to r^5/5!, times the tabulated
// 2^(j'/64), and 2^k' added to the exponent field.  Tables: 1/c_j rounded from the exact
// quotient, ln c_j and 2^(j/64) rounded from long-double log1p and exp2 (pow_tables_init).
// Relative error below 6e-16 (1 + |a ln x|).  Any other x, or |a ln x| >= 700, goes to the
// library's pow.
// tab: the device copy of the three tables.
__device__ __forceinline__ double pow_tab(double x, double a, const double* __restrict__ tab) {
  if (!(x >= 2.2250738585072014e-308) || !(x <= 1.7976931348623157e308)) return pow(x, a);
  const int hi = __double2hiint(x);
  const int e = ((hi >> 20) & 0x7ff) - 1023;
  const int j = (hi >> 14) & 63;
  const double m = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(x));  // [1, 2)
  const double u = fma(m, __ldg(tab + j), -1.0);
  double p = 1.0 / 7.0;
  p = fma(p, u, -1.0 / 6.0);
  p = fma(p, u, 1.0 / 5.0);
  p = fma(p, u, -1.0 / 4.0);
  p = fma(p, u, 1.0 / 3.0);
  p = fma(p, u, -0.5);
  p = fma(p, u, 1.0);
  const double l1p = p * u;
  const double LN2_HEAD = 0.6931471803691238, LN2_TAIL = 1.9082149292705877e-10;
  const double ed = (double)e;
  // (e ln2_head + ln c_j) is exact where it cancels (x just below 1: Sterbenz), then the tails
  const double y = a * (fma(ed, LN2_HEAD, __ldg(tab + 64 + j)) + fma(ed, LN2_TAIL, l1p));
  if (!(fabs(y) < 700.0)) return pow(x, a);
  const double kd = rint(y * (64.0 / 0.6931471805599453));
  double r = fma(-kd, LN2_HEAD / 64.0, y);
  r = fma(-kd, LN2_TAIL / 64.0, r);
  double q = 1.0 / 120.0;
  q = fma(q, r, 1.0 / 24.0);
  q = fma(q, r, 1.0 / 6.0);
  q = fma(q, r, 0.5);
  q = fma(q, r, 1.0);
  q = fma(q, r, 1.0);
  const int k = (int)kd;
  q *= __ldg(tab + 128 + (k & 63));
  return __hiloint2double(__double2hiint(q) + ((k >> 6) << 20), __double2loint(q));
}

}  // namespace cfs

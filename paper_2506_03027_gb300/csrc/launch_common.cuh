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

}  // namespace cfs

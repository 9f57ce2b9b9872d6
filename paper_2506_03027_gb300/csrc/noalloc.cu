// noalloc.cu -- cfs_diagnostics_static: the diagnostics reduction for callers that must not
// allocate device memory.
//
// Some callers cannot call cudaMalloc: an in-situ monitoring hook running inside a larger
// simulation whose own pool allocator already owns the GPU's memory, or a time-critical loop in
// which an allocation (which may synchronise the device) is not allowed.  This entry point
// computes the same quantities as cfs_diagnostics on a state the caller holds in device memory,
// with its only scratch (the per-block partial sums) in a fixed array compiled into the library.
#include <cuda_runtime.h>

#include <cstdio>
#include <mutex>

#include "cfs.h"
#include "device_common.cuh"

namespace {

// The rows of partial sums fit 4 MiB.  Every GPU that loads the library keeps this array until exit.
constexpr int kMaxRows = CFS_DIAG_STATIC_MAX_POINTS / 256 * 8 / DIAG_NQ;
constexpr int kMaxDevices = 64;

__device__ __align__(256) double g_partials[(long long)kMaxRows * DIAG_NQ];

std::mutex g_mu;
double* g_dev_ptr[kMaxDevices] = {nullptr};

void put(char* err, size_t len, const char* msg) {
  if (err && len) std::snprintf(err, len, "%s", msg);
}

}  // namespace

extern "C" cfs_status cfs_diagnostics_static(const double* U, int nx, int ny, int nz, const double* spacing, int order,
                                             double* out, void* cuda_stream, char* err, size_t err_len) {
  if (!U || !out || !spacing) {
    put(err, err_len, "cfs_diagnostics_static: null pointer");
    return CFS_EINVAL;
  }
  if (nx < 1 || ny < 1 || nz < 1 || (order != 2 && order != 4)) {
    put(err, err_len, "cfs_diagnostics_static: bad grid size or order");
    return CFS_EINVAL;
  }
  const long long N = (long long)nx * ny * nz;
  if (N > CFS_DIAG_STATIC_MAX_POINTS) {
    char msg[160];
    std::snprintf(msg, sizeof(msg),
                  "cfs_diagnostics_static: %lld points exceed the static scratch limit of %lld points",
                  N, (long long)CFS_DIAG_STATIC_MAX_POINTS);
    put(err, err_len, msg);
    return CFS_EINVAL;
  }
  for (int a = 0; a < 3; ++a)
    if (!(spacing[a] > 0.0)) {
      put(err, err_len, "cfs_diagnostics_static: spacing must be positive");
      return CFS_EINVAL;
    }
  // Set-up, once per device: the array's name is only a host-side stand-in, so look up its
  // device address with that device current.
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    put(err, err_len, "cfs_diagnostics_static: no usable CUDA device");
    return CFS_ECUDA;
  }
  double* partials = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_dev_ptr[dev]) {
      e = cudaGetSymbolAddress((void**)&g_dev_ptr[dev], g_partials);
      if (e != cudaSuccess) {
        g_dev_ptr[dev] = nullptr;
        put(err, err_len, cudaGetErrorString(e));
        return CFS_ECUDA;
      }
    }
    partials = g_dev_ptr[dev];
  }
  cfs::DiagBlock b{};
  b.nx = nx; b.ny = ny; b.nz = nz; b.bN = N;
  const double a = order == 4 ? 4.0 / 3.0 : 1.0, c = order == 4 ? -1.0 / 3.0 : 0.0;
  for (int k = 0; k < 3; ++k) {
    b.c1[k] = (a / 2.0) / spacing[k];
    b.c2[k] = (c / 4.0) / spacing[k];
    b.cg[k] = cfs::pair_of(order == 4 ? b.c2[k] : b.c1[k]);
  }
  b.rs = order == 4 ? 2 : 1;
  b.dV = spacing[0] * spacing[1] * (nz > 1 ? spacing[2] : 1.0);
  const int rows = cfs::diag_rows(nx, ny, nz, kMaxRows);
  int rc = cfs::launch_diagnostics_block(b, U, partials, 0, rows, cuda_stream);
  if (rc == 0) rc = cfs::launch_diagnostics_final(partials, rows, out, b.dV * (double)N, cuda_stream);
  if (rc != 0) {
    put(err, err_len, cudaGetErrorString((cudaError_t)rc));
    return CFS_ECUDA;
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) {
    put(err, err_len, cudaGetErrorString(e));
    return CFS_ECUDA;
  }
  return CFS_OK;
}

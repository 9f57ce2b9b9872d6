// Test harness for launch shapes: the halo store of a synchronous step, which its kernel leaves at once without
// reading anything, for any number of sub-domains.
#include <cuda_runtime.h>

#include "cfs_internal.h"

extern "C" int halo_block_launch(int nsub, int n) {
  cfs::Geometry g{};
  g.nsub = nsub;
  const int rc = cfs::launch_halo_block(g, cfs::Physics{}, cfs::StepSched{}, nullptr, nullptr, n, nullptr, nullptr, -1, nullptr,
                                        nullptr, nullptr);
  return rc ? rc : (int)cudaDeviceSynchronize();
}

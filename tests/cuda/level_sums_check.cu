// Test harness for level_sums.cuh: the five variables' sums over five levels, r [n][5][5], with weights c.
#include "level_sums.cuh"

using namespace cfs;

__global__ void k_sums(const double* r, const float2* c, float* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double lv[CFS_MAX_LEVELS][5];
  for (int l = 0; l < 5; ++l)
    for (int v = 0; v < 5; ++v) lv[l][v] = r[(i * 5 + l) * 5 + v];
  float2 w[CFS_MAX_LEVELS];
  for (int l = 0; l < 5; ++l) w[l] = c[l];
  LevelDiffs d;
  level_diffs(lv, 5, d);
  at_sums(d, w, 5, out + i * 5);
}

extern "C" int level_sums(const double* r, const float2* c, float* out, int n) {
  k_sums<<<(n + 255) / 256, 256>>>(r, c, out, n);
  return (int)cudaDeviceSynchronize();
}

// Test harness for p_double_int (pairs.cuh): normalised pairs to FP64 on the integer pipe.
#include <cuda_runtime.h>

#include "pairs.cuh"

using namespace cfs;

__global__ void k_double(const float2* a, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = p_double_int(p_of(a[i]));
}

extern "C" int pair_double(const float2* a, double* out, int n) {
  k_double<<<(n + 255) / 256, 256>>>(a, out, n);
  return (int)cudaDeviceSynchronize();
}

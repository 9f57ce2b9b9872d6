// Test harness for pairs.cuh: the operations on pairs split from FP64 values, returned as (h, l).
#include <cuda_runtime.h>

#include "pairs.cuh"

using namespace cfs;

__global__ void k_pairs(const double* a, const double* b, const double* c, float2* out, double* dbl, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const P1 x = p_split(a[i]), y = p_split(b[i]), z = p_split(c[i]);
  const P2 xx = p_pair(x, y), yy = p_pair(y, z), zz = p_pair(z, x);
  const P1 r[7] = {x, p_add(x, y), p_sub(x, y), p_mul(x, y), p_fma(x, y, z), p_recip(x), p_x(p_fma(xx, yy, zz))};
  for (int k = 0; k < 7; ++k) out[(long long)k * n + i] = p_store(r[k]);
  dbl[i] = p_double(x);
}

extern "C" int pairs_check(const double* a, const double* b, const double* c, float2* out, double* dbl, int n) {
  k_pairs<<<(n + 255) / 256, 256>>>(a, b, c, out, dbl, n);
  return (int)cudaDeviceSynchronize();
}

__global__ void k_pairs_pow(const double* x, double a, const float* tab, float2* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = p_store(p_pow(p_split(x[i]), p_split(a), tab));
}

extern "C" int pairs_pow(const double* x, double a, float2* out, int n) {
  float t[POW_PAIR_TAB], *d = nullptr;
  pow_pair_table(t);
  if (cudaMalloc(&d, sizeof(t)) != cudaSuccess) return 1;
  cudaMemcpy(d, t, sizeof(t), cudaMemcpyHostToDevice);
  k_pairs_pow<<<(n + 255) / 256, 256>>>(x, a, d, out, n);
  const int rc = (int)cudaDeviceSynchronize();
  cudaFree(d);
  return rc;
}

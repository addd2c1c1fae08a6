// Device functions of the packed rows, one kernel each, for test_gpu_rows_probe.py.
#include "packed_kernels.cuh"

using namespace sbi;

__global__ void k_quotients(const float2* a, const float2* d, float2* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = pk::parts(pk::quotient(pk::f2(a[i]), pk::f2(d[i])));
}
extern "C" int probe_quotients(const void* a, const void* d, void* out, int n) {
  k_quotients<<<(n + 255) / 256, 256>>>((const float2*)a, (const float2*)d, (float2*)out, n);
  return (int)cudaDeviceSynchronize();
}

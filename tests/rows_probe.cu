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

// out[m][k], k < N / RP: the factor w_N^{m k} by which the third pass of a transform
// of N elements multiplies input m of butterfly k (a lone input of one comes out as it)
template <int N>
__global__ void k_third(const void* tw, float2* out) {
  using F = pk::PackedFft<pk::One, N, 16, false>;
  constexpr int R = 16, T = F::T, RP = N / 256, Q = R / RP;
  for (int m = 1; m < RP; ++m) {
    pk::One x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = pk::f2(r / Q == m ? 1.f : 0.f, 0.f);
    F::template last_pass<RP, false>(x, threadIdx.x, F::twiddles(nullptr, 0), (const float2*)tw);
#pragma unroll
    for (int q = 0; q < Q; ++q) out[m * Q * T + q * T + threadIdx.x] = pk::parts(x[q]);
  }
}
template <int N>
int third(const void* tw, void* out) {
  k_third<N><<<1, N / 16>>>(tw, (float2*)out);
  return (int)cudaDeviceSynchronize();
}
extern "C" int probe_third_pass(int n, const void* tw, void* out) {
  return n == 512 ? third<512>(tw, out) : n == 1024 ? third<1024>(tw, out) : n == 2048 ? third<2048>(tw, out) : -1;
}

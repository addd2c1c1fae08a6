// Row and RK pass instantiations of packed groups (two-dimensional, FP32) and
// the FP32 state conversions.
#include "packed_kernels.cuh"

namespace sbi {
// the long rows are compiled in inst_packed_row_long.cu
#define SBI_LONG_ROWS(N)                                                                    \
  extern template cudaError_t pk::prepare_packed_row_n<N>();                                  \
  extern template cudaError_t pk::launch_packed_row_n<N>(const RowParams&, cudaStream_t, bool);     \
  extern template cudaError_t pk::launch_packed_rk_n<N>(const RkParams&, cudaStream_t, bool);
SBI_LONG_ROWS(512) SBI_LONG_ROWS(1024) SBI_LONG_ROWS(2048) SBI_LONG_ROWS(4096)

#define SBI_PACKED_NX(X) X(16) X(32) X(64) X(128) X(256) X(512) X(1024) X(2048) X(4096)
#define SBI_SWITCH(N, F, BAD) switch (nx) { SBI_PACKED_NX(F) default: return BAD; }

cudaError_t prepare_packed_row_kernels(int nx) {
#define SBI_CASE(N) case N: return pk::prepare_packed_row_n<N>();
  SBI_SWITCH(nx, SBI_CASE, cudaErrorInvalidValue)
#undef SBI_CASE
}
cudaError_t launch_packed_row(int nx, const RowParams& p, cudaStream_t st, bool chained) {
#define SBI_CASE(N) case N: return pk::launch_packed_row_n<N>(p, st, chained);
  SBI_SWITCH(nx, SBI_CASE, cudaErrorInvalidValue)
#undef SBI_CASE
}
cudaError_t launch_packed_rk(int nx, const RkParams& p, cudaStream_t st, bool chained) {
#define SBI_CASE(N) case N: return pk::launch_packed_rk_n<N>(p, st, chained);
  SBI_SWITCH(nx, SBI_CASE, cudaErrorInvalidValue)
#undef SBI_CASE
}
int packed_row_geometry(int nx, int* threads) {
  *threads = 0;
#define SBI_CASE(N) case N: *threads = pk::RowGeo<N>::T; return pk::RowGeo<N>::MAXR;
  SBI_SWITCH(nx, SBI_CASE, 0)
#undef SBI_CASE
}
template <> cudaError_t state_convert<float>(const void* src, void* dst, long long n, bool to_double,
                                             cudaStream_t st) {
  return state_convert_impl<float>(src, dst, n, to_double, st);
}
}  // namespace sbi

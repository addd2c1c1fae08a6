// Row and RK pass instantiations of packed groups, rows of 512 points and more.
#include "packed_kernels.cuh"

namespace sbi {
#define SBI_LONG_ROWS(N)                                                             \
  template cudaError_t pk::prepare_packed_row_n<N>();                                  \
  template cudaError_t pk::launch_packed_row_n<N>(const RowParams&, cudaStream_t, bool);     \
  template cudaError_t pk::launch_packed_rk_n<N>(const RkParams&, cudaStream_t, bool);
SBI_LONG_ROWS(512) SBI_LONG_ROWS(1024) SBI_LONG_ROWS(2048) SBI_LONG_ROWS(4096)
}  // namespace sbi

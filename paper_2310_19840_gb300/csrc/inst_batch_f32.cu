// Row, column and RK pass instantiations of large ensembles of one-dimensional
// FP32 members.
#include "kernels.cuh"

namespace sbi {
template <> cudaError_t launch_row<float>(int nx, const RowParams& p, cudaStream_t st) {
  return launch_row_impl<float>(nx, p, st);
}
template <> cudaError_t launch_rk<float>(int nx, const RkParams& p, cudaStream_t st) {
  return launch_rk_impl<float>(nx, p, st);
}
template <> cudaError_t launch_col<float>(int ny, const ColParams& p, cudaStream_t st) {
  return ny == 1 ? launch_col_n<float, 1>(p, st) : cudaErrorInvalidValue;
}
template <> cudaError_t prepare_row_kernels<float>(int nx) { return prepare_row_impl<float>(nx); }
template <> cudaError_t prepare_col_kernels<float>(int ny) {
  return ny == 1 ? prepare_ny<float, 1>() : cudaErrorInvalidValue;
}
template <> int row_rpc<float>(int nx, int W, int nslots) { return row_rpc_impl<float>(nx, W, nslots); }
template <> int row_tpr<float>(int nx) { return row_tpr_impl<float>(nx); }
template <> int col_geometry<float>(int ny, int* tpc) {
  *tpc = ny == 1 ? ColCfg<float, 1>::TPC : 0;
  return ny == 1 ? ColCfg<float, 1>::CPB : 0;
}
}  // namespace sbi

// Instantiations of the one-dimensional FP32 step.
#include "line.cuh"

namespace sbi {
#define SBI_LINE_NX(X) X(16) X(32) X(64) X(128) X(256) X(512) X(1024) X(2048) X(4096)
#define SBI_SWITCH(F) switch (nx) { SBI_LINE_NX(F) default: return cudaErrorInvalidValue; }

cudaError_t prepare_line_kernels(int nx) {
#define SBI_CASE(N) case N: return pk::prepare_line_n<N>();
  SBI_SWITCH(SBI_CASE)
#undef SBI_CASE
}
cudaError_t launch_line(int nx, const LineParams& p, cudaStream_t st) {
#define SBI_CASE(N) case N: return pk::launch_line_n<N>(p, st);
  SBI_SWITCH(SBI_CASE)
#undef SBI_CASE
}
cudaError_t line_clusters(int nx, int cluster, int* most) {
#define SBI_CASE(N) case N: return pk::line_clusters_n<N>(cluster, most);
  SBI_SWITCH(SBI_CASE)
#undef SBI_CASE
}
}  // namespace sbi

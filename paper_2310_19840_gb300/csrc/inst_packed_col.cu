// Column pass instantiations of packed groups (two-dimensional, FP32) and the
// FP32 multiplier tables.
#include "packed_kernels.cuh"

namespace sbi {
#define SBI_PACKED_NY(X) X(8) X(16) X(32) X(64) X(128) X(256) X(512) X(1024) X(2048)
#define SBI_SWITCH(N, F, BAD) switch (ny) { SBI_PACKED_NY(F) default: return BAD; }

cudaError_t prepare_packed_col_kernels(int ny) {
#define SBI_CASE(N) case N: return pk::prepare_packed_col_n<N>();
  SBI_SWITCH(ny, SBI_CASE, cudaErrorInvalidValue)
#undef SBI_CASE
}
cudaError_t launch_packed_col(int ny, const ColParams& p, cudaStream_t st, bool chained) {
#define SBI_CASE(N) case N: return pk::launch_packed_col_n<N>(p, st, chained);
  SBI_SWITCH(ny, SBI_CASE, cudaErrorInvalidValue)
#undef SBI_CASE
}
namespace {
template <typename G>
int geometry(int* tpc, int* group) {
  *tpc = G::T;
  *group = G::CI;
  return G::CPB;
}
}  // namespace
int packed_col_geometry(const ColParams& p, int* tpc, int* group) {
  const int ny = p.ny;
  const bool half = pk::col_half(p);
  *tpc = *group = 0;
#define SBI_CASE(N) \
  case N: return half ? geometry<pk::ColGeo<N, true>>(tpc, group) : geometry<pk::ColGeo<N, false>>(tpc, group);
  SBI_SWITCH(ny, SBI_CASE, 0)
#undef SBI_CASE
}
bool packed_col_stageable(int ny) {
#define SBI_CASE(N) case N: return pk::ColGeo<N, true>::STAGEABLE;
  SBI_SWITCH(ny, SBI_CASE, false)
#undef SBI_CASE
}
int packed_col_most_wide(const ColParams& p) {
  const int ny = p.ny;
  const bool half = pk::col_half(p);
#define SBI_CASE(N) case N: return half ? pk::col_most_wide<N, true>(p) : pk::col_most_wide<N, false>(p);
  SBI_SWITCH(ny, SBI_CASE, 0)
#undef SBI_CASE
}
template <> cudaError_t launch_coef_table<float>(void* out, const TableSpec& s, cudaStream_t st) {
  return launch_coef_table_impl<float>(out, s, st);
}
}  // namespace sbi

// FP32 instantiation of the DG passes (mixed-precision V-cycle, Section 4).
#include "dg_launch.cuh"

namespace sipg {

template <>
void upload_tables_dg<float>(const Tables<float> &t, const BoxTables<float> &bt) {
  upload_tables_tu(t);
  upload_box_tu(bt);
}
template <>
cudaError_t launch_dg_eval<float>(int n, const DGArgs<float> &a, cudaStream_t s, int cb) {
  return dispatch_dg<float>(0, n, &a, s, cb);
}
template <>
cudaError_t launch_dg_integrate<float>(int n, const DGArgs<float> &a, cudaStream_t s, int cb) {
  return dispatch_dg<float>(1, n, &a, s, cb);
}
template <>
cudaError_t launch_dg_box<float>(int n, const DGArgs<float> &a, cudaStream_t s) {
  return dispatch_dg<float>(2, n, &a, s, 0);
}
template <>
BoxShape dg_box_shape<float>(int n, const int m[3], int cb) { return box_shape<float>(n, m, cb); }
template <>
TileLaunch dg_tile<float>(int n, bool curved, const int m[3], int64_t ncells, int cb) {
  return dg_tile_launch<float>(n, curved, m, ncells, cb);
}
template <>
int dg_cells_per_block<float>(int n, bool curved) { return curved ? default_cb(n) : box_default_cells<float>(n); }
template <>
int dg_max_cells_per_block<float>(int n) { return max_cb(n, sizeof(float)); }
template <>
cudaError_t dg_blocks_per_sm<float>(int n, bool curved, int pass, int groups, int *blocks) {
  return dispatch_dg<float>(3, n, nullptr, nullptr, groups, curved, pass == 1, blocks);
}
template <>
cudaError_t prepare_dg_kernels<float>() { return prep_dg_all<float>(); }

}  // namespace sipg

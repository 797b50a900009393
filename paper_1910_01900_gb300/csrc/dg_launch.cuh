// Launchers of the DG passes: dispatch over the runtime tile size n to the
// compile-time kernels.  Included once per precision.
#pragma once
#include <algorithm>

#include "dg_kernels.cuh"

namespace sipg {

// the width that a setting of cb cells runs at: kCurvedThreads threads and the
// shared memory at most
template <typename T>
static int curved_cb(int n, int cb) {
  return std::min({cb, kCurvedThreads / (n * n), 232448 / (curved_cell_values(n, true) * (int)sizeof(T))});
}

template <typename T, int N>
static cudaError_t run_dg(bool integrate, const DGArgs<T> &a, cudaStream_t s, int cb) {
  if (cb <= 0) cb = default_cb(N);
  if (cb > max_cb(N, sizeof(T))) return cudaErrorInvalidValue;
  cb = curved_cb<T>(N, cb);
  const size_t smem = (size_t)cb * curved_cell_values(N, integrate) * sizeof(T);
  const int64_t grid = (int64_t)((a.ncells + cb - 1) / cb) * a.nv;
  if (grid == 0) return cudaSuccess;
  if (grid > 0x7fffffff) return cudaErrorInvalidValue;
  if (a.ufn) {   // unstructured mesh: single vector
    if (a.nv != 1) return cudaErrorInvalidValue;
    if (integrate)
      dg_integrate_unstr_kernel<T, N><<<(unsigned)grid, cb * N * N, smem, s>>>(a, cb);
    else
      dg_eval_unstr_kernel<T, N><<<(unsigned)grid, cb * N * N, smem, s>>>(a, cb);
  } else if (a.nv > 1) {
    if (integrate)
      dg_integrate_kernel<T, N, true><<<(unsigned)grid, cb * N * N, smem, s>>>(a, cb);
    else
      dg_eval_kernel<T, N, true><<<(unsigned)grid, cb * N * N, smem, s>>>(a, cb);
  } else {
    if (integrate)
      dg_integrate_kernel<T, N, false><<<(unsigned)grid, cb * N * N, smem, s>>>(a, cb);
    else
      dg_eval_kernel<T, N, false><<<(unsigned)grid, cb * N * N, smem, s>>>(a, cb);
  }
  note_launch();
  return cudaGetLastError();
}

// The one pass of axis-aligned cells.  Grid y and z hold at most 65535
// blocks: longer meshes, or more vectors, go in several launches.
template <typename T, int N>
static cudaError_t run_dg_box(const DGArgs<T> &a, cudaStream_t s) {
  const int groups = box_groups<T>(a.box);
  if (groups < 1 || groups * N * N > kCellThreads) return cudaErrorInvalidValue;
  if (a.ncells == 0) return cudaSuccess;
  int nb[3];
  for (int d = 0; d < 3; ++d) {
    const int w = a.box.w[d] * (d == 0 ? a.box.bricks : 1);
    nb[d] = (a.m[d] + w - 1) / w;
  }
  const size_t smem = (size_t)groups * box_group_values(N) * 8;
  constexpr int most = 65535;
  for (int oz = 0; oz < nb[2]; oz += most)
    for (int oy = 0; oy < nb[1]; oy += most) {
      const int ny = std::min(most, nb[1] - oy), nz = std::min(most, nb[2] - oz), step = most / nz;
      for (int r = 0; r < a.nv; r += step) {
        DGArgs<T> b = a;
        b.nv = std::min(step, a.nv - r);
        b.u = a.u + r * a.vs;
        b.out = a.out + r * a.vs;
        b.x = a.x ? a.x + r * a.vs : nullptr;
        b.xp = a.xp ? a.xp + r * a.vs : nullptr;
        b.b = a.b ? a.b + r * a.vs : nullptr;
        const dim3 grid((unsigned)nb[0], (unsigned)ny, (unsigned)(nz * b.nv));
        if (b.nv > 1)
          dg_box_kernel<T, N, true><<<grid, groups * N * N, smem, s>>>(b, oy, oz, nz);
        else
          dg_box_kernel<T, N, false><<<grid, groups * N * N, smem, s>>>(b, oy, oz, nz);
        note_launch();
      }
    }
  return cudaGetLastError();
}

// Resident thread blocks per SM of one pass in blocks of groups x N^2 threads.
template <typename T, int N>
static cudaError_t occ_dg(bool curved, bool integrate, int groups, int *blocks) {
  if (!curved)
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, dg_box_kernel<T, N, false>, groups * N * N,
                                                         (size_t)groups * box_group_values(N) * 8);
  const size_t smem = (size_t)groups * curved_cell_values(N, integrate) * sizeof(T);
  return integrate ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, dg_integrate_kernel<T, N, false>,
                                                                   groups * N * N, smem)
                   : cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, dg_eval_kernel<T, N, false>,
                                                                   groups * N * N, smem);
}

// Opt every kernel into the shared memory of its widest block (once per
// device, before any launch or stream capture).
template <typename T, int N>
static cudaError_t prep_dg_n() {
  constexpr cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const int smem = curved_cb<T>(N, max_cb(N, sizeof(T))) * curved_cell_values(N, true) * (int)sizeof(T);
  const int bsmem = std::min(232448, kCellThreads / (N * N) * box_group_values(N) * 8);
  cudaError_t e = cudaSuccess;
  for (cudaError_t r : {cudaFuncSetAttribute(dg_integrate_kernel<T, N, false>, at, smem),
                        cudaFuncSetAttribute(dg_eval_kernel<T, N, false>, at, smem),
                        cudaFuncSetAttribute(dg_integrate_kernel<T, N, true>, at, smem),
                        cudaFuncSetAttribute(dg_eval_kernel<T, N, true>, at, smem),
                        cudaFuncSetAttribute(dg_integrate_unstr_kernel<T, N>, at, smem),
                        cudaFuncSetAttribute(dg_eval_unstr_kernel<T, N>, at, smem),
                        cudaFuncSetAttribute(dg_box_kernel<T, N, false>, at, bsmem),
                        cudaFuncSetAttribute(dg_box_kernel<T, N, true>, at, bsmem)})
    if (r != cudaSuccess) e = r;
  return e;
}

template <typename T>
static cudaError_t prep_dg_all() {
  cudaError_t e = cudaSuccess;
  for (cudaError_t r : {prep_dg_n<T, 2>(), prep_dg_n<T, 3>(), prep_dg_n<T, 4>(), prep_dg_n<T, 5>(),
                        prep_dg_n<T, 6>(), prep_dg_n<T, 7>(), prep_dg_n<T, 8>(), prep_dg_n<T, 9>()})
    if (r != cudaSuccess) e = r;
  return e;
}

// The block shape of at most cb cells.  A brick of 2 x 2 x 2 reads one
// neighbour line per line and direction from memory, narrower ones two in
// their narrow directions, so the brick is as wide as cb and the mesh allow
// (z first, whose lines read best), then as many bricks side by side.  FP32
// works on pairs, so its blocks hold at least two cells.
template <typename T>
static BoxShape box_shape(int n, const int m[3], int cb) {
  if (cb <= 0) cb = box_default_cells<T>(n);
  BoxShape b;
  b.w[0] = (kBoxLanes<T> == 2 || (cb >= 2 && m[0] > 1)) ? 2 : 1;
  int left = std::max(1, cb / b.w[0]);
  for (int d : {2, 1}) {
    b.w[d] = left >= 2 && m[d] > 1 ? 2 : 1;
    left /= b.w[d];
  }
  const int nx = (m[0] + b.w[0] - 1) / b.w[0];
  // the fewest blocks that left bricks each can cover the row with, evenly
  const int blocks = (nx + left - 1) / left;
  b.bricks = (nx + blocks - 1) / blocks;
  return b;
}

// what a width setting of cb cells (0 = default) launches on a mesh of m cells
template <typename T>
static TileLaunch dg_tile_launch(int n, bool curved, const int m[3], int64_t ncells, int cb) {
  if (curved) {
    const int c = curved_cb<T>(n, cb > 0 ? cb : default_cb(n));
    return {c, c * n * n, (ncells + c - 1) / c};
  }
  const BoxShape b = box_shape<T>(n, m, cb);
  TileLaunch t{b.bricks * b.w[0] * b.w[1] * b.w[2], box_groups<T>(b) * n * n, 1};
  for (int d = 0; d < 3; ++d) {
    const int w = b.w[d] * (d == 0 ? b.bricks : 1);
    t.blocks *= (m[d] + w - 1) / w;
  }
  return t;
}

// op 0 evaluation, 1 integration, 2 the one pass of axis-aligned cells; 3 an
// occupancy query of the given pass in blocks of cb n^2 threads into *blocks
template <typename T>
static cudaError_t dispatch_dg(int op, int n, const DGArgs<T> *a, cudaStream_t s, int cb, bool curved = true,
                               bool integrate = true, int *blocks = nullptr) {
#define SIPG_DG_CASE(NN)                                                 \
  case NN:                                                               \
    if (op == 3) return occ_dg<T, NN>(curved, integrate, cb, blocks);    \
    return op == 2 ? run_dg_box<T, NN>(*a, s) : run_dg<T, NN>(op == 1, *a, s, cb);
  switch (n) {
    SIPG_DG_CASE(2)
    SIPG_DG_CASE(3)
    SIPG_DG_CASE(4)
    SIPG_DG_CASE(5)
    SIPG_DG_CASE(6)
    SIPG_DG_CASE(7)
    SIPG_DG_CASE(8)
    SIPG_DG_CASE(9)
    default:
      return cudaErrorInvalidValue;
  }
#undef SIPG_DG_CASE
}

}  // namespace sipg

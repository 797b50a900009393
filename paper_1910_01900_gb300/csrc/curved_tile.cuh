// Tiles and the cell term of curved cells, shared by the DG passes and the FE
// cell pass.
#pragma once
#include "sumfac.cuh"

namespace sipg {

// Shared memory of one cell of the curved passes.  Data goes from the lines of one
// direction to the lines of the next through tiles, and a tile that only two
// directions touch can be laid out so that the lines of both start on
// different banks; no affine layout does that for all three (with one layout
// for all, 45-54% of the shared-memory wavefronts were conflicts, and the L1
// data pipe bounds these passes).  So there is a tile per pair of directions,
// strides of (x, y, z):
//   X (1, X2, X3)  between y- and z-lines (two of them, but one in the evaluation)
//   Z (Z3, Z2, 1)  between x- and y-lines
//   Y (1, Y2, Y3)  between x- and z-lines
// and the x-lines are dealt to the threads z first.  Strides and the cells'
// distance CS were searched per N for the fewest wavefronts over a block's
// warps, weighted by the accesses: 1.21 per access at N = 6 (1.60 with one
// layout for all), 1.02 at N = 4 (1.31), 1.14 at N = 8 (1.44).  Faces: N lines
// of N values FP apart, F2 per face array.
struct CurvedLayout {
  int x2, x3, z2, z3, y2, y3, fp, f2, cs, ce;   // cs, ce: the DG integration and the evaluation pass
};
__host__ __device__ constexpr CurvedLayout curved_layout(int n) {
  return n == 2   ? CurvedLayout{2, 6, 2, 6, 2, 5, 2, 4, 100, 68}
         : n == 3 ? CurvedLayout{3, 11, 3, 11, 3, 10, 3, 9, 233, 137}
         : n == 4 ? CurvedLayout{4, 20, 4, 20, 4, 17, 4, 19, 528, 496}
         : n == 5 ? CurvedLayout{5, 37, 5, 26, 5, 33, 5, 25, 953, 761}
         : n == 6 ? CurvedLayout{6, 38, 6, 37, 6, 37, 6, 37, 1348, 1124}
         : n == 7 ? CurvedLayout{7, 52, 7, 55, 7, 49, 7, 51, 2065, 1681}
         : n == 8 ? CurvedLayout{8, 72, 8, 68, 8, 65, 8, 67, 3008, 2336}
                  : CurvedLayout{9, 81, 9, 81, 9, 81, 9, 81, 3889, 2929};
}
// shared-memory values per cell of a DG pass
__host__ __device__ constexpr int curved_cell_values(int n, bool integrate) {
  return integrate ? curved_layout(n).cs : curved_layout(n).ce;
}
template <int N>
struct CurvedTile {
  static constexpr CurvedLayout L = curved_layout(N);
  static constexpr int FP = L.fp, F2 = L.f2, CS = L.cs, CE = L.ce;
  static constexpr int X2 = L.x2, X3 = L.x3, Z2 = L.z2, Z3 = L.z3, Y2 = L.y2, Y3 = L.y3;
  static constexpr int SX = (N - 1) * (X2 + X3) + N, SZ = (N - 1) * (Z2 + Z3) + N, SY = (N - 1) * (Y2 + Y3) + N;
  // offsets: X, Z, Y, the second X, face arrays (evaluation: after X and Z)
  static constexpr int Z = SX, Y = Z + SZ, G = Y + SY, F = G + SX, FE = Y;
  static_assert(F2 >= (N - 1) * FP + N && CS >= F + 12 * F2 && CE >= FE + (N > 3 ? 18 : 6) * F2,
                "curved cell layout overlaps");
  // the FE cell pass: the four tiles, cells as far apart modulo the banks
  static constexpr int CF = F + ((CS - F) % 32);
};
// shared-memory values per cell of the FE cell pass
__host__ __device__ constexpr int fe_curved_cell_values(int n) {
  const CurvedLayout l = curved_layout(n);
  const int f = (n - 1) * (2 * (l.x2 + l.x3) + l.z2 + l.z3 + l.y2 + l.y3) + 4 * n;
  return f + (l.cs - f) % 32;
}
// A line's values: p[q * STEP].
template <typename T, int N, int STEP>
__device__ __forceinline__ void tile_load(const T *p, T (&x)[N]) {
#pragma unroll
  for (int q = 0; q < N; ++q) x[q] = p[q * STEP];
}
template <typename T, int N, int STEP>
__device__ __forceinline__ void tile_store(T *p, const T (&x)[N]) {
#pragma unroll
  for (int q = 0; q < N; ++q) p[q * STEP] = x[q];
}
// The lines of a thread in its cell's tiles; (la, lb) = (l % N, l / N) is its
// z-line's (x, y), its y-line's (x, z) and its x-line's (z, y).
template <typename T, int N>
struct CurvedLines {
  using C = CurvedTile<N>;
  T *xz, *xy;   // X tile: z-line, y-line (the second X tile C::G further on)
  T *zy, *zx;   // Z tile: y-line, x-line
  T *yx, *yz;   // Y tile: x-line, z-line
  static constexpr int XZ = C::X3, XY = C::X2, ZY = C::Z2, ZX = C::Z3, YX = 1, YZ = C::Y3;
  __device__ __forceinline__ CurvedLines(T *s, const int la, const int lb) {
    xz = s + la + C::X2 * lb;
    xy = s + la + C::X3 * lb;
    zy = s + C::Z + C::Z3 * la + lb;
    zx = s + C::Z + la + C::Z2 * lb;
    yx = s + C::Y + C::Y2 * lb + C::Y3 * la;
    yz = s + C::Y + la + C::Y2 * lb;
  }
};

// The interpolation of a cell's values to the Gauss points: x comes with the
// thread's z-line of u (u[l + q n^2], coalesced over the cell's threads) and
// leaves with its x-line of the result.  Every thread of the block takes part
// in the barriers.
template <typename T, int N>
__device__ __forceinline__ void curved_interpolate(const CurvedLines<T, N> &t, const bool act, T (&x)[N]) {
  using L = CurvedLines<T, N>;
  T y[N];
  if (act) {
    apply_mat<T, N, MS>(x, y);
    tile_store<T, N, L::XZ>(t.xz, y);
  }
  __syncthreads();
  if (act) {
    tile_load<T, N, L::XY>(t.xy, x);
    apply_mat<T, N, MS>(x, y);
    tile_store<T, N, L::ZY>(t.zy, y);
  }
  __syncthreads();
  if (act) {
    tile_load<T, N, L::ZX>(t.zx, y);
    apply_mat<T, N, MS>(y, x);
  }
}

// The cell term (grad v, grad u) from the x-line x of the values at the Gauss
// points to the thread's z-line x of the result: gradient (D), metric M (six
// components of N^3 values, M at the thread's z-line), transposed derivatives
// and transposed interpolation.  sweep(d, in, out) is D^T along a line of
// direction d with whatever a caller adds to it; extra() runs beside the
// y-lines of the gradient.  The z component of the gradient never leaves its
// thread.  Every thread of the block takes part in the barriers.
template <typename T, int N, typename Extra, typename Sweep>
__device__ __forceinline__ void curved_cell_term(const CurvedLines<T, N> &t, const bool act, const T *__restrict__ M,
                                                 T (&x)[N], Extra extra, Sweep sweep) {
  using L = CurvedLines<T, N>;
  constexpr int N2 = N * N, N3 = N2 * N, G = CurvedTile<N>::G;
  T y[N];
  if (act) {
    tile_store<T, N, L::ZX>(t.zx, x);
    apply_mat<T, N, MD>(x, y);
    tile_store<T, N, L::YX>(t.yx, y);
  }
  __syncthreads();
  if (act) {   // y-lines: the y component; the values on to the z-lines
    tile_load<T, N, L::ZY>(t.zy, x);
    tile_store<T, N, L::XY>(t.xy, x);
    apply_mat<T, N, MD>(x, y);
    tile_store<T, N, L::XY>(t.xy + G, y);
    extra();
  }
  __syncthreads();
  if (act) {   // z-lines: derivative, metric and transposed derivative
    tile_load<T, N, L::XZ>(t.xz, x);
    apply_mat<T, N, MD>(x, y);
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const T *m = M + q * N2;
      const T xx = m[0], yy = m[N3], zz = m[2 * N3], xy = m[3 * N3], xz = m[4 * N3], yz = m[5 * N3];
      T *p0 = t.yz + q * L::YZ, *p1 = t.xz + G + q * L::XZ;
      const T g0 = *p0, g1 = *p1, g2 = y[q];
      *p0 = xx * g0 + xy * g1 + xz * g2;
      *p1 = xy * g0 + yy * g1 + yz * g2;
      y[q] = xz * g0 + yz * g1 + zz * g2;
    }
    sweep(2, y, x);
    tile_store<T, N, L::XZ>(t.xz, x);
  }
  __syncthreads();
  if (act) {
    tile_load<T, N, L::XY>(t.xy + G, x);
    sweep(1, x, y);
#pragma unroll
    for (int q = 0; q < N; ++q) y[q] += t.xy[q * L::XY];
    tile_store<T, N, L::ZY>(t.zy, y);
  }
  __syncthreads();
  if (act) {   // x-lines, and the transposed interpolation along them
    tile_load<T, N, L::YX>(t.yx, x);
    sweep(0, x, y);
#pragma unroll
    for (int q = 0; q < N; ++q) y[q] += t.zx[q * L::ZX];
    apply_mat<T, N, MSt>(y, x);
    tile_store<T, N, L::ZX>(t.zx, x);
  }
  __syncthreads();
  if (act) {
    tile_load<T, N, L::ZY>(t.zy, x);
    apply_mat<T, N, MSt>(x, y);
    tile_store<T, N, L::XY>(t.xy, y);
  }
  __syncthreads();
  if (act) {
    tile_load<T, N, L::XZ>(t.xz, y);
    apply_mat<T, N, MSt>(y, x);
  }
}

}  // namespace sipg

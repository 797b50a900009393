// The polynomial transfers between FE levels on one mesh (Section 3.2), by
// bricks of cells.
//
// P is the tensor product of the 1D interpolation from the coarse to the fine
// nodes of a cell, and both spaces are continuous, so assembled it is a tensor
// product of block 1D matrices on the node grids: three passes of lines walked
// cell by cell, as the operator on axis-aligned cells is (fe_box.cuh).  A fine
// node on a cell's face counts once: there only the coarse function of the
// same node is not zero.  The kernels these replace for the degrees below took
// one thread block per coarse cell with a barrier and index divisions per
// contraction (restriction) or evaluated every fine node from its nc^3 coarse
// nodes (prolongation).
#pragma once
#include "fe_box.cuh"

namespace sipg {

// rc = P^T rf on the coarse nodes that brick bi of b cells owns (constrained
// ones 0, constrained fine nodes read as 0); with x0 the first Chebyshev step
// of the coarse level too, x0 = c3 D^-1 rc.
template <typename T, int NF, int NC>
__global__ void __launch_bounds__(256) fe_restrict_box_kernel(const XferGeom G, const int b0, const int b1, const int b2,
                                                             const T *__restrict__ P1, const T *__restrict__ rf,
                                                             T *__restrict__ rc, T *__restrict__ x0,
                                                             const T *__restrict__ dinv, const T c3) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *A = reinterpret_cast<T *>(smem_raw);
  constexpr int PF = NF - 1, PC = NC - 1;
  rf += blockIdx.y * G.sf;   // vector blockIdx.y
  rc += blockIdx.y * G.sc;
  if (x0) x0 += blockIdx.y * G.sc;
  T w[PF][NC];   // P1 without its last row (the next cell's first, or the grid's last node)
#pragma unroll
  for (int i = 0; i < PF; ++i)
#pragma unroll
    for (int j = 0; j < NC; ++j) w[i][j] = P1[i * NC + j];
  const int n0 = (G.mc[0] + b0 - 1) / b0, n1 = (G.mc[1] + b1 - 1) / b1, bi = blockIdx.x, r = bi / n0;
  const FESpan X = fe_span<PF>(bi - r * n0, b0, G.mc[0]), Y = fe_span<PF>(r % n1, b1, G.mc[1]),
               Z = fe_span<PF>(r / n1, b2, G.mc[2]);
  const int NT = blockDim.x, XP = X.ext | 1, SZ = XP * Y.ext;
  const int ox = X.cells * PC + X.last, oz = Z.cells * PC + Z.last;
  const int64_t gsz = (int64_t)G.gf[0] * G.gf[1];
  T x[NF], y[NC], carry;
  // one cell: y = its contributions to the coarse nodes from all fine nodes but the last
  auto cell = [&] {
#pragma unroll
    for (int j = 0; j < NC; ++j) {
      T s = w[0][j] * x[0];
#pragma unroll
      for (int i = 1; i < PF; ++i) s = fma(w[i][j], x[i], s);
      y[j] = s;
    }
  };
  for (int i = threadIdx.x; i < X.ext * Y.ext; i += NT) {   // along z, from memory
    const int yy = i / X.ext, xx = i - yy * X.ext, gx = X.first + xx, gy = Y.first + yy;
    const bool zero = (gx == 0 && G.bc[0] == 0) || (gx == G.gf[0] - 1 && G.bc[1] == 0) ||
                      (gy == 0 && G.bc[2] == 0) || (gy == G.gf[1] - 1 && G.bc[3] == 0);
    const T *p = rf + gx + (int64_t)G.gf[0] * gy + gsz * Z.first;
    T *o = A + xx + XP * yy;
    x[PF] = zero || (Z.first == 0 && G.bc[4] == 0) ? T(0) : p[0];
    carry = T(0);
    fe_walk(Z.halo, Z.cells,
            [&](const int c) {
              x[0] = x[PF];
#pragma unroll
              for (int j = 1; j < NF; ++j) {
                const int z = c * PF + j;
                x[j] = zero || (Z.first + z == G.gf[2] - 1 && G.bc[5] == 0) ? T(0) : p[gsz * z];
              }
              cell();
            },
            [](int) {},
            [&] {
              o[0] = carry + y[0];
#pragma unroll
              for (int j = 1; j < PC; ++j) o[j * SZ] = y[j];
              o += PC * SZ;
            },
            [&] { carry = y[PC]; });
    if (Z.last) o[0] = carry + x[PF];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < Y.ext * oz; i += NT) {   // along x, in place
    T *p = A + XP * i, *o = p;
    x[PF] = p[0];
    carry = T(0);
    fe_walk(X.halo, X.cells,
            [&](int) {
              x[0] = x[PF];
#pragma unroll
              for (int j = 1; j < NF; ++j) x[j] = p[j];
              p += PF;
              cell();
            },
            [](int) {},
            [&] {
              o[0] = carry + y[0];
#pragma unroll
              for (int j = 1; j < PC; ++j) o[j] = y[j];
              o += PC;
            },
            [&] { carry = y[PC]; });
    if (X.last) o[0] = carry + x[PF];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < ox * oz; i += NT) {   // along y, to the coarse nodes
    const int z = i / ox, xx = i - z * ox;
    int g[3] = {X.c0 * PC + xx, Y.c0 * PC, Z.c0 * PC + z};
    const T *p = A + xx + SZ * z;
    int64_t gid = g[0] + (int64_t)G.gc[0] * (g[1] + (int64_t)G.gc[1] * g[2]);
    auto out = [&](const T v) {
      const bool cons = (g[0] == 0 && G.bc[0] == 0) || (g[0] == G.gc[0] - 1 && G.bc[1] == 0) ||
                        (g[1] == 0 && G.bc[2] == 0) || (g[1] == G.gc[1] - 1 && G.bc[3] == 0) ||
                        (g[2] == 0 && G.bc[4] == 0) || (g[2] == G.gc[2] - 1 && G.bc[5] == 0);
      const T s = cons ? T(0) : v;
      rc[gid] = s;
      if (x0) x0[gid] = c3 * dinv[gid] * s;
      gid += G.gc[0];
      ++g[1];
    };
    x[PF] = p[0];
    carry = T(0);
    fe_walk(Y.halo, Y.cells,
            [&](int) {
              x[0] = x[PF];
#pragma unroll
              for (int j = 1; j < NF; ++j) x[j] = p[j * XP];
              p += PF * XP;
              cell();
            },
            [](int) {},
            [&] {
              out(carry + y[0]);
#pragma unroll
              for (int j = 1; j < PC; ++j) out(y[j]);
            },
            [&] { carry = y[PC]; });
    if (Y.last) out(carry + x[PF]);
  }
}

// xf += P xc on the fine nodes that brick bi of b cells owns (constrained ones
// keep their value).
template <typename T, int NF, int NC>
__global__ void __launch_bounds__(256) fe_prolongate_box_kernel(const XferGeom G, const int b0, const int b1,
                                                               const int b2, const T *__restrict__ P1,
                                                               const T *__restrict__ xc, T *__restrict__ xf) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int PF = NF - 1, PC = NC - 1;
  xc += blockIdx.y * G.sc;   // vector blockIdx.y
  xf += blockIdx.y * G.sf;
  T w[PF][NC];
#pragma unroll
  for (int i = 0; i < PF; ++i)
#pragma unroll
    for (int j = 0; j < NC; ++j) w[i][j] = P1[i * NC + j];
  const int n0 = (G.mc[0] + b0 - 1) / b0, n1 = (G.mc[1] + b1 - 1) / b1, bi = blockIdx.x, r = bi / n0;
  const FESpan X = fe_span<PF>(bi - r * n0, b0, G.mc[0]), Y = fe_span<PF>(r % n1, b1, G.mc[1]),
               Z = fe_span<PF>(r / n1, b2, G.mc[2]);
  // coarse nodes of the brick's own cells
  const int NT = blockDim.x, cx = X.cells * PC + 1, cy = Y.cells * PC + 1;
  T *A = reinterpret_cast<T *>(smem_raw), *B = A + cx * cy * Z.own;   // [z][cy][cx], [z][cy][x]
  const int64_t gsz = (int64_t)G.gc[0] * G.gc[1];
  T c[NC], y[PF];
  auto cell = [&] {
#pragma unroll
    for (int i = 0; i < PF; ++i) {
      T s = w[i][0] * c[0];
#pragma unroll
      for (int j = 1; j < NC; ++j) s = fma(w[i][j], c[j], s);
      y[i] = s;
    }
  };
  for (int i = threadIdx.x; i < cx * cy; i += NT) {   // along z, from memory
    const int yy = i / cx, xx = i - yy * cx;
    const T *p = xc + X.c0 * PC + xx + (int64_t)G.gc[0] * (Y.c0 * PC + yy) + gsz * (Z.c0 * PC);
    T *o = A + i;
    c[PC] = p[0];
#pragma unroll 1
    for (int k = 0; k < Z.cells; ++k) {
      c[0] = c[PC];
#pragma unroll
      for (int j = 1; j < NC; ++j) c[j] = p[gsz * (k * PC + j)];
      cell();
#pragma unroll
      for (int j = 0; j < PF; ++j) o[j * cx * cy] = y[j];
      o += PF * cx * cy;
    }
    if (Z.last) o[0] = c[PC];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < cy * Z.own; i += NT) {   // along x
    const T *p = A + cx * i;
    T *o = B + X.own * i;
    c[PC] = p[0];
#pragma unroll 1
    for (int k = 0; k < X.cells; ++k) {
      c[0] = c[PC];
#pragma unroll
      for (int j = 1; j < NC; ++j) c[j] = p[j];
      p += PC;
      cell();
#pragma unroll
      for (int j = 0; j < PF; ++j) o[j] = y[j];
      o += PF;
    }
    if (X.last) o[0] = c[PC];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < X.own * Z.own; i += NT) {   // along y, onto the fine nodes
    const int z = i / X.own, xx = i - z * X.own, gx = X.c0 * PF + xx, gz = Z.c0 * PF + z, g1 = Y.c0 * PF;
    if ((gx == 0 && G.bc[0] == 0) || (gx == G.gf[0] - 1 && G.bc[1] == 0) || (gz == 0 && G.bc[4] == 0) ||
        (gz == G.gf[2] - 1 && G.bc[5] == 0))
      continue;
    const T *p = B + xx + X.own * cy * z;
    T *o = xf + gx + (int64_t)G.gf[0] * (g1 + (int64_t)G.gf[1] * gz);
    c[PC] = p[0];
#pragma unroll 1
    for (int k = 0; k < Y.cells; ++k) {
      T f[PF];   // ahead of the stores
#pragma unroll
      for (int j = 0; j < PF; ++j) f[j] = o[(int64_t)G.gf[0] * j];
      c[0] = c[PC];
#pragma unroll
      for (int j = 1; j < NC; ++j) c[j] = p[j * X.own];
      p += PC * X.own;
      cell();
#pragma unroll
      for (int j = 0; j < PF; ++j)
        if (j || g1 + k || G.bc[2] != 0) o[(int64_t)G.gf[0] * j] = f[j] + y[j];
      o += (int64_t)G.gf[0] * PF;
    }
    if (Y.last && G.bc[3] != 0) o[0] += c[PC];
  }
}

}  // namespace sipg

// The FE operator on axis-aligned cells in one pass (Eq. WeakFormFE; Section
// 4, sum factorisation), with the node pass's epilogues.
//
// A box cell's matrix is sum_d alpha_d K1_d (x) M1 (x) M1, so the assembled
// operator is the same sum of products of assembled 1D matrices.  One thread
// block computes the nodes that a brick of cells owns (each cell its lower
// faces, the last brick of a direction the upper one too) from the nodes of
// those cells and of one more layer of cells below: along z a = M u and
// b = alpha_z K u on every (x, y) line of the extended brick, along x
// c = M a and f = alpha_x K a + M b on the lines of its (y, z), along y
// v = alpha_y K c + M f and the epilogue; every line is walked cell by cell
// with the shared node's partial sum carried over.  Only two tiles live in
// shared memory, and the lanes of a warp read and write neighbouring x.
//
// The cell pass and node pass this replaces on such cells moved (p+1)^3/p^3
// values per node more through an element buffer, took two launches, and the
// node pass was bound by its instructions (eight gathers per node).  The halo
// layer costs arithmetic instead: as much as the cell pass's doubled nodes at
// 4 x 4 x 2 cells of degree 4.  Every node is the same sum of the same cells'
// products whatever the brick, so its size changes no bit.  Measured (GB300),
// one smoothing step with its launch: FP32 32^3 cells of degree 4 45 -> 29 us,
// degree 2 13 us, 16^3 cells of degree 4 13 us; FP64 32^3 of degree 4 290 -> 273
// us (FP64 pipe); FP64 levels where the halo costs more than that saves take the
// two passes (fe_two_pass).  FP32 is bound by latency and occupancy: three stages with a
// barrier between them, 4 blocks of 256 threads per SM.
#pragma once
#include "sumfac.cuh"

namespace sipg {

// nodes of a brick along one direction
struct FESpan {
  int c0, cells, halo, last;   // first own cell, own cells, a layer below, the upper face is owned
  int first, ext, own;         // first node of the extended brick, its nodes, owned nodes
};
template <int P>
__device__ __forceinline__ FESpan fe_span(const int g, const int b, const int m) {
  FESpan s;
  s.c0 = g * b;
  s.cells = min(b, m - s.c0);
  s.halo = s.c0 > 0;
  s.last = s.c0 + s.cells == m;
  s.first = (s.c0 - s.halo) * P;
  s.ext = (s.cells + s.halo) * P + 1;
  s.own = s.cells * P + s.last;
  return s;
}
// One row's output (modes 0 to 2 of FEArgs): load() reads what it needs besides
// the operator's value y, value() forms it.  Apart, so that a thread can read
// for several rows before it stores the first (the output may be one of the
// vectors read, so loads never pass stores).
template <typename T>
struct FERow {
  T b, d, x, xp, u;
  bool cons;   // constrained: the identity row
  __device__ __forceinline__ void load(const FEArgs<T> &a, const int64_t vo, const int64_t gid, const bool constrained) {
    cons = constrained;
    b = d = x = xp = u = T(0);
    if (cons) u = a.u[vo + gid];
    if (a.mode == 0) return;
    b = a.b[vo + gid];
    if (a.mode == 2) return;
    d = a.dinv[gid];
    if (a.x) x = a.x[vo + gid];
    if (a.xp) xp = a.xp[vo + gid];
  }
  __device__ __forceinline__ T value(const FEArgs<T> &a, const T y) const {
    const T r = cons ? u : y;
    if (a.mode == 0) return r;
    if (a.mode == 2) return b - r;
    T v = a.c3 * d * (b - r);
    if (a.x) v = fma(a.c1, x, v);
    if (a.xp) v = fma(a.c2, xp, v);
    return v;
  }
};
// The output of row gid with operator value y, one row per thread.  FP32 reads
// the row's operands together, which FP64 is slower for (smoothing step on curved
// cells, FP32 16^3 of degree 4 17.3 us together, 17.7 us each where it is used;
// FP64 8^3 of degree 4 24.3 and 23.3 us).
template <typename T>
__device__ __forceinline__ void fe_row(const FEArgs<T> &a, const int64_t vo, const int64_t gid, const T y) {
  const int64_t gv = vo + gid;
  if constexpr (sizeof(T) == 4) {
    FERow<T> e;
    e.load(a, vo, gid, false);
    a.out[gv] = e.value(a, y);
  } else if (a.mode == 0) {
    a.out[gv] = y;
  } else if (a.mode == 2) {
    a.out[gv] = a.b[gv] - y;
  } else {
    T v = a.c3 * a.dinv[gid] * (a.b[gv] - y);
    if (a.x) v = fma(a.c1, a.x[gv], v);
    if (a.xp) v = fma(a.c2, a.xp[gv], v);
    a.out[gv] = v;
  }
}

// The cells of a line: ahead(c) for an own cell, product(c) of every cell,
// emit() of the own nodes, carry() of the last one's partial sum.  Of the halo
// cell only the carry is used; taken apart, the compiler drops the other rows
// of its product (FP64 32^3 cells of degree 4: 294 -> 273 us).
template <typename Product, typename Ahead, typename Emit, typename Carry>
__device__ __forceinline__ void fe_walk(const int halo, const int cells, Product product, Ahead ahead, Emit emit,
                                        Carry carry) {
  if (halo) {
    product(0);
    carry();
  }
#pragma unroll 1
  for (int c = halo; c < cells + halo; ++c) {
    ahead(c);
    product(c);
    emit();
    carry();
  }
}

// brick number bi (x fastest) of bricks of b0 x b1 x b2 cells, vector at vo
template <typename T, int N>
__device__ __forceinline__ void fe_box_body(const FEArgs<T> &a, const int64_t vo, const int b0, const int b1,
                                            const int b2, const int bi, T *sm) {
  constexpr int P = N - 1;
  const int n0 = (a.m[0] + b0 - 1) / b0, n1 = (a.m[1] + b1 - 1) / b1, r = bi / n0;
  const FESpan X = fe_span<P>(bi - r * n0, b0, a.m[0]), Y = fe_span<P>(r % n1, b1, a.m[1]),
               Z = fe_span<P>(r / n1, b2, a.m[2]);
  const int NT = blockDim.x, XP = X.ext | 1, SZ = XP * Y.ext;
  T *A = sm, *B = sm + (size_t)SZ * Z.own;
  const T *__restrict__ u = a.u + vo;
  const int64_t gsz = (int64_t)a.grid[0] * a.grid[1];

  for (int i = threadIdx.x; i < X.ext * Y.ext; i += NT) {
    const int y = i / X.ext, x = i - y * X.ext, gx = X.first + x, gy = Y.first + y;
    const bool zero = (gx == 0 && a.bc[0] == 0) || (gx == a.grid[0] - 1 && a.bc[1] == 0) ||
                      (gy == 0 && a.bc[2] == 0) || (gy == a.grid[1] - 1 && a.bc[3] == 0);
    const T *p = u + gx + (int64_t)a.grid[0] * gy + gsz * Z.first;
    T *pa = A + x + XP * y, *pb = B + x + XP * y;
    T v[N], nx[P], k[N], m[N], ca = T(0), cb = T(0);
    v[P] = zero || (Z.first == 0 && a.bc[4] == 0) ? T(0) : p[0];
    const int cells = Z.cells + Z.halo;
    auto fetch = [&](const int c) {   // the nodes of cell c above its first one
#pragma unroll
      for (int j = 0; j < P; ++j) {
        const int z = c * P + j + 1;
        nx[j] = zero || (Z.first + z == a.grid[2] - 1 && a.bc[5] == 0) ? T(0) : p[gsz * z];
      }
    };
    auto next = [&](const int c) {   // to cell c, the one after it on its way
      v[0] = v[P];
#pragma unroll
      for (int j = 0; j < P; ++j) v[j + 1] = nx[j];
      if (c + 1 < cells) fetch(c + 1);
      apply_mat<T, N, MM1>(v, m);
      apply_mat<T, N, MK1>(v, k);
    };
    fetch(0);
    fe_walk(Z.halo, Z.cells, [&](const int c) { next(c); }, [](int) {},
               [&] {
                 pa[0] = ca + m[0];
                 pb[0] = a.alpha[2] * (cb + k[0]);
#pragma unroll
                 for (int j = 1; j < P; ++j) {
                   pa[j * SZ] = m[j];
                   pb[j * SZ] = a.alpha[2] * k[j];
                 }
                 pa += P * SZ;
                 pb += P * SZ;
               },
               [&] {
                 ca = m[P];
                 cb = k[P];
               });
    if (Z.last) {
      pa[0] = ca;
      pb[0] = a.alpha[2] * cb;
    }
  }
  __syncthreads();
  // along x, in place: a line's own nodes land on nodes already read
  for (int i = threadIdx.x; i < Y.ext * Z.own; i += NT) {
    T *pa = A + XP * i, *pb = B + XP * i;
    T *oa = pa, *ob = pb;
    T v[N], w[N], k[N], m[N], mb[N], cc = T(0), cf = T(0);
    v[P] = pa[0];
    w[P] = pb[0];
    auto next = [&](int) {
      v[0] = v[P];
      w[0] = w[P];
#pragma unroll
      for (int j = 1; j < N; ++j) {
        v[j] = pa[j];
        w[j] = pb[j];
      }
      pa += P;
      pb += P;
      apply_mat<T, N, MM1>(v, m);
      apply_mat<T, N, MK1>(v, k);
      apply_mat<T, N, MM1>(w, mb);
#pragma unroll
      for (int j = 0; j < N; ++j) k[j] = fma(a.alpha[0], k[j], mb[j]);
    };
    fe_walk(X.halo, X.cells, next, [](int) {},
               [&] {
                 oa[0] = cc + m[0];
                 ob[0] = cf + k[0];
#pragma unroll
                 for (int j = 1; j < P; ++j) {
                   oa[j] = m[j];
                   ob[j] = k[j];
                 }
                 oa += P;
                 ob += P;
               },
               [&] {
                 cc = m[P];
                 cf = k[P];
               });
    if (X.last) {
      oa[0] = cc;
      ob[0] = cf;
    }
  }
  __syncthreads();
  // along y, and the rows out
  for (int i = threadIdx.x; i < X.own * Z.own; i += NT) {
    const int z = i / X.own, x = i - z * X.own, gx = X.c0 * P + x, gz = Z.c0 * P + z;
    const bool cons = (gx == 0 && a.bc[0] == 0) || (gx == a.grid[0] - 1 && a.bc[1] == 0) ||
                      (gz == 0 && a.bc[4] == 0) || (gz == a.grid[2] - 1 && a.bc[5] == 0);
    const T *pa = A + x + SZ * z, *pb = B + x + SZ * z;
    int64_t gid = gx + (int64_t)a.grid[0] * (Y.c0 * P) + gsz * gz;
    T v[N], w[N], k[N], m[N], cv = T(0);
    v[P] = pa[0];
    w[P] = pb[0];
    auto next = [&](int) {
      v[0] = v[P];
      w[0] = w[P];
#pragma unroll
      for (int j = 1; j < N; ++j) {
        v[j] = pa[j * XP];
        w[j] = pb[j * XP];
      }
      pa += P * XP;
      pb += P * XP;
      apply_mat<T, N, MK1>(v, k);
      apply_mat<T, N, MM1>(w, m);
#pragma unroll
      for (int j = 0; j < N; ++j) k[j] = fma(a.alpha[1], k[j], m[j]);
    };
    FERow<T> e[P];   // what the rows of a cell's own nodes read, ahead of their stores
    fe_walk(Y.halo, Y.cells, next,
               [&](const int c) {
#pragma unroll
                 for (int j = 0; j < P; ++j)
                   e[j].load(a, vo, gid + (int64_t)a.grid[0] * j,
                             cons || (j == 0 && c == 0 && !Y.halo && a.bc[2] == 0));
               },
               [&] {
#pragma unroll
                 for (int j = 0; j < P; ++j) {
                   a.out[vo + gid] = e[j].value(a, j == 0 ? cv + k[0] : k[j]);
                   gid += a.grid[0];
                 }
               },
               [&] { cv = k[P]; });
    if (Y.last) {
      FERow<T> e;
      e.load(a, vo, gid, cons || a.bc[3] == 0);
      a.out[vo + gid] = e.value(a, cv);
    }
  }
}

// Most threads of a block (the widest stage of the default bricks in two
// rounds), and blocks per SM to leave registers for: FP64 takes what a cell's
// lines need.
template <typename T>
__host__ __device__ constexpr int fe_box_threads(int) { return sizeof(T) == 8 ? 384 : 256; }
template <typename T>
__host__ __device__ constexpr int fe_box_blocks(int n) { return sizeof(T) == 8 ? 1 : (n <= 5 ? 4 : 3); }

// Cells per direction of a brick.  kFEBoxBrick[p]: about 16 own nodes along x
// and y and 8 along z, where a thin brick's tiles leave room for more blocks
// per SM (FP32 smoothing step on 32^3 cells of degree 4: 27.2 us for 4 x 4 x 2
// against 36.7 us for 4 x 4 x 4 and 35.3 us for 2 x 2 x 2).  Where that gives
// fewer bricks than the GPU can use, the side of most cells is halved until it
// does: FP32 below 140 bricks (16^3 of degree 4: 128 bricks 14.4 us, 256 12.9
// us), FP64, where the halo's arithmetic costs more, below 100 (50 us against
// 61 us) and at degree 1, where it costs little, below 200 (16^3: 128 bricks 10.3
// us, 256 8.5 us, in two passes 9.5 us).  cb > 0: the first brick of that sequence
// with at most cb cells.  Sides are evened out over the bricks of a direction.
constexpr int kFEBoxBrick[kMaxN][3] = {{1, 1, 1}, {16, 8, 4}, {8, 4, 4}, {5, 4, 2}, {4, 4, 2},
                                       {4, 2, 2}, {3, 2, 2},  {2, 2, 2}, {2, 2, 2}};
constexpr int kFEBoxSmem = 96 * 1024;   // degree 8 in FP32: 85 KB
template <typename T>
static void fe_box_brick(int n, const int m[3], int cb, int brick[3]) {
  const int p = n - 1, least = sizeof(T) == 4 ? 140 : (p == 1 ? 200 : 100);
  int b[3] = {kFEBoxBrick[p][0], kFEBoxBrick[p][1], kFEBoxBrick[p][2]};
  for (;;) {
    int64_t bricks = 1;
    for (int d = 0; d < 3; ++d) {
      const int k = (m[d] + b[d] - 1) / b[d];
      brick[d] = (m[d] + k - 1) / k;
      bricks *= k;
    }
    int d = 2;
    for (int e : {1, 0})
      if (b[e] > b[d]) d = e;
    if (b[d] == 1 || (cb > 0 ? brick[0] * brick[1] * brick[2] <= cb : bricks >= least)) break;
    b[d] = (b[d] + 1) / 2;
  }
}

// the launch of a brick: one round of the widest stage's lines, or two of half
// its width
template <typename T>
static TileLaunch fe_box_launch(int n, const int m[3], const int brick[3]) {
  TileLaunch t{brick[0] * brick[1] * brick[2], 0, 1};
  int w[3];
  for (int d = 0; d < 3; ++d) {
    t.blocks *= (m[d] + brick[d] - 1) / brick[d];
    w[d] = (brick[d] + 1 < m[d] ? brick[d] + 1 : m[d]) * (n - 1) + 1;
  }
  const int a = w[0] * w[1], b = w[1] * (brick[2] * (n - 1) + 1), lines = a > b ? a : b, rounds = lines > 256 ? 2 : 1;
  t.threads = ((lines + rounds - 1) / rounds + 31) / 32 * 32;
  if (t.threads > fe_box_threads<T>(n)) t.threads = fe_box_threads<T>(n);
  return t;
}

template <typename T, int N>
__global__ void __launch_bounds__(fe_box_threads<T>(N), fe_box_blocks<T>(N)) fe_box_kernel(const FEArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fe_box_body<T, N>(a, blockIdx.y * a.vs, a.brick[0], a.brick[1], a.brick[2], blockIdx.x,
                    reinterpret_cast<T *>(smem_raw));   // vector blockIdx.y
}

}  // namespace sipg

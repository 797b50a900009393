// Matrix-free SIPG operator on the DG level (Section 4, Eq.
// MatrixFreeAbstractNotation; weak form Eq. WeakFormDG with the fluxes of
// Eqs. InteriorPenaltyFlux1/2 and the mirror boundary conditions of
// Eq. BoundaryConditions).
//
// Face integrals without atomics, in two passes over the cells:
//
//  eval pass      : u_e -> u at the Gauss points (3 interpolation sweeps);
//                   the value and its normal derivative extrapolated to all
//                   six faces along the face normal, the tangential
//                   derivatives by 1D products on the faces themselves, and
//                   from them the value and the outward normal derivative,
//                   stored as the cell's face traces.
//  integrate pass : for every face the SIPG flux from the cell's own trace and
//                   the neighbour's trace, tested against the cell's own basis
//                   only (the neighbour integrates its own side in its own
//                   launch thread); the reference gradient at the Gauss points
//                   (3 collocation-derivative sweeps), the metric, 3
//                   transposed derivative sweeps with the face terms and 3
//                   transposed interpolation sweeps, and the fused epilogue.
//
// What the tangential derivatives of a face's trace need, and what its
// tangential test functions give, are 1D products of n lines on the face
// (12 n lines of a cell): the sweeps of the volume gradient to the faces and
// back that they replace read and wrote 12 and 12 values per DoF more.  The
// gradient's z component, the metric and its transposed derivative stay in the
// thread that owns the z-line.  Shared-memory accesses per DoF at n = 6:
// 23 -> 15 (evaluation), 48 -> 32 (integration).
//
// Each cell writes only its own outputs, so no two threads ever update the
// same global value.  Per face point the own side computes, with [u] =
// u_own - u_nb and q = outward normal derivative of each side,
//   value coefficient   A = dA (tau_f [u] - (q_own - q_nb)/2)     (times v)
//   normal-deriv coeff. B = -dA [u] / 2                           (times d_n v)
// and on Dirichlet faces A = dA (2 tau_e u - q), B = -dA u; on Neumann faces
// A = B = 0.  This is the per-side form of
//   -{d_n v}[u] - [v]{d_n u} + tau [v][u]  and  -d_n v u - v d_n u + 2 tau v u.
//
// Axis-aligned cells take one pass (dg_box.cuh); these two serve curved cells,
// structured or not.
#pragma once
#include "curved_tile.cuh"
#include "dg_box.cuh"

namespace sipg {

// Face point of the neighbour that sits at the own face point l = q1 + N q2
// (unstructured meshes): orientation code bit 0 swaps the two face
// directions, bits 1 and 2 reverse the first and second of them.
template <int N>
__device__ __forceinline__ int face_perm(const int code, const int l) {
  const int q1 = l % N, q2 = l / N;
  int a = (code & 1) ? q2 : q1, b = (code & 1) ? q1 : q2;
  if (code & 2) a = N - 1 - a;
  if (code & 4) b = N - 1 - b;
  return a + N * b;
}

// A line x at the Gauss points extrapolated to its two ends: the values l_s . x
// and the derivatives l_s . (D x) = (D^T l_s) . x.  l_1 is l_0 mirrored and D^T
// l_1 minus D^T l_0 mirrored, so both ends share the products of the even and
// the odd part (half the products; le, lo, de, do of Tables).
template <typename T, int N>
__device__ __forceinline__ void line_ends(const T (&x)[N], T &v0, T &v1, T &g0, T &g1) {
  constexpr int H = N / 2;
  const Tables<T> &t = tab<T>();
  if constexpr (N == 2) {   // two points: plain values, one derivative (Tables: le, lo = l_0)
    const T l0 = t.le[2][0], l1 = t.lo[2][0];
    v0 = fma(l1, x[1], l0 * x[0]);
    v1 = fma(l0, x[1], l1 * x[0]);
    g0 = g1 = t.D[2][1] * (x[1] - x[0]);
    return;
  }
  T ve = T(0), vo = T(0), ge = T(0), go = T(0);
#pragma unroll
  for (int j = 0; j < H; ++j) {
    const T e = x[j] + x[N - 1 - j], o = x[j] - x[N - 1 - j];
    ve = j ? fma(t.le[N][j], e, ve) : t.le[N][j] * e;
    ge = j ? fma(t.de[N][j], e, ge) : t.de[N][j] * e;
    vo = j ? fma(t.lo[N][j], o, vo) : t.lo[N][j] * o;
    go = j ? fma(t.dod[N][j], o, go) : t.dod[N][j] * o;
  }
  if constexpr (N & 1) {
    ve = fma(t.le[N][H], x[H], ve);
    ge = fma(t.de[N][H], x[H], ge);
  }
  v0 = ve + vo;
  v1 = ve - vo;
  g0 = go + ge;
  g1 = go - ge;
}

// The transpose, with the derivative sweep it meets: y = D^T x + l_0 a0 + l_1
// a1 + (D^T l_0) b0 + (D^T l_1) b1, the end terms added to the even and odd
// parts of y before they are put together (D^T swaps the parts).
template <typename T, int N>
__device__ __forceinline__ void sweep_with_ends(const T (&x)[N], const T a0, const T a1, const T b0, const T b1,
                                                T (&y)[N]) {
  constexpr int H = N / 2, HC = (N + 1) / 2;
  const Tables<T> &t = tab<T>();
  if constexpr (N == 2) {   // D^T l_0 = D^T l_1 = the rows of D
    const T l0 = t.le[2][0], l1 = t.lo[2][0], m = t.D[2][1] * ((x[0] + x[1]) + (b0 + b1));
    y[0] = fma(l0, a0, fma(l1, a1, -m));
    y[1] = fma(l1, a0, fma(l0, a1, m));
    return;
  }
  const T ap = a0 + a1, am = a0 - a1, bm = b0 - b1, bp = b0 + b1;
  T e[HC], o[H];
#pragma unroll
  for (int j = 0; j < H; ++j) {
    e[j] = x[j] + x[N - 1 - j];
    o[j] = x[j] - x[N - 1 - j];
  }
  if constexpr (N & 1) e[H] = x[H];
#pragma unroll
  for (int i = 0; i < HC; ++i) {
    T even = fma(t.le[N][i], ap, t.de[N][i] * bm);
#pragma unroll
    for (int j = 0; j < H; ++j) even = fma(t.DtO[N][i * 4 + j], o[j], even);
    if (i == N - 1 - i) {
      y[i] = even;
      continue;
    }
    T odd = fma(t.lo[N][i], am, t.dod[N][i] * bp);
#pragma unroll
    for (int j = 0; j < HC; ++j) odd = fma(t.DtE[N][i * 5 + j], e[j], odd);
    y[i] = even + odd;
    y[N - 1 - i] = even - odd;
  }
}

// Tangential 1D products on the cell's faces, thread by thread a line: the 12
// N lines (face f, tangential direction t, line j) of the cell go round its
// N^2 threads; line (f, t, j) is read from in(f, t) and written to out(f, t).
template <typename T, int N, int MAT, typename In, typename Out>
__device__ __forceinline__ void face_lines(const int l, In in, Out out) {
  constexpr int FP = CurvedTile<N>::FP;
#pragma unroll 1
  for (int k = l; k < 12 * N; k += N * N) {
    const int f = k / (2 * N), r = k - f * 2 * N, t = r / N, j = r - t * N;
    const int base = t ? j : FP * j, st = t ? FP : 1;
    T x[N], y[N];
    load_line<T, N>(in(f, t), base, st, x);
    apply_mat<T, N, MAT>(x, y);
    store_line<T, N>(out(f, t), base, st, y);
  }
}

// The same for one face point (q1, q2), whose own rows of the 1D matrix D or
// D^T for the two tangential directions it keeps: for N <= 3, where the 12 N lines would
// go round N^2 threads four or six times.
template <typename T, int N>
struct FacePoint {
  T r1[N], r2[N];
  int b1, b2;
  // rows q1 (first direction) and q2 (second) of D (TR: of D^T)
  template <bool TR>
  __device__ __forceinline__ void init(const int q1, const int q2) {
    const T *D = TR ? tab<T>().Dt[N] : tab<T>().D[N];
    b1 = CurvedTile<N>::FP * q2;
    b2 = q1;
#pragma unroll
    for (int j = 0; j < N; ++j) {
      r1[j] = D[j];
      r2[j] = D[j];
    }
#pragma unroll
    for (int i = 1; i < N; ++i)
#pragma unroll
      for (int j = 0; j < N; ++j) {   // selects: a constant read by thread would serialise
        r1[j] = q1 == i ? D[i * N + j] : r1[j];
        r2[j] = q2 == i ? D[i * N + j] : r2[j];
      }
  }
  __device__ __forceinline__ T first(const T *f) const {
    T v = r1[0] * f[b1];
#pragma unroll
    for (int j = 1; j < N; ++j) v = fma(r1[j], f[b1 + j], v);
    return v;
  }
  __device__ __forceinline__ T second(const T *f) const {
    T v = r2[0] * f[b2];
#pragma unroll
    for (int j = 1; j < N; ++j) v = fma(r2[j], f[b2 + CurvedTile<N>::FP * j], v);
    return v;
  }
};
template <int N>
constexpr bool kFacePoints = N <= 3;

// Evaluation pass for the cells cell0 .. cell0+ncta-1 of one problem, on a
// thread block of blockDim.x >= ncta * N^2 threads with curved_cell_values
// of shared memory per cell at sm.  Shared by the per-problem and the
// batched kernels.
template <typename T, int N, bool UNSTR = false>
__device__ __forceinline__ void dg_eval_body(const DGArgs<T> &a, const VecPtrs<T> &v, const int cell0, const int ncta, T *sm) {
  using C = CurvedTile<N>;
  using L = CurvedLines<T, N>;
  constexpr int N2 = N * N, N3 = N2 * N, F2 = C::F2;
  const int tid = threadIdx.x, cl = tid / N2, l = tid - cl * N2, la = l % N, lb = l / N;
  const bool act = cl < ncta;
  const int cell = cell0 + (act ? cl : 0);
  T *sc = sm + cl * C::CE, *sf = sc + C::FE, *sg = sf + 6 * F2;
  const L t(sc, la, lb);
  // the face point of the thread's line, in memory and in a face array: faces
  // normal to x, and the others (l, fi)
  const int lx = lb + N * la, fx = lb + C::FP * la, fi = la + C::FP * lb;
  T w[6];   // reference derivative along the normal, per face
  T *tr = v.trace + (size_t)cell * 12 * N2;
  auto ends = [&](const int d, const T (&x)[N]) {
    T v0, v1;
    line_ends<T, N>(x, v0, v1, w[2 * d], w[2 * d + 1]);
    const int f = d ? fi : fx, p = d ? l : lx;
    sf[2 * d * F2 + f] = v0;
    sf[(2 * d + 1) * F2 + f] = v1;
    tr[4 * d * N2 + p] = v0;
    tr[(4 * d + 2) * N2 + p] = v1;
  };
  T x[N];
#pragma unroll
  for (int q = 0; q < N; ++q) x[q] = v.u[(size_t)cell * N3 + l + q * N2];
  curved_interpolate<T, N>(t, act, x);
  if (act) {
    if (!a.recompute) {   // the values at the Gauss points, [cell][x][x-line]
      T *gg = v.grad + (size_t)cell * N3 + l;
#pragma unroll
      for (int q = 0; q < N; ++q) gg[q * N2] = x[q];
    }
    ends(0, x);
    tile_store<T, N, L::ZX>(t.zx, x);
  }
  __syncthreads();
  if (act) {
    tile_load<T, N, L::ZY>(t.zy, x);
    ends(1, x);
    tile_store<T, N, L::XY>(t.xy, x);
  }
  __syncthreads();
  if (act) {
    tile_load<T, N, L::XZ>(t.xz, x);
    ends(2, x);
  }
  __syncthreads();
  if constexpr (!kFacePoints<N>) {
    if (act)
      face_lines<T, N, MD>(l, [&](int f, int) { return sf + f * F2; }, [&](int f, int k) { return sg + (2 * f + k) * F2; });
    __syncthreads();
  }
  if (!act) return;
  int ijk[3] = {0, 0, 0};
  if constexpr (!UNSTR) {
    ijk[0] = cell % a.m[0];
    ijk[1] = (cell / a.m[0]) % a.m[1];
    ijk[2] = cell / (a.m[0] * a.m[1]);
  }
  FacePoint<T, N> fp;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int t1 = d == 0 ? 1 : 0, t2 = d == 2 ? 1 : 2, p = d ? l : lx;
    const T *c0, *c1;   // own side's J^-1 n of the faces xi_d = 0 and xi_d = 1
    if constexpr (UNSTR) {
      c0 = a.fc[0] + ((size_t)cell * 6 + 2 * d) * 3 * N2 + p;
      c1 = c0 + 3 * N2;
    } else {
      const size_t nfp = (size_t)a.m[t1] * a.m[t2];
      const size_t f0 = (size_t)ijk[d] * nfp + ijk[t1] + (size_t)a.m[t1] * ijk[t2];
      const size_t f1 = f0 + nfp;
      c0 = a.fc[d] + (f0 * 2 + 1) * 3 * N2 + p;   // this cell is the upper cell of plane i_d
      c1 = a.fc[d] + (f1 * 2 + 0) * 3 * N2 + p;   // and the lower cell of plane i_d+1
    }
    T g[4];   // tangential derivatives at the two faces' points
    if constexpr (kFacePoints<N>) {
      if (d < 2) fp.template init<false>(d ? la : lb, d ? lb : la);
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        g[2 * s] = fp.first(sf + (2 * d + s) * F2);
        g[2 * s + 1] = fp.second(sf + (2 * d + s) * F2);
      }
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) g[k] = sg[(4 * d + k) * F2 + (d ? fi : fx)];
    }
    tr[(4 * d + 1) * N2 + p] = c0[d * N2] * w[2 * d] + c0[t1 * N2] * g[0] + c0[t2 * N2] * g[1];
    tr[(4 * d + 3) * N2 + p] = c1[d * N2] * w[2 * d + 1] + c1[t1 * N2] * g[2] + c1[t2 * N2] * g[3];
  }
}

// Integration pass (same thread and shared-memory contract as the evaluation).
template <typename T, int N, bool UNSTR = false>
__device__ __forceinline__ void dg_integrate_body(const DGArgs<T> &a, const VecPtrs<T> &v, const int cell0, const int ncta,
                                                  T *sm) {
  using C = CurvedTile<N>;
  using L = CurvedLines<T, N>;
  constexpr int N2 = N * N, N3 = N2 * N, F2 = C::F2;
  const int tid = threadIdx.x, cl = tid / N2, l = tid - cl * N2, la = l % N, lb = l / N;
  const bool act = cl < ncta;
  const int cell = cell0 + (act ? cl : 0);
  T *sc = sm + cl * C::CS, *st = sc + C::F;   // st: tangential test coefficients [face][t1, t2]
  const L t(sc, la, lb);
  const int lx = lb + N * la, fx = lb + C::FP * la, fi = la + C::FP * lb;   // as in the evaluation

  // Face fluxes at the face points of the thread's lines: value coefficient A,
  // normal test coefficient bn, and the tangential ones, which become value
  // coefficients through D^T on the face below (tangential derivatives commute
  // with the extrapolation to the face).
  // (the thread's line of u, or of the stored values, is on its way meanwhile)
  T x[N], A[6], bn[6];
  {
    const T *p = (a.recompute ? v.u : v.grad) + (size_t)cell * N3 + l;
#pragma unroll
    for (int q = 0; q < N; ++q) x[q] = p[q * N2];
  }
  if (act) {
    int i0 = 0, i1 = 0, i2 = 0;
    if constexpr (!UNSTR) {
      i0 = cell % a.m[0];
      i1 = (cell / a.m[0]) % a.m[1];
      i2 = cell / (a.m[0] * a.m[1]);
    }
    const T tau_e = a.tau[cell];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int t1 = d == 0 ? 1 : 0, t2 = d == 2 ? 1 : 2, p = d ? l : lx;
      const int id = d == 0 ? i0 : (d == 1 ? i1 : i2), j1 = d == 0 ? i1 : i0, j2 = d == 2 ? i1 : i2;
      const size_t nfp = (size_t)a.m[t1] * a.m[t2], ftan = j1 + (size_t)a.m[t1] * j2;
      const int cs = d == 0 ? 1 : (d == 1 ? a.m[0] : a.m[0] * a.m[1]);
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const int f = 2 * d + s;
        const T *tr = v.trace + ((size_t)cell * 6 + f) * 2 * N2 + p;
        const T uo = tr[0], qo = tr[N2];
        T dA;
        const T *c, *tn = nullptr;   // own J^-1 n; the neighbour's trace
        T tau_f = tau_e;
        bool dir;
        if constexpr (UNSTR) {
          // neighbour, its local face and the orientation of the shared face
          const size_t cf = (size_t)cell * 6 + f;
          const int2 nf = a.ufn[cf];
          dA = a.fdA[0][cf * N2 + p];
          c = a.fc[0] + cf * 3 * N2 + p;
          if (nf.x >= 0) {
            tn = v.trace + ((size_t)nf.x * 6 + (nf.y & 7)) * 2 * N2 + face_perm<N>(nf.y >> 3, p);
            tau_f = max(tau_e, a.tau[nf.x]);
          }
          dir = nf.x == -1;
        } else {
          const size_t face = (size_t)(id + s) * nfp + ftan;
          dA = a.fdA[d][face * N2 + p];
          c = a.fc[d] + (face * 2 + (s ? 0 : 1)) * 3 * N2 + p;
          if (s ? id < a.m[d] - 1 : id > 0) {
            const int nb = cell + (s ? cs : -cs);
            tn = v.trace + ((size_t)nb * 6 + 2 * d + (1 - s)) * 2 * N2 + p;
            tau_f = max(tau_e, a.tau[nb]);
          }
          dir = a.bc[f] == 0;
        }
        T B;
        if (tn) {
          const T un = tn[0], qn = tn[N2];
          const T jump = uo - un, hdA = T(0.5) * dA;
          A[f] = fma(dA * tau_f, jump, -hdA * (qo - qn));
          B = -hdA * jump;
        } else if (dir) {
          A[f] = fma(T(2) * dA * tau_e, uo, -dA * qo);
          B = -dA * uo;
        } else {
          A[f] = T(0);
          B = T(0);
        }
        bn[f] = c[d * N2] * B;
        st[2 * f * F2 + (d ? fi : fx)] = c[t1 * N2] * B;
        st[(2 * f + 1) * F2 + (d ? fi : fx)] = c[t2 * N2] * B;
      }
    }
  }
  // the x-lines of the values at the Gauss points: again from u (FP32), or as
  // the evaluation stored them; the gradient's x component
  if (a.recompute) {
    curved_interpolate<T, N>(t, act, x);
  }
  FacePoint<T, N> fp;
  // D^T along a line of direction d, with the line's face terms: every point
  // gets l_s(q) times side s's value coefficient and (D^T l_s)(q) times its
  // normal coefficient
  const auto sweep = [&](const int d, const T (&in)[N], T (&out)[N]) {
    if constexpr (kFacePoints<N>) {
      if (d != 1) fp.template init<true>(d ? la : lb, d ? lb : la);   // z, y, then x
    }
    T e[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const T *p = st + (4 * d + 2 * s) * F2;
      if constexpr (kFacePoints<N>) e[s] = A[2 * d + s] + (fp.first(p) + fp.second(p + F2));
      else e[s] = A[2 * d + s] + (p[d ? fi : fx] + p[F2 + (d ? fi : fx)]);
    }
    sweep_with_ends<T, N>(in, e[0], e[1], bn[2 * d], bn[2 * d + 1], out);
  };
  curved_cell_term<T, N>(
      t, act, a.metric + (size_t)cell * 6 * N3 + l, x,
      [&] {   // beside the y-lines: D^T on the faces
        if constexpr (!kFacePoints<N>) {
          const auto same = [&](int f, int k) { return st + (2 * f + k) * F2; };
          face_lines<T, N, MDt>(l, same, same);
        }
      },
      sweep);
  if (act) dg_epilogue<T, N>(a, v, (size_t)cell * N3 + l, N2, T(1), x);
}

// Per-vector pointers of a multi-vector launch: vector r of u, out, x, xp, b
// and its scratch (geometry and inverse diagonal are shared).  A small
// struct of pointers only, so it stays in registers.
template <typename T>
__device__ __forceinline__ VecPtrs<T> vec_ptrs(const DGArgs<T> &a, const int r) {
  const int64_t o = r * a.vs;
  VecPtrs<T> v;
  v.u = a.u + o;
  v.out = a.out + o;
  v.x = a.x ? a.x + o : nullptr;
  v.xp = a.xp ? a.xp + o : nullptr;
  v.b = a.b ? a.b + o : nullptr;
  v.grad = a.grad ? a.grad + r * a.gs : nullptr;
  v.trace = a.trace + r * a.ts;
  return v;
}

// One thread block handles cb consecutive cells of one vector with cb N^2
// threads.  MULTI (several vectors of one operator): block b is cell group
// b / nv of vector b % nv, so the vectors of one group run side by side and
// share its geometry in L2.  The single-vector kernels are compiled apart:
// the per-vector offsets cost registers, which cost resident blocks (the FP32
// integration pass at 16 MDoF ran 14% slower with them).  cb is a launch
// parameter (picked per level and size by the tile-shape autotuner): one
// compiled kernel serves every block width.
// kCurvedThreads bounds a block (wider settings run at this width).
constexpr int kCurvedThreads = 512;
// blocks of kCurvedThreads to leave registers for: FP32 40 (evaluation) and
// 64, FP64 64 at N = 2 and 128
template <typename T, int N, bool INTEGRATE>
constexpr int kCurvedBlocks = sizeof(T) == 8 ? (N == 2 ? 2 : 1) : (INTEGRATE ? 2 : 3);

template <typename T, int N, bool MULTI>
__global__ void __launch_bounds__(kCurvedThreads, kCurvedBlocks<T, N, false>) dg_eval_kernel(const DGArgs<T> a, const int cb) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int grp = MULTI ? blockIdx.x / a.nv : blockIdx.x, vec = MULTI ? blockIdx.x - grp * a.nv : 0;
  const int cell0 = grp * cb;
  dg_eval_body<T, N>(a, vec_ptrs(a, vec), cell0, min(cb, a.ncells - cell0), reinterpret_cast<T *>(smem_raw));
}

template <typename T, int N, bool MULTI>
__global__ void __launch_bounds__(kCurvedThreads, kCurvedBlocks<T, N, true>) dg_integrate_kernel(const DGArgs<T> a, const int cb) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int grp = MULTI ? blockIdx.x / a.nv : blockIdx.x, vec = MULTI ? blockIdx.x - grp * a.nv : 0;
  const int cell0 = grp * cb;
  dg_integrate_body<T, N>(a, vec_ptrs(a, vec), cell0, min(cb, a.ncells - cell0),
                                  reinterpret_cast<T *>(smem_raw));
}

// Axis-aligned cells: one pass; grid x, y, z are the blocks of a.box from oy,
// oz on (MULTI: nz blocks of each vector behind one another).
template <typename T, int N, bool MULTI>
__global__ void __launch_bounds__(kCellThreads) dg_box_kernel(const DGArgs<T> a, const int oy, const int oz,
                                                              const int nz) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int gz = blockIdx.z, vec = 0;
  if constexpr (MULTI) {
    vec = gz / nz;
    gz -= vec * nz;
  }
  dg_box_body<T, N>(a, vec_ptrs(a, vec), a.box, blockIdx.x, oy + blockIdx.y, oz + gz, smem_raw);
}

// Unstructured meshes: single-vector passes with general (curved) cell and
// face geometry and the neighbour of every local face from a.ufn.
template <typename T, int N>
__global__ void __launch_bounds__(kCurvedThreads, kCurvedBlocks<T, N, false>) dg_eval_unstr_kernel(const DGArgs<T> a, const int cb) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int cell0 = blockIdx.x * cb;
  dg_eval_body<T, N, true>(a, vec_ptrs(a, 0), cell0, min(cb, a.ncells - cell0), reinterpret_cast<T *>(smem_raw));
}

template <typename T, int N>
__global__ void __launch_bounds__(kCurvedThreads, kCurvedBlocks<T, N, true>) dg_integrate_unstr_kernel(const DGArgs<T> a,
                                                                                            const int cb) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int cell0 = blockIdx.x * cb;
  dg_integrate_body<T, N, true>(a, vec_ptrs(a, 0), cell0, min(cb, a.ncells - cell0),
                                      reinterpret_cast<T *>(smem_raw));
}

// Diagonal of the DG operator (setup, FP64), one thread per DoF: the cell
// term sum_q grad N_i^T M_q grad N_i and the face self-coupling
// dA (tau N_i^2 - N_i d_n N_i) on interior faces, dA (2 tau N_i^2 - 2 N_i d_n N_i)
// on Dirichlet faces.
struct DiagTabs {
  double S[81], Sd[81], lp0[9], lp1[9];
};

template <int N, bool CURVED>
__global__ void dg_diag_kernel(const DGArgs<double> a, const DiagTabs tb, double *diag) {
  constexpr int N2 = N * N, N3 = N2 * N;
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long)a.ncells * N3) return;
  const int cell = (int)(idx / N3), i = (int)(idx - (long)cell * N3);
  const int ii[3] = {i % N, (i / N) % N, i / N2};
  const int ijk[3] = {cell % a.m[0], (cell / a.m[0]) % a.m[1], cell / (a.m[0] * a.m[1])};
  double sum = 0;
  for (int qz = 0; qz < N; ++qz)
    for (int qy = 0; qy < N; ++qy)
      for (int qx = 0; qx < N; ++qx) {
        const int p = qx + N * qy + N2 * qz;
        const double sx = tb.S[qx * N + ii[0]], sy = tb.S[qy * N + ii[1]], sz = tb.S[qz * N + ii[2]];
        const double g0 = tb.Sd[qx * N + ii[0]] * sy * sz;
        const double g1 = sx * tb.Sd[qy * N + ii[1]] * sz;
        const double g2 = sx * sy * tb.Sd[qz * N + ii[2]];
        if (!CURVED) {
          sum += a.wcart[p] * g0 * g0 + a.wcart[N3 + p] * g1 * g1 + a.wcart[2 * N3 + p] * g2 * g2;
        } else {
          const double *M = a.metric + (size_t)cell * 6 * N3 + p;
          sum += M[0] * g0 * g0 + M[N3] * g1 * g1 + M[2 * N3] * g2 * g2 +
                 2.0 * (M[3 * N3] * g0 * g1 + M[4 * N3] * g0 * g2 + M[5 * N3] * g1 * g2);
        }
      }
  const int cstride[3] = {1, a.m[0], a.m[0] * a.m[1]};
  for (int d = 0; d < 3; ++d) {
    const int t1 = d == 0 ? 1 : 0, t2 = d == 2 ? 1 : 2;
    for (int s = 0; s < 2; ++s) {
      if (ii[d] != (s ? N - 1 : 0)) continue;   // basis vanishes on this face
      const bool has_nb = s ? (ijk[d] < a.m[d] - 1) : (ijk[d] > 0);
      if (!has_nb && a.bc[2 * d + s] != 0) continue;   // Neumann: no term
      const double tau_e = a.tau[cell];
      const double tau_f = has_nb ? fmax(tau_e, a.tau[cell + (s ? cstride[d] : -cstride[d])]) : tau_e;
      const double lp = s ? tb.lp1[ii[d]] : tb.lp0[ii[d]];
      const size_t nfp = (size_t)a.m[t1] * a.m[t2];
      const size_t face = (size_t)(ijk[d] + s) * nfp + ijk[t1] + (size_t)a.m[t1] * ijk[t2];
      for (int q2 = 0; q2 < N; ++q2)
        for (int q1 = 0; q1 < N; ++q1) {
          const int lq = q1 + N * q2;
          const double s1 = tb.S[q1 * N + ii[t1]], s2 = tb.S[q2 * N + ii[t2]];
          const double nv = s1 * s2;
          double dA, dn;
          if (!CURVED) {
            dA = a.fwcart[d * N2 + lq];
            dn = (s ? a.ih[d] : -a.ih[d]) * lp * nv;
          } else {
            dA = a.fdA[d][face * N2 + lq];
            const double *c = a.fc[d] + (face * 2 + (s ? 0 : 1)) * 3 * N2 + lq;
            double gr[3];
            gr[d] = lp * nv;
            gr[t1] = tb.Sd[q1 * N + ii[t1]] * s2;
            gr[t2] = s1 * tb.Sd[q2 * N + ii[t2]];
            dn = c[0] * gr[0] + c[N2] * gr[1] + c[2 * N2] * gr[2];
          }
          if (has_nb)
            sum += dA * (tau_f * nv * nv - nv * dn);
          else
            sum += dA * (2.0 * tau_e * nv * nv - 2.0 * nv * dn);
        }
    }
  }
  diag[idx] = sum;
}

}  // namespace sipg

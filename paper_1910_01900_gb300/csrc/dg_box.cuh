// The SIPG operator on axis-aligned cells in one pass (Section 4; weak form
// Eq. WeakFormDG with the fluxes of Eqs. InteriorPenaltyFlux1/2 and the mirror
// boundary conditions of Eq. BoundaryConditions).
//
// On a box cell every integral is a tensor product, so with the 1D mass matrix
// M of the GL basis under the Gauss rule
//   v = (M x M x M) sum_d M_d^-1 G_d u,
// where G_d acts along the lines of direction d only: for the line x with the
// neighbours' end values un_s and outward end derivatives Qn_s (reference
// coordinates) behind its two ends s
//   G x = alpha_d ( K x + sum_s [ e_s (tau_f h_d (x_s - un_s) - (Q_s - Qn_s)/2)
//                                 - q_s (x_s - un_s)/2 ] ),
// e_s the end's unit vector, q_s the outward derivative row (Q_s = q_s . x),
// alpha_d = prod(h)/h_d^2.  The own parts of the flux are folded into one
// matrix, K' = K - sum_s (e_s q_s^T + q_s e_s^T)/2, and everything is
// multiplied by M^-1 in advance (BoxTables::HE, HO): what is left per line is an
// n x (n + 4) product of (x, r_0, r_1, un_0, un_1) with
// r_s = tau_f h_d (x_s - un_s) + Qn_s/2, in even-odd form.  The mirror
// principle becomes a value of un and Qn: (-x_s, -Q_s) on a Dirichlet side,
// (x_s, Q_s) on a Neumann side.
//
// Cells are worked on in pairs per direction (2 i, 2 i + 1): the far end of a
// line is the one away from the partner.  A cell at an odd position is kept
// mirrored in that direction from its first load to its last store (the 1D
// matrices commute with the reflection), so that the far end is index 0 and
// the near end index n - 1 for every thread: no warp diverges on which
// neighbour is where, which cost the first version of this pass two thirds of
// its instructions.  What lies behind the near end comes from the partner
// through shared memory (two values per line), what lies behind the far end
// from the neighbour's line in memory, or, at the mesh's edge, from the own
// line read from its other end (the mirror image).  Both are the same dot
// product of the same values, so a block may also take single cells (small
// meshes) with the same result.
//
// Up to three points per line M^-1 stays out of it (kBoxDirect): with
//   v = M_z (M_y a + M_x b) + M_y M_x c,   (a, b, c) = (G_x, G_y, G_z) u,
// five mass sweeps instead of three and two more tiles.  M^-1 amplifies the
// parts of a line that M then damps again, by 6 : 2 at two points, and the
// rounding of w between them with it: FP32 error against 64 bits for random
// vectors (relative, 2-norm) at degree 1 / 2 1.2e-7 / 1.9e-7 that way and
// 7.6e-8 / 1.5e-7 this way, where the evaluation at the Gauss points gives
// 9.7e-8 / 1.54e-7 (time at 12 MDoF 69 / 75 us and 78 / 83 us; at the Gauss
// points 245 / 185 us).  From four points on the form with w rounds less than
// the Gauss points do (degree 3 / 5 / 7 1.5e-7 / 1.7e-7 / 1.6e-7, there 1.8e-7 /
// 2.5e-7 / 2.6e-7) and is kept.
//
// Measured at 16 MDoF (GB300) against the two-pass scheme with stored traces
// that axis-aligned cells had before: FP32 k = 3 / 5 / 7 204 / 191 / 165 us ->
// 69 / 71 / 75 us, FP64 k = 3 / 5 / 7 2440 / 2590 / 2860 us -> 1389 / 1495 /
// 1759 us; errors against 64 bits no larger (FP32 k = 7: 1.5e-7, before
// 2.5e-7: fewer roundings, end values read instead of extrapolated).  Now
// FP32 is bound by the L1 data pipe (k = 4: 73% of its wavefronts, 41% shared
// memory, 32% global lines), FP64 by the FP64 pipe (84% busy).
//
// FP32 works on two cells per thread, x neighbours of each other, with packed
// two-wide arithmetic and 8-byte shared-memory accesses: half the
// instructions per value, which is what bounds the FP32 pass.  FP64 is bound
// by the FP64 pipe and works on one cell per thread.
#pragma once
#include "sumfac.cuh"

namespace sipg {

template <typename T>
struct VecPtrs {
  const T *u;
  T *out;
  const T *x, *xp, *b;
  T *grad, *trace;
};

// The outputs of one line of N values (at g0 + q st) from s y, by mode.  What
// the Chebyshev step reads is loaded for the whole line before the first
// store: the output may be one of the inputs' vectors (out = xp), so the
// compiler keeps every load behind the stores before it, and a line would wait
// for memory N times (FP32 32^3 k = 4, one step: 42 us, now 27 us).
template <typename T, int N>
__device__ __forceinline__ void dg_epilogue(const DGArgs<T> &a, const VecPtrs<T> &v, const size_t g0, const int st,
                                            const T s, T (&y)[N]) {
  T *out = v.out + g0;
  if (a.mode == 0) {
#pragma unroll
    for (int q = 0; q < N; ++q) out[q * st] = s * y[q];
    return;
  }
  const T *b = v.b + g0;
  T r[N];
#pragma unroll
  for (int q = 0; q < N; ++q) r[q] = b[q * st];
  if (a.mode == 2) {
#pragma unroll
    for (int q = 0; q < N; ++q) out[q * st] = fma(-s, y[q], r[q]);
    return;
  }
  const T *d = a.dinv + g0;
  T e[N], x[N];
#pragma unroll
  for (int q = 0; q < N; ++q) e[q] = d[q * st];
#pragma unroll
  for (int q = 0; q < N; ++q) x[q] = T(0);
  if (v.x) {
    const T *p = v.x + g0;
#pragma unroll
    for (int q = 0; q < N; ++q) x[q] = a.c1 * p[q * st];
  }
  if (v.xp) {
    const T *p = v.xp + g0;
#pragma unroll
    for (int q = 0; q < N; ++q) x[q] = fma(a.c2, p[q * st], x[q]);
  }
#pragma unroll
  for (int q = 0; q < N; ++q) out[q * st] = fma(a.c3 * e[q], fma(-s, y[q], r[q]), x[q]);
}

// ------------------------------------------------ one or two values per lane
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ double vsub(double a, double b) { return a - b; }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }
// of positive numbers: their order is that of their bits, and integer
// instructions leave the FP64 pipe alone
__device__ __forceinline__ double vmax(double a, double b) {
  return __longlong_as_double(max(__double_as_longlong(a), __double_as_longlong(b)));
}
// -a where s is negative (the sign bit alone: no FP64 instruction)
__device__ __forceinline__ double vsign(double a, bool s) {
  return __longlong_as_double(__double_as_longlong(a) ^ ((long long)s << 63));
}
__device__ __forceinline__ unsigned long long f2_bits(F2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ F2 f2_of(unsigned long long v) {
  F2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ F2 vfma(F2 a, F2 b, F2 c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)), "l"(f2_bits(c)));
  return f2_of(r);
}
__device__ __forceinline__ F2 vadd(F2 a, F2 b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
  return f2_of(r);
}
__device__ __forceinline__ F2 vsub(F2 a, F2 b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
  return f2_of(r);
}
__device__ __forceinline__ F2 vmul(F2 a, F2 b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
  return f2_of(r);
}
__device__ __forceinline__ F2 vmax(F2 a, F2 b) { return F2{fmaxf(a.x, b.x), fmaxf(a.y, b.y)}; }
__device__ __forceinline__ F2 vsign(F2 a, bool s) {
  const unsigned m = (unsigned)s << 31;
  return F2{__uint_as_float(__float_as_uint(a.x) ^ m), __uint_as_float(__float_as_uint(a.y) ^ m)};
}
// Each translation unit owns its copy of the tables (static __constant__).
static __constant__ BoxTables<double> c_box_d;
static __constant__ BoxTables<float> c_box_f;
template <typename V>
struct BoxLane;
template <>
struct BoxLane<F2> {
  using T = float;
  static constexpr bool pair = true;
  static __device__ __forceinline__ F2 all(float a) { return F2{a, a}; }
  static __device__ __forceinline__ const BoxTables<float> &tab() { return c_box_f; }
};
template <>
struct BoxLane<double> {
  using T = double;
  static constexpr bool pair = false;
  static __device__ __forceinline__ double all(double a) { return a; }
  static __device__ __forceinline__ const BoxTables<double> &tab() { return c_box_d; }
};
template <typename T>
static void upload_box_tu(const BoxTables<T> &t) {
  if constexpr (sizeof(T) == 8)
    cudaMemcpyToSymbol(c_box_d, &t, sizeof(t));
  else
    cudaMemcpyToSymbol(c_box_f, &t, sizeof(t));
}

// Shared memory of one cell (FP32: cell pair), in 8-byte values: the tiles of
// u and w (N <= 3: and two more; x fastest, y step XP, z step ZP) and the
// near-end derivatives of two phases.  Pitches chosen per N by counting the wavefronts of the three
// line directions (weighted by their 3, 5 and 3 accesses) over 8 cells: 1.27
// per half-warp at N = 4 (3.18 unpadded), 1.63 at N = 5, 1.64 at N = 6 (1.79),
// 1.57 at N = 7 (1.90), 1.27 at N = 8 (3.36), 1.50 at N = 9.
__host__ __device__ constexpr int box_xp(int n) { return n == 4 ? 5 : n == 8 ? 9 : n; }
__host__ __device__ constexpr int box_zp(int n) {
  return n == 2 ? 6 : n == 3 ? 9 : n == 4 ? 20 : n == 5 ? 25 : n == 6 ? 38 : n == 7 ? 55 : n == 8 ? 72 : 81;
}
__host__ __device__ constexpr int box_group_values(int n) {
  return n == 2 ? 68 : n == 3 ? 139 : n == 4 ? 192 : n == 5 ? 301 : n == 6 ? 532 : n == 7 ? 881 : n == 8 ? 1280 : 1633;
}
// the form without M^-1 (see above; also in the tables, BoxTables)
template <int N>
constexpr bool kBoxDirect = box_direct(N);
// cells that one thread works on
template <typename T>
constexpr int kBoxLanes = sizeof(T) == 4 ? 2 : 1;
// Cells of a block by default.  Swept at 16 MDoF: FP32 wants small blocks
// (one brick of 8 cells from n = 4 on: at n = 5 74.4 us against 79.9 us for
// two), whose barriers hold up few warps; FP64 wants blocks whose threads fill
// whole warps (n = 5: 400 threads in 13 warps 1500 us, 200 in 7 warps 1578 us).
template <typename T>
__host__ __device__ constexpr int box_default_cells(int n) {
  if (sizeof(T) == 4) return n == 2 ? 20 : n == 3 ? 24 : n == 9 ? 4 : 8;
  return n == 2 ? 64 : n == 3 ? 32 : n <= 5 ? 16 : 8;
}
// thread groups (of n^2 threads) of a block
template <typename T>
__host__ __device__ inline int box_groups(const BoxShape &b) {
  return b.bricks * b.w[0] * b.w[1] * b.w[2] / kBoxLanes<T>;
}

template <int N>
struct BoxTile {
  static constexpr int XP = box_xp(N), ZP = box_zp(N), T3 = ZP * N, N2 = N * N;
  static constexpr int Q = (kBoxDirect<N> ? 4 : 2) * T3;
  static constexpr int GS = box_group_values(N);
  static_assert(XP >= N && ZP >= XP * N && GS >= Q + 2 * N2, "box layout overlaps");
};
// position of line l of direction D (l = a + N b over the other two
// directions in increasing order) and its step
template <int N, int D>
__device__ __forceinline__ int box_base(const int l) {
  const int a = l % N, b = l / N;
  return D == 0 ? BoxTile<N>::XP * a + BoxTile<N>::ZP * b : (D == 1 ? a + BoxTile<N>::ZP * b : a + BoxTile<N>::XP * b);
}
template <int N, int D>
__device__ constexpr int box_step() {
  return D == 0 ? 1 : (D == 1 ? BoxTile<N>::XP : BoxTile<N>::ZP);
}

// y = H x + sum_s (E_s r_s + L_s un_s) of one line (see above)
template <typename V, int N>
__device__ __forceinline__ void box_line(const V (&x)[N], const V r0, const V r1, const V un0, const V un1,
                                         V (&y)[N]) {
  constexpr int H = N / 2, HC = (N + 1) / 2;
  const V *__restrict__ E = BoxLane<V>::tab().HE[N - 2], *__restrict__ O = BoxLane<V>::tab().HO[N - 2];
  V e[HC], o[H];
#pragma unroll
  for (int j = 0; j < H; ++j) {
    e[j] = vadd(x[j], x[N - 1 - j]);
    o[j] = vsub(x[j], x[N - 1 - j]);
  }
  if constexpr (N & 1) e[H] = x[H];
  const V rp = vadd(r0, r1), rm = vsub(r0, r1), up = vadd(un0, un1), um = vsub(un0, un1);
#pragma unroll
  for (int i = 0; i < HC; ++i) {
    V se = vmul(E[i * 7], e[0]);
#pragma unroll
    for (int j = 1; j < HC; ++j) se = vfma(E[i * 7 + j], e[j], se);
    se = vfma(E[i * 7 + HC], rp, se);
    se = vfma(E[i * 7 + HC + 1], up, se);
    if (i == N - 1 - i) {
      y[i] = se;
    } else {
      V so = vmul(O[i * 6], o[0]);
#pragma unroll
      for (int j = 1; j < H; ++j) so = vfma(O[i * 6 + j], o[j], so);
      so = vfma(O[i * 6 + H], rm, so);
      so = vfma(O[i * 6 + H + 1], um, so);
      y[i] = vadd(se, so);
      y[N - 1 - i] = vsub(se, so);
    }
  }
}

// y = M x, even-odd
template <typename V, int N>
__device__ __forceinline__ void box_mass(const V (&x)[N], V (&y)[N]) {
  constexpr int H = N / 2, HC = (N + 1) / 2;
  const V *__restrict__ E = BoxLane<V>::tab().ME[N - 2], *__restrict__ O = BoxLane<V>::tab().MO[N - 2];
  V e[HC], o[H];
#pragma unroll
  for (int j = 0; j < H; ++j) {
    e[j] = vadd(x[j], x[N - 1 - j]);
    o[j] = vsub(x[j], x[N - 1 - j]);
  }
  if constexpr (N & 1) e[H] = x[H];
#pragma unroll
  for (int i = 0; i < HC; ++i) {
    V se = vmul(E[i * 5], e[0]);
#pragma unroll
    for (int j = 1; j < HC; ++j) se = vfma(E[i * 5 + j], e[j], se);
    if (i == N - 1 - i) {
      y[i] = se;
    } else {
      V so = vmul(O[i * 4], o[0]);
#pragma unroll
      for (int j = 1; j < H; ++j) so = vfma(O[i * 4 + j], o[j], so);
      y[i] = vadd(se, so);
      y[N - 1 - i] = vsub(se, so);
    }
  }
}

// half the outward derivative of a line at its end n - 1
template <typename V, int N>
__device__ __forceinline__ V box_end(const V (&x)[N]) {
  const V *__restrict__ q = BoxLane<V>::tab().qh[N - 2];
  V v = vmul(q[0], x[0]);
#pragma unroll
  for (int j = 1; j < N; ++j) v = vfma(q[j], x[j], v);
  return v;
}

template <typename V, int N>
__device__ __forceinline__ void box_load(const V *s, const int base, const int step, V (&x)[N]) {
#pragma unroll
  for (int q = 0; q < N; ++q) x[q] = s[base + q * step];
}
template <typename V, int N>
__device__ __forceinline__ void box_store(V *s, const int base, const int step, const V (&x)[N]) {
#pragma unroll
  for (int q = 0; q < N; ++q) s[base + q * step] = x[q];
}
// A line in memory: the values at p0 + q st (FP32: and at p1 + q st1 for the second cell)
template <int N>
__device__ __forceinline__ void box_fetch(const double *p0, const int st0, const double *, int, double (&x)[N]) {
#pragma unroll
  for (int q = 0; q < N; ++q) x[q] = p0[q * st0];
}
template <int N>
__device__ __forceinline__ void box_fetch(const float *p0, const int st0, const float *p1, const int st1, F2 (&x)[N]) {
#pragma unroll
  for (int q = 0; q < N; ++q) x[q] = F2{p0[q * st0], p1[q * st1]};
}

// Where a thread's cell (FP32: cell pair) sits along one direction.
struct BoxDir {
  int p;        // parity: mirrored, the partner is one cell back
  bool far_edge, near_edge;   // the mesh ends there
  bool shared;  // the partner is in the same block
  int cs, gs;   // cells and 8-byte values to the partner
  bool far_dir, near_dir;     // Dirichlet sides
};
template <typename T>
__device__ __forceinline__ BoxDir box_dir(const DGArgs<T> &a, const int d, const int c, const bool shared, const int cs,
                                          const int gs) {
  BoxDir b;
  b.p = c & 1;
  b.far_edge = b.p ? c == a.m[d] - 1 : c == 0;
  b.near_edge = !b.p && c == a.m[d] - 1;
  b.shared = shared;
  b.cs = b.p ? -cs : cs;
  b.gs = b.near_edge ? 0 : (b.p ? -gs : gs);
  b.far_dir = a.bc[2 * d + b.p] == 0;
  b.near_dir = a.bc[2 * d + 1 - b.p] == 0;
  return b;
}
// tau_f h_d, the neighbour's end value and half its outward derivative there, at one end
template <typename V>
struct BoxEnd {
  V t, u, q;
};

// The penalty of the thread's cells.  FP64 reads tau_e h_d of the direction
// (tauh; on the FP64 pipe the products would cost two of its instructions per
// line: 4.1 MDoF of degree 4 410 us with them, now 384 us), FP32 tau_e once for
// the three directions and multiplies (its loads are what it is short of: 16.8
// MDoF of degree 7 74 us, with tauh 80 us).
template <typename V, typename T>
__device__ __forceinline__ V box_tau(const DGArgs<T> &a, const int d, const int cell, const int cell1) {
  if constexpr (BoxLane<V>::pair) return F2{a.tau[cell], a.tau[cell1]};
  else return a.tauh[(size_t)d * a.ncells + cell];
}
// tau_f h_d of the larger of two such penalties
template <typename V, typename T>
__device__ __forceinline__ V box_penalty(const DGArgs<T> &a, const int d, const V t0, const V t1) {
  if constexpr (BoxLane<V>::pair) return vmul(vmax(t0, t1), BoxLane<V>::all(a.hd[d]));
  else return vmax(t0, t1);
}

// The end read from memory: the neighbour dc cells away, whose line (start o0,
// o1 in the two cells, step st) is read towards us, or at an edge the own line.
template <typename T, int N, typename V>
__device__ __forceinline__ void box_outside(const DGArgs<T> &a, const T *u0, const T *u1, const int cell,
                                            const int cell1, const V tau, const int d, const bool edge, const bool neg,
                                            const int dc, const bool rev, const int o0, const int o1, const int st,
                                            BoxEnd<V> &b) {
  V f[N];
  const int c = edge ? 0 : dc, q = rev ? -st : st;
  const ptrdiff_t w = (ptrdiff_t)c * (N * N * N) + (rev ? (N - 1) * st : 0);
  box_fetch<N>(u0 + (w + o0), q, u1 + (w + o1), q, f);
  b.t = box_penalty(a, d, tau, box_tau<V>(a, d, cell + c, cell1 + c));
  b.u = vsign(f[N - 1], edge && neg);
  b.q = vsign(box_end<V, N>(f), edge && neg);
}

// w line along D of the thread's cell: H of the own line and the two ends
template <typename V, int N>
__device__ __forceinline__ void box_flux(const V (&x)[N], const BoxEnd<V> &f, const BoxEnd<V> &n, V (&y)[N]) {
  box_line<V, N>(x, vfma(f.t, vsub(x[0], f.u), f.q), vfma(n.t, vsub(x[N - 1], n.u), n.q), f.u, n.u, y);
}

// One block's cells at block coordinates (bx, gy, gz) (bx counts blocks of
// s.bricks bricks), N^2 threads per cell (FP32: per cell pair),
// box_group_values(N) 8-byte values of shared memory per N^2 threads.
template <typename T, int N>
__device__ __forceinline__ void dg_box_body(const DGArgs<T> &a, const VecPtrs<T> &v, const BoxShape &s, const int bx,
                                            const int gy, const int gz, unsigned char *smem) {
  using V = typename BoxNum<T>::type;
  using L = BoxLane<V>;
  constexpr bool P2 = L::pair;
  constexpr int N2 = N * N, N3 = N2 * N, T3 = BoxTile<N>::T3, GS = BoxTile<N>::GS, Q = BoxTile<N>::Q;
  const int tid = threadIdx.x, g = tid / N2, l = tid - g * N2, la = l % N, lb = l / N;
  // thread group -> place in the brick (1 or 2 cells per direction) and brick
  const int w0 = !P2 && s.w[0] == 2, w1 = s.w[1] == 2, w2 = s.w[2] == 2;
  const int ix = g & w0, iy = (g >> w0) & w1, iz = (g >> (w0 + w1)) & w2, r = g >> (w0 + w1 + w2);
  const int bk = bx * s.bricks + r;
  const int cx = P2 ? 2 * bk : (bk << w0) + ix, cy = (gy << w1) + iy, cz = (gz << w2) + iz;
  const bool act = r < s.bricks && cx < a.m[0] && cy < a.m[1] && cz < a.m[2];
  const int sy = a.m[0], sz = a.m[0] * a.m[1];
  const int cell = act ? cx + sy * cy + sz * cz : 0;
  const bool two = P2 && cx + 1 < a.m[0];   // FP32: the pair's second cell exists (else the first stands in)
  const int cell1 = two ? cell + 1 : cell;
  const BoxDir dx = box_dir(a, 0, cx, w0, 1, GS), dy = box_dir(a, 1, cy, w1, sy, GS << w0),
               dz = box_dir(a, 2, cz, w2, sz, GS << (w0 + w1));
  V *su = reinterpret_cast<V *>(smem) + g * GS, *sw = su + T3, *sq = su + Q + l;
  const T *u0 = v.u + (size_t)cell * N3, *u1 = v.u + (size_t)cell1 * N3;
  // the global offset of coordinate c (in the thread's frame) of a direction of parity p
  auto at = [](const int p, const int c) { return p ? N - 1 - c : c; };
  const int stx = (!P2 && dx.p) ? -1 : 1, sty = dy.p ? -N : N, stz = dz.p ? -N2 : N2;
  const int bxa = P2 ? la : at(dx.p, la), bxb = N - 1 - la;   // x = la in the first and in the second cell
  const int oz = N * at(dy.p, lb) + (dz.p ? (N - 1) * N2 : 0);                    // z-line (x, y) = (la, lb)
  const int oy = N2 * at(dz.p, lb) + (dy.p ? (N - 1) * N : 0);                    // y-line (x, z) = (la, lb)
  const int ox = N * at(dy.p, la) + N2 * at(dz.p, lb);                            // x-line (y, z) = (la, lb)
  V tau;   // the own cells' penalty
  if constexpr (P2) tau = box_tau<V>(a, 0, cell, cell1);

  V x[N], y[N];
  BoxEnd<V> ef, en;
  // both ends of a y- or z-line (and an FP64 x-line) as far as they come from memory
  auto outer = [&](const int d, const BoxDir &b, const int o0, const int o1, const int st) {
    if constexpr (!P2) tau = box_tau<V>(a, d, cell, cell1);
    box_outside<T, N, V>(a, u0, u1, cell, cell1, tau, d, b.far_edge, b.far_dir, -b.cs, b.far_edge, o0, o1, st, ef);
    if (!b.shared)
      box_outside<T, N, V>(a, u0, u1, cell, cell1, tau, d, b.near_edge, b.near_dir, b.cs, !b.near_edge, o0, o1, st, en);
  };
  // the near end from the partner in this block (the own line at an edge)
  auto inner = [&](const int d, const BoxDir &b, const int end, const int q) {
    if (!b.shared) return;
    en.u = vsign(su[b.gs + end], b.near_edge && b.near_dir);
    en.q = vsign(sq[b.gs + q], b.near_edge && b.near_dir);
    const int c = b.near_edge ? 0 : b.cs;
    en.t = box_penalty(a, d, tau, box_tau<V>(a, d, cell + c, cell1 + c));
  };
  // M along the thread's line of a tile, in place
  auto mass_along = [&](V *t, const int base, const int step) {
    V in[N], out[N];
    box_load<V, N>(t, base, step, in);
    box_mass<V, N>(in, out);
    box_store<V, N>(t, base, step, out);
  };
  if (act) {
    box_fetch<N>(u0 + oz + bxa, stz, u1 + oz + bxb, stz, x);
    box_store<V, N>(su, box_base<N, 2>(l), box_step<N, 2>(), x);
    if (dz.shared) sq[0] = box_end<V, N>(x);
    outer(2, dz, oz + bxa, oz + bxb, stz);
  }
  __syncthreads();
  if (act) {   // w = M_z^-1 G_z u / alpha_z (N <= 3: G_z u / alpha_z, and so on)
    inner(2, dz, box_base<N, 2>(l) + (N - 1) * box_step<N, 2>(), 0);
    box_flux<V, N>(x, ef, en, y);
    box_store<V, N>(sw, box_base<N, 2>(l), box_step<N, 2>(), y);
    box_load<V, N>(su, box_base<N, 1>(l), box_step<N, 1>(), x);
    if (dy.shared) sq[N2] = box_end<V, N>(x);
    outer(1, dy, oy + bxa, oy + bxb, sty);
  }
  __syncthreads();
  if (act) {   // + M_y^-1 G_y u
    inner(1, dy, box_base<N, 1>(l) + (N - 1) * box_step<N, 1>(), N2);
    box_flux<V, N>(x, ef, en, y);
    const V c = L::all(a.ralpha[0]);
    V *p = sw + box_base<N, 1>(l);
    if constexpr (kBoxDirect<N>) {   // b, and M_y c
#pragma unroll
      for (int q = 0; q < N; ++q) p[T3 + q * box_step<N, 1>()] = vmul(c, y[q]);
      mass_along(sw, box_base<N, 1>(l), box_step<N, 1>());
    } else {
#pragma unroll
      for (int q = 0; q < N; ++q) p[q * box_step<N, 1>()] = vfma(c, y[q], p[q * box_step<N, 1>()]);
    }
    box_load<V, N>(su, box_base<N, 0>(l), box_step<N, 0>(), x);
    if constexpr (P2) {
      // the far ends lie on both sides of the pair, the near ends are each other's
      V f[N];
      const bool e0 = cx == 0, e1 = !two || cx + 1 == a.m[0] - 1;
      const T *p0 = u0 + ox - (e0 ? 0 : N3), *p1 = u1 + ox + (e1 ? 0 : N3);
      box_fetch<N>(p0 + (e0 ? N - 1 : 0), e0 ? -1 : 1, p1 + (e1 ? 0 : N - 1), e1 ? 1 : -1, f);
      ef.t = box_penalty(a, 0, tau, box_tau<V>(a, 0, cell - !e0, cell1 + !e1));
      ef.q = box_end<V, N>(f);
      const bool n0 = e0 && a.bc[0] == 0, n1 = e1 && a.bc[1] == 0, nn = !two && a.bc[1] == 0;
      ef.u = F2{n0 ? -f[N - 1].x : f[N - 1].x, n1 ? -f[N - 1].y : f[N - 1].y};
      ef.q = F2{n0 ? -ef.q.x : ef.q.x, n1 ? -ef.q.y : ef.q.y};
      const V q = box_end<V, N>(x);
      en.t = vmul(L::all(fmaxf(tau.x, tau.y)), L::all(a.hd[0]));
      en.u = F2{two ? x[N - 1].y : (nn ? -x[N - 1].x : x[N - 1].x), x[N - 1].x};
      en.q = F2{two ? q.y : (nn ? -q.x : q.x), q.x};
    } else {
      if (dx.shared) sq[0] = box_end<V, N>(x);
      outer(0, dx, ox + (dx.p ? N - 1 : 0), 0, stx);
    }
  }
  __syncthreads();
  if (act) {   // + M_x^-1 G_x u, and M_x of the sum
    if constexpr (!P2) inner(0, dx, box_base<N, 0>(l) + N - 1, 0);
    box_flux<V, N>(x, ef, en, y);
    const V c = L::all(a.ralpha[1]);
    if constexpr (kBoxDirect<N>) {   // a, M_x b and M_x M_y c
#pragma unroll
      for (int q = 0; q < N; ++q) y[q] = vmul(c, y[q]);
      box_store<V, N>(sw + 2 * T3, box_base<N, 0>(l), box_step<N, 0>(), y);
      mass_along(sw + T3, box_base<N, 0>(l), box_step<N, 0>());
      mass_along(sw, box_base<N, 0>(l), box_step<N, 0>());
    } else {
      box_load<V, N>(sw, box_base<N, 0>(l), box_step<N, 0>(), x);
#pragma unroll
      for (int q = 0; q < N; ++q) x[q] = vfma(c, y[q], x[q]);
      box_mass<V, N>(x, y);
      box_store<V, N>(sw, box_base<N, 0>(l), box_step<N, 0>(), y);
    }
  }
  __syncthreads();
  if (act) {
    if constexpr (kBoxDirect<N>) {   // M_y a + M_x b
      box_load<V, N>(sw + 2 * T3, box_base<N, 1>(l), box_step<N, 1>(), x);
      box_mass<V, N>(x, y);
      V *p = sw + T3 + box_base<N, 1>(l);
#pragma unroll
      for (int q = 0; q < N; ++q) p[q * box_step<N, 1>()] = vadd(y[q], p[q * box_step<N, 1>()]);
    } else {
      mass_along(sw, box_base<N, 1>(l), box_step<N, 1>());
    }
  }
  __syncthreads();
  if (!act) return;
  box_load<V, N>(kBoxDirect<N> ? sw + T3 : sw, box_base<N, 2>(l), box_step<N, 2>(), x);
  box_mass<V, N>(x, y);
  if constexpr (kBoxDirect<N>) {
    box_load<V, N>(sw, box_base<N, 2>(l), box_step<N, 2>(), x);
#pragma unroll
    for (int q = 0; q < N; ++q) y[q] = vadd(y[q], x[q]);
  }
  // the epilogue, cell by cell
#pragma unroll
  for (int k = 0; k < (P2 ? 2 : 1); ++k) {
    if (k && !two) break;
    T z[N];
#pragma unroll
    for (int q = 0; q < N; ++q) {
      if constexpr (P2) z[q] = k ? y[q].y : y[q].x;
      else z[q] = y[q];
    }
    dg_epilogue<T, N>(a, v, (size_t)(k ? cell1 : cell) * N3 + oz + (k ? bxb : bxa), stz, a.alphaz, z);
  }
}

}  // namespace sipg

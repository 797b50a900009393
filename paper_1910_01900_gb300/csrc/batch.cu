// Many independent SIPG problems (uneven mesh size and degree) or many
// right-hand sides of one problem, solved together.
//
// * The finest-level DG operator of all problems runs as one launch per degree
//   and pass, a block per item of a static list (axis-aligned cells: one pass
//   over the problems' blocks, dg_box.cuh; curved cells: two passes over groups
//   of cells, dg_kernels.cuh); in the captured graphs the degrees' launches are
//   side by side.  The same bodies as the per-problem kernels.
// * The flexible-CG iterations of all problems run in lockstep: batched
//   operator applications, batched inner products and updates (one launch for
//   all problems, deterministic per-problem reductions), and each problem's
//   V-cycle replayed from its CUDA graph on its own stream, so the cycles of
//   different problems overlap on the GPU.
// Not in the paper (its solver handles one problem per run); the method per
// problem is unchanged.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "dg_kernels.cuh"
#include "stride_loop.cuh"

namespace sipg {

constexpr int kBatchThreads = 256;

// this translation unit's copy of the 1D tables (constant memory is per unit)
template <>
void upload_tables_batch<double>(const Tables<double> &t, const BoxTables<double> &bt) {
  upload_tables_tu(t);
  upload_box_tu(bt);
}
template <>
void upload_tables_batch<float>(const Tables<float> &t, const BoxTables<float> &bt) {
  upload_tables_tu(t);
  upload_box_tu(bt);
}

// segs (optional): the flexible-CG systems; a problem whose system has left
// the iteration (segs[p].active == 0, set on the device) is skipped too.
// One kernel per degree, with the register budget of the single-problem
// passes: with every degree's body in one kernel the compiler kept 600 (FP32)
// and 904 bytes (FP64) of the integration pass in local memory.
// One V-cycle of 12 curved problems of 8^3 cells of degree 4 in FP32, FP32 cycle
// of two of 16^3 and 12^3 of degrees 3 and 5: 1006 and 635 us so, now 857 and 551
// us; operator of 16 problems in FP64 2665 us, now 2542 us.
template <typename T, int N, bool INTEGRATE>
__global__ void __launch_bounds__(kBatchThreads, kCurvedThreads / kBatchThreads * kCurvedBlocks<T, N, INTEGRATE>)
    dg_batched_kernel(const BatchProb<T> *__restrict__ probs, const WorkItem *__restrict__ items,
                      const Seg *__restrict__ segs) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *sm = reinterpret_cast<T *>(smem_raw);
  const WorkItem w = items[blockIdx.x];
  const BatchProb<T> &P = probs[w.p];
  if (!P.active || (segs && !segs[w.p].active)) return;
  if constexpr (INTEGRATE) dg_integrate_body<T, N>(P.a, vec_ptrs(P.a, 0), w.cell0, w.ncta, sm);
  else dg_eval_body<T, N>(P.a, vec_ptrs(P.a, 0), w.cell0, w.ncta, sm);
}

// Axis-aligned problems: the one pass of all problems of one degree, a block
// per item (block w.cell0 of problem w.p's mesh, cut by shape, which is the
// plan's whatever the problem's own launches use).  One kernel per degree: with
// every degree's body in one kernel the FP32 pass needed 80 registers and 900
// bytes of stack.
template <typename T, int N>
__global__ void __launch_bounds__(kBatchThreads) dg_box_batched_kernel(const BatchProb<T> *__restrict__ probs,
                                                                       const WorkItem *__restrict__ items,
                                                                       const Seg *__restrict__ segs) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const WorkItem w = items[blockIdx.x];
  const BatchProb<T> &P = probs[w.p];
  if (!P.active || (segs && !segs[w.p].active)) return;
  BoxShape b;
  b.w[0] = (w.ncta & 1) + 1;
  b.w[1] = ((w.ncta >> 1) & 1) + 1;
  b.w[2] = ((w.ncta >> 2) & 1) + 1;
  b.bricks = w.ncta >> 3;
  const int wx = b.w[0] * b.bricks, nx = (P.a.m[0] + wx - 1) / wx, ny = (P.a.m[1] + b.w[1] - 1) / b.w[1],
            r = w.cell0 / nx;
  dg_box_body<T, N>(P.a, vec_ptrs(P.a, 0), b, w.cell0 - r * nx, r % ny, r / ny, smem_raw);
}
static int pack_shape(const BoxShape &b) { return (b.w[0] - 1) | (b.w[1] - 1) << 1 | (b.w[2] - 1) << 2 | b.bricks << 3; }

// shared memory of a block of kBatchThreads / n^2 curved cells
template <typename T>
static size_t curved_batch_smem(int n, bool integrate) {
  return (size_t)(kBatchThreads / (n * n)) * curved_cell_values(n, integrate) * sizeof(T);
}
template <typename T>
static cudaError_t prep_batched() {
  constexpr cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaSuccess;
#define SIPG_BATCH_PREP(NN)                                                                                     \
  for (cudaError_t r : {cudaFuncSetAttribute(dg_box_batched_kernel<T, NN>, at,                                  \
                                             kBatchThreads / (NN * NN) * box_group_values(NN) * 8),             \
                        cudaFuncSetAttribute(dg_batched_kernel<T, NN, false>, at,                               \
                                             (int)curved_batch_smem<T>(NN, false)),                             \
                        cudaFuncSetAttribute(dg_batched_kernel<T, NN, true>, at,                                \
                                             (int)curved_batch_smem<T>(NN, true))})                             \
    if (r != cudaSuccess) e = r;
  SIPG_BATCH_PREP(2)
  SIPG_BATCH_PREP(3)
  SIPG_BATCH_PREP(4)
  SIPG_BATCH_PREP(5)
  SIPG_BATCH_PREP(6)
  SIPG_BATCH_PREP(7)
  SIPG_BATCH_PREP(8)
  SIPG_BATCH_PREP(9)
#undef SIPG_BATCH_PREP
  return e;
}

// Blocks of the batched vector kernels: system p gets g.nb[p] blocks (one
// per kSegChunk entries, at least one), block b works on system g.map[b].x as
// its g.map[b].y-th block, so that a large system gets as many blocks as its
// size asks for and the launch is balanced over the GPU.

__device__ void seg_reduce2(const SegGrid &g, int p, int j, double a, double b, double *partials, unsigned *counter,
                            double *out) {
  // per block partial sums; the last block of the system sums them (each
  // thread a strided part in order, then the same tree: deterministic) and
  // resets the system's counter
  __shared__ double sa[256], sb[256];
  __shared__ bool last;
  const int nb = g.nb[p], off = g.off[p];
  auto tree = [&] {
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
      if (threadIdx.x < w) {
        sa[threadIdx.x] += sa[threadIdx.x + w];
        sb[threadIdx.x] += sb[threadIdx.x + w];
      }
      __syncthreads();
    }
  };
  sa[threadIdx.x] = a;
  sb[threadIdx.x] = b;
  tree();
  if (threadIdx.x == 0) {
    partials[(off + j) * 2] = sa[0];
    partials[(off + j) * 2 + 1] = sb[0];
    __threadfence();
    last = atomicAdd(&counter[p], 1u) == (unsigned)nb - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double ta = 0, tb = 0;
  for (int q = threadIdx.x; q < nb; q += 256) {
    ta += ((volatile double *)partials)[(off + q) * 2];
    tb += ((volatile double *)partials)[(off + q) * 2 + 1];
  }
  sa[threadIdx.x] = ta;
  sb[threadIdx.x] = tb;
  tree();
  if (threadIdx.x == 0) {
    out[0] = sa[0];
    out[1] = sb[0];
    counter[p] = 0;
  }
}

// which: 0 -> (b.b, r.r); 1 -> (r.z, 0); 2 -> (p.v, 0); 3 -> (r.z, z.v)
__global__ void seg_dot_kernel(const Seg *segs, const SegGrid g, int which, double *partials, unsigned *counter,
                               double *sc, int sc_stride, int slot) {
  const int p = g.map[blockIdx.x].x, j = g.map[blockIdx.x].y, nb = g.nb[p];
  const Seg S = segs[p];
  if (!S.active) return;   // whole system inactive: every block of it returns
  double a = 0, b = 0;
  // a = sum u v, b = sum w w' (which 1 and 2: a alone)
  const double *u = which == 0 ? S.b : (which == 2 ? S.p : S.r), *v = which == 0 ? S.b : (which == 2 ? S.v : S.z);
  const double *w = which == 0 ? S.r : S.z, *w2 = which == 0 ? S.r : S.v;
  const bool two = which == 0 || which == 3;
  double ui[kAhead], vi[kAhead], wi[kAhead], xi[kAhead];
  stride_loop(
      (long)j * blockDim.x + threadIdx.x, (long)nb * blockDim.x, S.n,
      [&](int k, long i) {
        ui[k] = u[i];
        vi[k] = v[i];
        wi[k] = two ? w[i] : 0.0;
        xi[k] = two ? w2[i] : 0.0;
      },
      [&](int k, long) {
        a = fma(ui[k], vi[k], a);
        if (two) b = fma(wi[k], xi[k], b);
      });
  seg_reduce2(g, p, j, a, b, partials, counter, sc + (size_t)p * sc_stride + slot);
}

// x += alpha p, r -= alpha v, alpha = sc[0]/sc[2]; sc[3] = r.r
__global__ void seg_update_xr_kernel(const Seg *segs, const SegGrid g, double *partials, unsigned *counter, double *sc,
                                     int sc_stride) {
  const int p = g.map[blockIdx.x].x, j = g.map[blockIdx.x].y, nb = g.nb[p];
  const Seg S = segs[p];
  if (!S.active) return;
  const double *s = sc + (size_t)p * sc_stride;
  const double alpha = s[0] / s[2];
  double a = 0;
  double xi[kAhead], pi[kAhead], vi[kAhead], ri[kAhead];
  stride_loop(
      (long)j * blockDim.x + threadIdx.x, (long)nb * blockDim.x, S.n,
      [&](int k, long i) {
        xi[k] = S.x[i];
        pi[k] = S.p[i];
        vi[k] = S.v[i];
        ri[k] = S.r[i];
      },
      [&](int k, long i) {
        S.x[i] = fma(alpha, pi[k], xi[k]);
        const double r = fma(-alpha, vi[k], ri[k]);
        S.r[i] = r;
        a = fma(r, r, a);
      });
  seg_reduce2(g, p, j, a, 0.0, partials, counter, sc + (size_t)p * sc_stride + 3);
}

// p = z + beta p, beta = -sc[1]/sc[2]; or p = z (init)
__global__ void seg_update_p_kernel(const Seg *segs, const SegGrid g, const double *sc, int sc_stride, int init) {
  const int p = g.map[blockIdx.x].x, j = g.map[blockIdx.x].y, nb = g.nb[p];
  const Seg S = segs[p];
  if (!S.active) return;
  const double *s = sc + (size_t)p * sc_stride;
  const double beta = init ? 0.0 : -s[1] / s[2];
  double pi[kAhead], zi[kAhead];
  stride_loop(
      (long)j * blockDim.x + threadIdx.x, (long)nb * blockDim.x, S.n,
      [&](int k, long i) {
        pi[k] = init ? 0.0 : S.p[i];
        zi[k] = S.z[i];
      },
      [&](int k, long i) { S.p[i] = init ? zi[k] : fma(beta, pi[k], zi[k]); });
}

// ------------------------------------------ lockstep flexible CG gated on the device
// After x += alpha p, r -= alpha v of every active system: count the
// iteration, record ||r||, and take each system out of the iteration on
// convergence (||r|| <= rtol ||r_0||, the host loop's test), breakdown
// (status 1) or maxit (status 2); the next step's condition is 1 while any
// system is still active.  prm = {rtol, maxit} in device memory (the
// captured launch outlives one solve's arguments).  One block; systems
// strided over its threads.
__global__ void batch_fcg_check_kernel(const double *sc, int stride, Seg *segs, int np, int *it, int *status,
                                       double *hist, double *rn, const double *r0, const double *prm, int *any,
                                       cudaGraphConditionalHandle next) {
  const double rtol = prm[0];
  const int maxit = (int)prm[1];
  __shared__ int s_any;
  if (threadIdx.x == 0) s_any = 0;
  __syncthreads();
  int live = 0;
  for (int p = threadIdx.x; p < np; p += blockDim.x) {
    if (!segs[p].active) continue;
    const double *q = sc + (size_t)p * stride;
    const int k = it[p] + 1;
    it[p] = k;
    if (!(q[2] > 0) || !isfinite(q[3])) {
      segs[p].active = 0;
      status[p] = 1;
      continue;
    }
    const double r = sqrt(q[3]);
    rn[p] = r;
    if (k <= 256) hist[(size_t)p * 257 + k] = r;
    if (r <= rtol * r0[p]) {
      segs[p].active = 0;
    } else if (k >= maxit) {
      segs[p].active = 0;
      status[p] = 2;
    } else {
      live = 1;
    }
  }
  if (live) atomicOr(&s_any, 1);
  __syncthreads();
  if (threadIdx.x == 0) {
    *any = s_any;
    cudaGraphSetConditional(next, s_any ? 1u : 0u);
  }
}

__global__ void batch_fcg_cond_kernel(const int *any, cudaGraphConditionalHandle h) {
  cudaGraphSetConditional(h, *any ? 1u : 0u);
}

cudaError_t launch_batch_fcg_check(const double *sc, int stride, Seg *segs, int np, int *it, int *status, double *hist,
                                   double *rn, const double *r0, const double *prm, int *any,
                                   cudaGraphConditionalHandle next, cudaStream_t s) {
  batch_fcg_check_kernel<<<1, 256, 0, s>>>(sc, stride, segs, np, it, status, hist, rn, r0, prm, any, next);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_batch_fcg_cond(const int *any, cudaGraphConditionalHandle h, cudaStream_t s) {
  batch_fcg_cond_kernel<<<1, 1, 0, s>>>(any, h);
  note_launch();
  return cudaGetLastError();
}

// ------------------------------------------------------------------ host side

template <typename T>
cudaError_t batch_plan_build(BatchPlan<T> &P, const std::vector<DGArgs<T>> &args, const std::vector<int> &ns,
                             bool curved) {
  const int np = (int)args.size();
  P.curved = curved;
  P.probs.resize(np);
  P.items.clear();
  P.degrees.clear();
  for (int p = 0; p < np; ++p) {
    P.probs[p].a = args[p];
    P.probs[p].n = ns[p];
    P.probs[p].active = 1;
  }
  for (int n = kMaxN; n >= 2; --n) {   // the degrees' items one after another
    typename BatchPlan<T>::Degree d{n, (int)P.items.size(), 0, 0, {0, 0}};
    for (int p = 0; p < np; ++p) {
      if (ns[p] != n || args[p].ncells == 0) continue;
      if (curved) {
        d.groups = kBatchThreads / (n * n);
        for (int c = 0; c < args[p].ncells; c += d.groups)
          P.items.push_back({p, c, std::min(d.groups, args[p].ncells - c)});
        continue;
      }
      // a default block, as far as kBatchThreads allow
      const int cb = std::min(dg_cells_per_block<T>(n, false), kBatchThreads / (n * n) * kBoxLanes<T>);
      const BoxShape w = dg_box_shape<T>(n, args[p].m, cb);
      int nb = 1;
      for (int e = 0; e < 3; ++e) {
        const int we = w.w[e] * (e == 0 ? w.bricks : 1);
        nb *= (args[p].m[e] + we - 1) / we;
      }
      d.groups = std::max(d.groups, box_groups<T>(w));
      for (int b = 0; b < nb; ++b) P.items.push_back({p, b, pack_shape(w)});
    }
    d.count = (int)P.items.size() - d.first;
    for (int pass = 0; pass < 2; ++pass)
      d.smem[pass] = curved ? curved_batch_smem<T>(n, pass == 1) : (size_t)d.groups * box_group_values(n) * 8;
    if (d.count) P.degrees.push_back(d);
  }
  cudaError_t e;
  if ((e = cudaMalloc(&P.d_probs, np * sizeof(BatchProb<T>))) != cudaSuccess) return e;
  if ((e = cudaMalloc(&P.d_items, std::max<size_t>(1, P.items.size()) * sizeof(WorkItem))) != cudaSuccess) return e;
  if ((e = cudaMemcpy(P.d_items, P.items.data(), P.items.size() * sizeof(WorkItem), cudaMemcpyHostToDevice)) !=
      cudaSuccess)
    return e;
  return prep_batched<T>();
}

template <typename T>
void batch_plan_free(BatchPlan<T> &P) {
  cudaFree(P.d_probs);
  cudaFree(P.d_items);
  P.d_probs = nullptr;
  P.d_items = nullptr;
}

// One degree's items with the descriptors probs (device): the evaluation (pass
// 0) or the integration pass of curved cells, or the one pass of axis-aligned
// cells (1).
template <typename T>
cudaError_t batch_dg_degree(const BatchPlan<T> &P, const typename BatchPlan<T>::Degree &d, const BatchProb<T> *probs,
                            int pass, const Seg *segs, cudaStream_t s) {
  const WorkItem *it = P.d_items + d.first;
  const int threads = d.groups * d.n * d.n;
  switch (d.n) {
#define SIPG_BATCH_CASE(NN)                                                                            \
  case NN:                                                                                             \
    if (!P.curved) dg_box_batched_kernel<T, NN><<<d.count, threads, d.smem[1], s>>>(probs, it, segs);  \
    else if (pass == 0)                                                                                \
      dg_batched_kernel<T, NN, false><<<d.count, threads, d.smem[0], s>>>(probs, it, segs);            \
    else dg_batched_kernel<T, NN, true><<<d.count, threads, d.smem[1], s>>>(probs, it, segs);          \
    break;
    SIPG_BATCH_CASE(2)
    SIPG_BATCH_CASE(3)
    SIPG_BATCH_CASE(4)
    SIPG_BATCH_CASE(5)
    SIPG_BATCH_CASE(6)
    SIPG_BATCH_CASE(7)
    SIPG_BATCH_CASE(8)
    SIPG_BATCH_CASE(9)
#undef SIPG_BATCH_CASE
  }
  note_launch();
  return cudaGetLastError();
}

// ---------------------------------------------- batched vector steps of the V-cycle
// op 0: y (FP32) = x (FP64); 1: y (FP64) = x (FP32); 2: y = c d x in FP32;
// 3: y = c d x in FP64; 4: y = x (FP64).  kBatchNodeThreads entries per item.
__global__ void __launch_bounds__(kBatchNodeThreads)
    vec_batched_kernel(const VecTask *__restrict__ tasks, const NodeItem *__restrict__ items,
                       const Seg *__restrict__ segs) {
  const NodeItem w = items[blockIdx.x];
  if (segs && !segs[w.p].active) return;
  const VecTask &V = tasks[w.p];
  const long i = (long)w.blk * kBatchNodeThreads + threadIdx.x;
  if (i >= V.n) return;
  switch (V.op) {
    case 0:
      ((float *)V.y)[i] = (float)((const double *)V.x)[i];
      break;
    case 1:
      ((double *)V.y)[i] = (double)((const float *)V.x)[i];
      break;
    case 2: {
      const float c = (float)V.c;
      ((float *)V.y)[i] = c * ((const float *)V.d)[i] * ((const float *)V.x)[i];
      break;
    }
    case 3:
      ((double *)V.y)[i] = V.c * ((const double *)V.d)[i] * ((const double *)V.x)[i];
      break;
    default:
      ((double *)V.y)[i] = ((const double *)V.x)[i];
  }
}

cudaError_t launch_vec_batched(const VecTask *tasks, const NodeItem *items, int nitems, const Seg *segs,
                               cudaStream_t s) {
  if (nitems <= 0) return cudaSuccess;
  vec_batched_kernel<<<nitems, kBatchNodeThreads, 0, s>>>(tasks, items, segs);
  note_launch();
  return cudaGetLastError();
}

template cudaError_t batch_plan_build<double>(BatchPlan<double> &, const std::vector<DGArgs<double>> &,
                                              const std::vector<int> &, bool);
template cudaError_t batch_plan_build<float>(BatchPlan<float> &, const std::vector<DGArgs<float>> &,
                                             const std::vector<int> &, bool);
template void batch_plan_free<double>(BatchPlan<double> &);
template void batch_plan_free<float>(BatchPlan<float> &);
template cudaError_t batch_dg_degree<double>(const BatchPlan<double> &, const BatchPlan<double>::Degree &,
                                             const BatchProb<double> *, int, const Seg *, cudaStream_t);
template cudaError_t batch_dg_degree<float>(const BatchPlan<float> &, const BatchPlan<float>::Degree &,
                                            const BatchProb<float> *, int, const Seg *, cudaStream_t);

cudaError_t seg_dot(const Seg *segs, const SegGrid &g, int which, double *partials, unsigned *counter, double *sc,
                    int sc_stride, int slot, cudaStream_t s) {
  if (g.blocks <= 0) return cudaSuccess;
  seg_dot_kernel<<<g.blocks, 256, 0, s>>>(segs, g, which, partials, counter, sc, sc_stride, slot);
  note_launch();
  return cudaGetLastError();
}
cudaError_t seg_update_xr(const Seg *segs, const SegGrid &g, double *partials, unsigned *counter, double *sc,
                          int sc_stride, cudaStream_t s) {
  if (g.blocks <= 0) return cudaSuccess;
  seg_update_xr_kernel<<<g.blocks, 256, 0, s>>>(segs, g, partials, counter, sc, sc_stride);
  note_launch();
  return cudaGetLastError();
}
cudaError_t seg_update_p(const Seg *segs, const SegGrid &g, const double *sc, int sc_stride, int init, cudaStream_t s) {
  if (g.blocks <= 0) return cudaSuccess;
  seg_update_p_kernel<<<g.blocks, 256, 0, s>>>(segs, g, sc, sc_stride, init);
  note_launch();
  return cudaGetLastError();
}

// The block map of systems of sizes n; device arrays appended to allocs.
cudaError_t seg_grid_build(const std::vector<long> &n, SegGrid &g, std::vector<void *> &allocs) {
  std::vector<int2> map;
  std::vector<int> off, nb;
  for (size_t p = 0; p < n.size(); ++p) {
    const long k = std::max<long>(1, (n[p] + kSegChunk - 1) / kSegChunk);
    off.push_back((int)map.size());
    nb.push_back((int)k);
    for (long j = 0; j < k; ++j) map.push_back(make_int2((int)p, (int)j));
  }
  g.blocks = (int)map.size();
  int2 *dm = nullptr;
  int *doff = nullptr, *dnb = nullptr;
  cudaError_t e = cudaMalloc(&dm, std::max<size_t>(1, map.size()) * sizeof(int2));
  if (e == cudaSuccess) allocs.push_back(dm);
  if (e == cudaSuccess && (e = cudaMalloc(&doff, std::max<size_t>(1, off.size()) * sizeof(int))) == cudaSuccess)
    allocs.push_back(doff);
  if (e == cudaSuccess && (e = cudaMalloc(&dnb, std::max<size_t>(1, nb.size()) * sizeof(int))) == cudaSuccess)
    allocs.push_back(dnb);
  if (e == cudaSuccess) e = cudaMemcpy(dm, map.data(), map.size() * sizeof(int2), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(doff, off.data(), off.size() * sizeof(int), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(dnb, nb.data(), nb.size() * sizeof(int), cudaMemcpyHostToDevice);
  g.map = dm;
  g.off = doff;
  g.nb = dnb;
  return e;
}

}  // namespace sipg

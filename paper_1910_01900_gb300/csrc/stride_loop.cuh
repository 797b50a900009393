// Strided loops of the vector kernels.
#pragma once

namespace sipg {

// Entries i0, i0 + step, ... below n, kAhead per turn: load(k, i) of all of
// them before store(k, i) of the first.  The stores may alias the loads, so the
// compiler moves no load ahead of one, and the accumulation of a dot product
// keeps few loads in flight; with one entry a turn a thread waits for memory
// once per entry (FP32 cast_xdb on 4.1 M entries 22 us, FP64 dot products of
// 0.9 M entries 10 us).  The order of the entries, and so of a sum, is the
// plain loop's.
constexpr int kAhead = 4;
template <typename Load, typename Store>
__device__ __forceinline__ void stride_loop(const long first, const long step, const long n, Load load, Store store) {
  for (long i0 = first; i0 < n; i0 += kAhead * step) {
#pragma unroll
    for (int k = 0; k < kAhead; ++k)
      if (i0 + k * step < n) load(k, i0 + k * step);
#pragma unroll
    for (int k = 0; k < kAhead; ++k)
      if (i0 + k * step < n) store(k, i0 + k * step);
  }
}
// over the whole grid
template <typename Load, typename Store>
__device__ __forceinline__ void stride_loop(const long n, Load load, Store store) {
  stride_loop((long)blockIdx.x * blockDim.x + threadIdx.x, (long)gridDim.x * blockDim.x, n, load, store);
}

}  // namespace sipg

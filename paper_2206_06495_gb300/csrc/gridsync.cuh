// Grid-wide barrier and reductions of the resident (cooperative) kernels.
#pragma once

#include "common.cuh"

namespace rbffd {

constexpr int kPT = 1024;      // threads per block, one block per SM
constexpr int kPW = kPT / 32;  // warps per block
constexpr int kNVMax = 4;      // values reduced together
constexpr long long kPolls = 1ll << 22;  // bounded barrier wait (a phase takes microseconds)

// The block's share of the grid-wide machinery.  Every block sees the same
// totals, so every block takes the same decisions.
struct Grid {
  double* sh;              // [kNVMax][kPT]
  double* part;            // [kNVMax][4]
  int* ok;                 // shared: the last barrier's verdict
  double* partials;
  unsigned int* arrivals;
  unsigned int target = 0;
  int phase = 0;

  // All blocks' writes before it are visible to all blocks after it.  Returns
  // false (in every thread of the block) if the other blocks did not arrive
  // within the bounded wait.
  __device__ __forceinline__ bool sync() {
    __syncthreads();
    target += gridDim.x;
    if (threadIdx.x == 0) {
      __threadfence();
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(arrivals) : "memory");
      unsigned int got;
      long long polls = 0;
      do {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(got) : "l"(arrivals) : "memory");
      } while ((int)(got - target) < 0 && ++polls < kPolls);
      __threadfence();
      *ok = (int)(got - target) >= 0;
    }
    __syncthreads();
    return *ok != 0;
  }

  // sync() and the grid-wide sums of NV values per thread, handed to fin(sums)
  // in thread 0 of every block; what fin leaves in shared memory is visible to
  // the block afterwards.  Only the first `active` threads (a multiple of 32)
  // hold values.  The threads store their values and 4 NV warps add them: a
  // butterfly in each of the 32 warps would issue five FP64 adds per value and
  // warp, and the FP64 pipe retires one warp-wide instruction in 16 cycles
  // (which is why the scalars are one thread's work, too).
  template <int NV, typename Fin>
  __device__ __forceinline__ bool reduce(const double (&v)[NV], int active, Fin fin) {
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    if (t < active) {
#pragma unroll
      for (int j = 0; j < NV; ++j) sh[j * kPT + t] = v[j];
    }
    __syncthreads();
    if (w < 4 * NV) {
      const int j = w >> 2, q = w & 3;
      double a = 0.0;
#pragma unroll
      for (int u = 0; u < kPW / 4; ++u) {
        const int e = (q + 4 * u) * 32;
        if (e < active) a += sh[j * kPT + e + lane];
      }
      if (q * 32 < active) a = warp_sum(a);
      if (lane == 0) part[j * 4 + q] = a;
    }
    __syncthreads();
    double* mine = partials + (size_t)(phase & 1) * kNVMax * gridDim.x;
    ++phase;
    if (t < NV) {
      const double* q = part + t * 4;
      mine[t * gridDim.x + blockIdx.x] = (q[0] + q[1]) + (q[2] + q[3]);
    }
    if (!sync()) return false;
    if (w == 0) {
      double a[NV];
#pragma unroll
      for (int j = 0; j < NV; ++j) a[j] = 0.0;
      for (int b = lane; b < (int)gridDim.x; b += 32) {
#pragma unroll
        for (int j = 0; j < NV; ++j) a[j] += mine[j * gridDim.x + b];
      }
#pragma unroll
      for (int j = 0; j < NV; ++j) a[j] = warp_sum(a[j]);
      if (lane == 0) fin(a);
    }
    __syncthreads();
    return true;
  }
};

}  // namespace rbffd

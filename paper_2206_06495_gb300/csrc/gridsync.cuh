// Grid-wide barrier and reductions of the resident (cooperative) kernels.
#pragma once

#include "common.cuh"

namespace rbffd {

constexpr int kNVMax = 4;  // values reduced together, where a kernel does not say otherwise
// bounded barrier wait (a phase takes microseconds), where a test does not
// lower it through rbffd_debug_set_barrier_limit
constexpr long long kPolls = 1ll << 22;
// The barrier's three words, `arrivals`: blocks arrived, blocks that have left
// (see leave()), and 1 once a block has given up a wait.

// The block's share of the grid-wide machinery.  Every block sees the same
// totals, so every block takes the same decisions.
// PT threads per block, one block per SM; at most NVM values reduced together.
template <int PT, int NVM = kNVMax>
struct Grid {
  double* sh;              // [NVM][PT]
  double* part;            // [NVM][4]
  int* ok;                 // shared: the last barrier's verdict
  double* partials;
  unsigned int* arrivals;
  long long limit;  // polls of a wait
  unsigned int target = 0;
  int phase = 0;

  // All blocks' writes before it are visible to all blocks after it.  Returns
  // false (in every thread of the block) if the other blocks did not arrive
  // within the bounded wait.  The block then sets arrivals[2]: at the last
  // barrier of a kernel the others may have passed.
  __device__ __forceinline__ bool sync() {
    __syncthreads();
    target += gridDim.x;
    if (threadIdx.x == 0) {
      // release and acquire order the whole block's accesses, through the
      // block barriers on both sides; a fence of its own on each side cost
      // another 0.4 us a barrier
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(arrivals) : "memory");
      unsigned int got;
      long long polls = 0;
      do {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(got) : "l"(arrivals) : "memory");
      } while ((int)(got - target) < 0 && ++polls < limit);
      *ok = (int)(got - target) >= 0;
      if (!*ok) arrivals[2] = 1u;
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
      for (int j = 0; j < NV; ++j) sh[j * PT + t] = v[j];
    }
    __syncthreads();
    for (int jq = w; jq < 4 * NV; jq += PT / 32) {
      const int j = jq >> 2, q = jq & 3;
      double a = 0.0;
#pragma unroll
      for (int u = 0; u < PT / 128; ++u) {
        const int e = (q + 4 * u) * 32;
        if (e < active) a += sh[j * PT + e + lane];
      }
      if (q * 32 < active) a = warp_sum(a);
      if (lane == 0) part[j * 4 + q] = a;
    }
    __syncthreads();
    double mine = 0.0;
    if (t < NV) {
      const double* q = part + t * 4;
      mine = (q[0] + q[1]) + (q[2] + q[3]);
    }
    return spread<NV>(mine, fin);
  }

  // The second half of reduce(): the block's sum j is in thread j.
  template <int NV, typename Fin>
  __device__ __forceinline__ bool spread(double sum, Fin fin) {
    const int t = threadIdx.x, lane = t & 31;
    double* mine = partials + (size_t)(phase & 1) * NVM * gridDim.x;
    ++phase;
    if (t < NV) mine[t * gridDim.x + blockIdx.x] = sum;
    if (!sync()) return false;
    if (t < 32) {
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

// A thread's share of a sum over its rows.  FP32 values are added as an
// unevaluated pair (Knuth's two-sum), exact to 2^-40 for the 13 rows a thread
// has at most, so that the sum over a grid is as good as one whose FP32 shares
// are single rows; FP64 additions would take the pipe that retires one warp in
// 16 cycles.  The intrinsics keep the compiler from fusing a product into the
// additions.
template <typename T>
struct Part {
  double s = 0.0;
  __device__ __forceinline__ void add(double v) { s += v; }
  __device__ __forceinline__ double value() const { return s; }
};
template <>
struct Part<float> {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float v) {
    const float t = __fadd_rn(hi, v), b = __fsub_rn(t, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, b)), __fsub_rn(v, b)));
    hi = t;
  }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// Ends a kernel whose arrival counter the next launch finds at zero again: the
// last block to come here resets it.
__device__ __forceinline__ void leave(unsigned int* arrivals) {
  __syncthreads();
  if (threadIdx.x == 0 && atomicAdd(arrivals + 1, 1u) == gridDim.x - 1u) {
    arrivals[0] = 0u;
    arrivals[1] = 0u;
  }
}

}  // namespace rbffd

// A barrier over all CTAs of a cooperative launch, with a bounded wait.
//
// For loops whose steps depend on one another and are too short for a launch each
// (pivoted Cholesky, Jacobi rotations): a step of a few microseconds costs one
// barrier (about 1.5 us over 152 CTAs) instead of three launches.
#pragma once

#include <cuda_runtime.h>

namespace dsrg {

// Device words of a barrier, zeroed by the host before the launch.
struct GridBar {
  unsigned count;  // arrivals, all generations
  int abort;       // set when a wait ran out
};

constexpr unsigned long long GRID_WAIT_NS = 2000000000ull;

// All threads of all CTAs call it; writes before it are visible after it. `gen` counts
// this CTA's barriers (starts at 0). False (in every thread of the CTA) if a wait ran
// out somewhere: the caller returns. The grid must be co-resident (cooperative launch).
__device__ __forceinline__ bool grid_barrier(GridBar* b, unsigned& gen) {
  __shared__ int sh_ok;
  __syncthreads();
  ++gen;
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(&b->count, 1u);
    const unsigned want = gen * gridDim.x;
    unsigned long long t0 = 0;
    int ok = 1;
    for (unsigned spins = 0;; ++spins) {
      unsigned c;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(&b->count) : "memory");
      if ((int)(c - want) >= 0) break;
      if ((spins & 63u) == 63u) {
        unsigned long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t0 == 0) t0 = t;
        if (*(volatile int*)&b->abort || t - t0 > GRID_WAIT_NS) {
          atomicExch(&b->abort, 1);
          ok = 0;
          break;
        }
      }
    }
    __threadfence();
    sh_ok = ok;
  }
  __syncthreads();
  return sh_ok != 0;
}

// CTAs of `threads` threads that fit the device at once, at most `want`.
template <typename K>
inline int coop_grid(K kernel, int threads, size_t smem, int want) {
  int dev = 0, nsm = 0, per = 0;
  cudaGetDevice(&dev);
  if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem) != cudaSuccess)
    return 0;
  const int fit = nsm * per;
  return want < fit ? want : fit;
}

}  // namespace dsrg

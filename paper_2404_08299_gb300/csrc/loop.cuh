// The grid barrier of the persistent loop kernels (sweep.cu, ppr.cu).
#pragma once

#include "internal.cuh"

namespace prdf {

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// Barrier over the whole (co-resident) grid: every block adds one arrival and
// waits until all of this barrier's are in. The wait is bounded: past the
// limit (minutes; no sweep takes that long) the block flags the loop as timed
// out and gives up, and so does every other block when it sees the flag.
// Returns false after a timeout.
constexpr unsigned long long kSpinLimit = 1ull << 28;

__device__ inline bool grid_barrier(LoopCtl* ctl, unsigned long long& target) {
  __shared__ int s_ok;
  target += gridDim.x;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(&ctl->bar, 1ull);
    int ok = 1;
    unsigned long long spins = 0;
    while (ld_acquire(&ctl->bar) < target) {
      if (++spins > kSpinLimit || ((spins & 1023) == 0 && *(volatile int*)&ctl->timeout)) {
        *(volatile int*)&ctl->timeout = 1;
        ok = 0;
        break;
      }
      if (spins > 256) __nanosleep(100);
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// Cooperative launch of a loop kernel. Where fewer blocks fit than the device's
// attributes say (a share of the GPU's SMs), it takes as many as do: the
// kernels work with any number.
inline int launch_coop(const void* k, int64_t blocks, int threads, void** args, cudaStream_t s) {
  for (;;) {
    const cudaError_t e = cudaLaunchCooperativeKernel(k, dim3((unsigned)blocks), dim3((unsigned)threads), args, 0, s);
    if (e != cudaErrorCooperativeLaunchTooLarge || blocks <= 1) {
      PRDF_CUDA(e);
      return PRDF_OK;
    }
    cudaGetLastError();
    blocks /= 2;
  }
}

}  // namespace prdf

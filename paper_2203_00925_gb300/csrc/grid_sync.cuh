// Grid-wide barrier of the library's cooperative kernels, with bounded waits.
#pragma once

#include <cuda_runtime.h>

#include "internal.h"

namespace fvgb {

constexpr unsigned long long kBarrierTimeoutNs = 1000000000ull;   // default wait limit

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Grid barrier on a monotone arrival counter with a bounded wait: the r-th barrier of a
// launch is passed once the counter (zeroed before the launch) reaches r * nblocks, so
// the last arrival itself releases the waiting blocks (no reset, no second word). One thread
// of the block arrives (release: what the block wrote before the preceding __syncthreads is
// visible with it), one warp waits (acquire). Measured over 152 blocks: 2,280 cycles a
// barrier; slots polled by every block instead of the counter 3,400 (one to a 128-byte line)
// to 10,900 (packed): stores to a line that is being polled are slow.
__device__ __forceinline__ void grid_arrive(Barrier* bar) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&bar->count) : "memory");
}
__device__ __forceinline__ unsigned count_acquire(const Barrier* bar) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&bar->count) : "memory");
  return v;
}
// False when the wait ran out, here or (status, the launch's common word) in another block; a
// whole warp calls.
__device__ __forceinline__ bool grid_wait(const Barrier* bar, int* status, unsigned target,
                                          unsigned long long limit_ns) {
  if ((int)(count_acquire(bar) - target) >= 0) return true;
  const unsigned long long t0 = global_ns();
  for (int spin = 1;; ++spin) {
    if ((int)(count_acquire(bar) - target) >= 0) return true;
    if ((spin & 15) != 0) continue;
    bool late = *(volatile int*)status != 0;
    if (!late && global_ns() - t0 > limit_ns) {
      late = true;
      if ((threadIdx.x & 31) == 0) atomicExch(status, 1);
    }
    if (__any_sync(0xffffffffu, late)) return false;
  }
}

// A value that other blocks wrote before the last grid barrier: a plain load that may hit L1 (an
// acquire in every barrier orders it behind the other blocks' stores), never moved across one.
__device__ __forceinline__ float load_synced(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ double load_synced(const double* p) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}

}  // namespace fvgb

// Grid-wide barrier with a bounded wait, for kernels launched with
// cudaLaunchCooperativeKernel (every CTA resident at once).
//
// The arrival counter only grows during a launch: barrier k completes when it
// reaches (k + 1) * gridDim.x.  The host zeroes it, stream-ordered, before each
// launch.  Arrival is a release add at GPU scope after a CTA barrier (which
// the release is cumulative over); the wait is an acquire load at GPU scope
// followed by a CTA barrier, so every write of every CTA before the barrier is
// visible to every thread after it.
//
// The wait ends after kBarrierTimeoutNs of global time (counted from its 64th
// poll) or kBarrierMaxSpins polls, whichever comes first.  The first polls
// follow one another without a sleep: most waits end within them.  The CTA that gives up stores RIX_ETIMEOUT in
// the job's status word and the barrier returns false; a CTA that sees a
// non-zero status while waiting gives up at once.  Callers return on false.
#pragma once

#include <cuda_runtime.h>

#include "../../include/rix.h"

namespace rix {

constexpr unsigned long long kBarrierTimeoutNs = 2000000000ull;   // 2 s
constexpr unsigned int kBarrierMaxSpins = 1u << 26;

struct GridBarrier {
  unsigned int* count;   // zeroed before the launch
  int* status;           // the job's device status word (0 = fine)
  unsigned int target;   // per-CTA copy: arrivals the next barrier waits for
};

__device__ __forceinline__ unsigned int ld_acquire_gpu(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void red_release_gpu_add(unsigned int* p, unsigned int v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// polls *p until it reaches `target` (bounded, see above); false when the wait
// gave up.  One thread per CTA.
__device__ __forceinline__ bool poll_counter(const unsigned int* p, unsigned int target, int* status) {
  unsigned int spins = 0;
  unsigned long long t0 = 0;
  while (ld_acquire_gpu(p) < target) {
    if ((++spins & 63u) == 0) {
      if (*reinterpret_cast<volatile int*>(status) != 0) return false;
      const unsigned long long t = global_ns();
      if (t0 == 0) t0 = t;
      if (spins >= kBarrierMaxSpins || t - t0 > kBarrierTimeoutNs) {
        atomicCAS(status, 0, RIX_ETIMEOUT);
        return false;
      }
    }
    if (spins > 16) __nanosleep(32);
  }
  return true;
}

__device__ __forceinline__ bool grid_barrier(GridBarrier& b) {
  __shared__ int ok;
  __syncthreads();
  b.target += gridDim.x;
  if (threadIdx.x == 0) {
    red_release_gpu_add(b.count, 1u);
    ok = poll_counter(b.count, b.target, b.status);
  }
  __syncthreads();
  return ok != 0;
}

}  // namespace rix

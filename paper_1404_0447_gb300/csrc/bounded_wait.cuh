// Waits of a CTA on counters that other CTAs of the same launch advance, bounded in
// time: when one runs out, the launch's abort flag is set, every other wait returns
// at once, and pselinv_sync_status reports it.
#pragma once

#include <cuda_runtime.h>

namespace psi {

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Thread 0 waits until *ctr >= target (device-scope acquire), bounded by
// limit_ns and by *abort, polled every nap_ns; returns false for the whole CTA on
// timeout or abort.
__device__ inline bool cta_wait(const int* ctr, int target, long long limit_ns, int* abort, unsigned nap_ns = 200) {
  __shared__ int ok;
  if (threadIdx.x == 0) {
    ok = 1;
    volatile const int* abort_flag = abort;
    const unsigned long long t0 = global_ns();
    for (;;) {
      if (*abort_flag) {
        ok = 0;
        break;
      }
      if (atomicAdd(const_cast<int*>(ctr), 0) >= target) break;
      if ((long long)(global_ns() - t0) > limit_ns) {
        atomicExch(abort, 1);  // timeout: abort the launch
        ok = 0;
        break;
      }
      __nanosleep(nap_ns);
    }
    __threadfence();
  }
  __syncthreads();
  const int r = ok;
  __syncthreads();
  return r != 0;
}

// Publish a finished task: all threads' writes, then a device-scope fence,
// then the counter.
__device__ inline void cta_signal(int* ctr) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(ctr, 1);
  }
}

}  // namespace psi

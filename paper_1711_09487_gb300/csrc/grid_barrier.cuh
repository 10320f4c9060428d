// Barrier among the CTAs of a cooperative launch (all of them resident), with a bounded wait.
#pragma once
#include "common.cuh"

namespace rfdd {

constexpr int GRID_SPIN = 1 << 22;

// Every CTA adds one to *cnt (zero before the launch) and waits until it has reached target, the number of CTAs
// times the number of barriers so far.  What any thread of a CTA wrote before is visible to all threads
// after it (global loads of other CTAs' data through L2).  false: the wait ran out.  A flag per CTA that
// every other CTA polls, in place of the counter, made a step of 152 CTAs 2.5 us longer.  polls: reads of the counter
// before a CTA gives up; one that does has already been counted, so the others pass this barrier and give up at the next.
__device__ __forceinline__ bool grid_barrier(unsigned *cnt, unsigned target, int polls = GRID_SPIN) {
  __shared__ int ok_s;
  __syncthreads();
  if (threadIdx.x == 0) {
    // the release is cumulative over what __syncthreads has ordered before it
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(cnt) : "memory");
    unsigned v = 0;
    int k = 0;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(cnt) : "memory");
    } while (v < target && ++k < polls);
    ok_s = v >= target;
  }
  __syncthreads();
  return ok_s != 0;
}

// CTAs of a cooperative launch: want of them, or half as many until the device has room for all at once (a process may be
// held to fewer SMs than the device attribute says); 0 when not even least fit.  launch(ctas) returns the launch's
// error.  A refused launch is a host-side error; nothing has run then.
template <typename L>
int cooperative_launch(int want, int least, L &&launch) {
  for (int n = want;; n = n / 2 > least ? n / 2 : least) {
    const cudaError_t e = launch(n);
    if (e == cudaErrorCooperativeLaunchTooLarge) {
      cudaGetLastError();
      if (n <= least) return 0;
      continue;
    }
    RFDD_CUDA(e);
    RFDD_CHECK_LAUNCH();
    return n;
  }
}

}  // namespace rfdd

// grid_sync.cuh -- a bounded barrier over all CTAs of a cooperative launch,
// used by the kernels that run several dependent phases (or whole steps) in
// one launch.
//
// The barrier is one counter in device memory, zero before the launch: a CTA's
// k-th arrival adds one and waits until k times the number of CTAs have
// arrived.  The counter is both what the arrivals write and what the waiting
// CTAs read (with acquire loads, which leave it in L2 and do not queue behind
// the arrivals as atomic reads do), so the last arrival releases everyone
// without a second word.  With 608 CTAs a barrier with a counter and a
// generation word, polled by atomics with a sleep between polls, cost 2.6 to
// 3.6 us; this one
// takes about 0.7 us less (the learned step, seven barriers: 75.8 -> 73.6 us at
// 256^2, 46.4 -> 41.1 at 32^2).
// A wait is bounded by about one second of %globaltimer: a CTA that gives up
// sets STATUS_TIMEOUT in *status and leaves, and every CTA leaves at its next
// barrier, so the launch ends instead of hanging.
#pragma once

#include "hydro_device.cuh"

namespace gh {

__device__ __forceinline__ unsigned long long global_timer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Barrier of all nblocks CTAs of the launch; false (on every thread of the
// CTA) if this CTA gave up waiting here or at an earlier barrier.  passed
// counts the barriers this CTA has been through (zero at launch).
__device__ inline bool grid_barrier(unsigned* count, unsigned nblocks, unsigned& passed, unsigned* status,
                                    bool& failed) {
  __syncthreads();
  if (threadIdx.x == 0 && !failed) {
    passed += 1u;
    const unsigned target = passed * nblocks;  // compared modulo 2^32
    __threadfence();                           // this CTA's writes before the arrival
    atomicAdd(count, 1u);
    unsigned seen;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(count) : "memory");
    if ((int)(seen - target) < 0) {
      const unsigned long long t0 = global_timer_ns();
      for (;;) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(count) : "memory");
        if ((int)(seen - target) >= 0) break;
        if (global_timer_ns() - t0 > 1000000000ull) {
          failed = true;
          atomicOr(status, STATUS_TIMEOUT);
          break;
        }
      }
    }
    __threadfence();  // the others' writes after the release
  }
  return __syncthreads_or(failed ? 1 : 0) == 0;
}

}  // namespace gh

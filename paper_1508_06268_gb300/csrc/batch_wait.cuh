// Bounded wait of an item of the batched kernel for its realization's interval before.
#pragma once
#include <cstdint>

#include "kernels_bits.cuh"

namespace rfim {

// Limit of the wait for `iv` intervals, in polls of at least 200 ns: more than they can take (a sweep of an item is
// far below 1 ms per replica).
__device__ __forceinline__ unsigned long long interval_polls(const SlotCtl &ctl, uint32_t iv, int gact) {
  return (1ull << 22) + (unsigned long long)iv * ctl.nsw * gact * 4096ull;
}

// Waits until the realization has completed `iv` intervals of this launch, with at most `polls` polls.  On
// expiry, or after another CTA's, the error word is set and the item is left out.
__device__ __forceinline__ bool await_interval(const SlotCtl *ctl, uint32_t iv, unsigned long long polls, unsigned *err) {
  for (unsigned long long n = 0; n < polls; ++n) {
    uint32_t done;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(done) : "l"(&ctl->done) : "memory");
    if (done >= iv) return true;
    if (*(volatile unsigned *)err & 2u) return false;
    __nanosleep(200);
  }
  atomicOr(err, 2u);
  return false;
}

}  // namespace rfim

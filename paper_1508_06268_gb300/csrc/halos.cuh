// Halo exchange between the slabs of a cluster: pushes of end planes counted by mbarriers, bounded
// waits for them, and an end of the launch that is safe also when a wait was given up.
//
// Push number h of a CTA goes into the halo planes of both neighbours (rank - 1 and rank + 1) and is
// counted by their mbarrier h & 1, phase h >> 1: the receiver expects the bytes of both neighbours with
// its only arrival of that phase, which it makes with its own push h.  A CTA makes push h only after
// all its waits for phase h - 1, i.e. for both neighbours' push h - 1, have ended well.  So
//   - the phase before on the same mbarrier (push h - 2) is complete when a CTA arrives for push h, and
//   - neighbours' numbers of pushes differ by at most one.
// A CTA in which a wait was given up stops as a whole: the thread sets a flag before the barrier that ends
// the half-sweep, the threads that push read it after, and from then on the CTA neither pushes nor
// arrives; all its threads leave the sweeps at the end of one, and the launch at the next exchange step.
// halo_leave then lets the cluster agree, and every CTA waits for exactly the pushes its neighbours made
// before it exits.
#pragma once
#include <cstdint>

#include "kernels_bits.cuh"

namespace rfim {

// Polls of a halo wait.  The CTAs of a cluster run in step, a push apart at most, and a half-sweep of a
// slab takes below 0.2 ms.
constexpr unsigned kMbarSpinLimit = 1u << 20;

// Waits of a CTA that were given up.  Half-sweeps (or tile visits) alternate between two flags: a thread that
// reads one late, just before the next barrier, must not see what others set in the half-sweep after.
// (L = 32, R = 70: 1.20 us per half-sweep, 1.18 with waits whose end nobody looks at; the flag read by every
// thread instead took 1.25, __syncthreads_or instead of the flags 1.28.)
struct GaveUp {
  uint32_t sweep[2], exchange;
};

struct HaloBars {
  uint64_t mbar[2];
  uint32_t bytes;    // of a push to one neighbour
  uint32_t pushed;   // pushes this CTA has made
  uint32_t stopped;  // a CTA of the cluster has given up a wait
};

__device__ __forceinline__ uint32_t mapa_shared(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

__device__ __forceinline__ uint32_t halo_bar(const HaloBars *hb, uint32_t h) {
  return (uint32_t)__cvta_generic_to_shared(hb->mbar) + 8u * (h & 1u);
}

// By one thread, before the cluster barrier that precedes the first push.
__device__ __forceinline__ void halo_init(HaloBars *hb, uint32_t bytes) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n\tmbarrier.init.shared::cta.b64 [%1], 1;" ::"r"(halo_bar(hb, 0)),
               "r"(halo_bar(hb, 1))
               : "memory");
  hb->bytes = bytes;
  hb->pushed = hb->stopped = 0u;
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Waits until the phase of parity `par` of an mbarrier of this CTA is complete, with at most `polls` polls.
// Gives up (false) after that, with bit 1 set in *err, or when *err already reports something.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t par, unsigned polls, unsigned *err) {
  for (unsigned it = 0; it < polls; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(mbar), "r"(par)
        : "memory");
    if (done) return true;
    if (err && (it & 63u) == 63u && *(volatile unsigned *)err) return false;
  }
  if (err) atomicOr(err, 2u);
  return false;
}

// Waits for both neighbours' push number h.
__device__ __forceinline__ bool halo_wait(const HaloBars *hb, uint32_t h, unsigned *err) {
  return mbar_wait(halo_bar(hb, h), (h >> 1) & 1u, kMbarSpinLimit, err);
}

// After the barrier that ends a half-sweep (tile visit), by the threads that push: whether they may, i.e. no wait of
// the CTA for the push before was given up (flag `f` of the two), nor one earlier: who sees a flag set sets
// the other one for the next time.
__device__ __forceinline__ bool halo_may_push(volatile GaveUp *g, int f) {
  if (g->sweep[f] == 0u) return true;
  g->sweep[f ^ 1] = 1u;
  return false;
}

// This CTA's arrival for push number h, `bytes` from both neighbours together (one thread).
__device__ __forceinline__ void halo_arrive(const HaloBars *hb, uint32_t h, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(halo_bar(hb, h)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void halo_expect(HaloBars *hb, uint32_t h, uint32_t bytes) {
  *(volatile uint32_t *)&hb->pushed = h + 1;
  halo_arrive(hb, h, bytes);
}

// 16 bytes of push number h to where `to` lies in CTA `peer`.
__device__ __forceinline__ void halo_store(const HaloBars *hb, uint32_t h, const void *to, uint32_t peer, uint4 x) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
                   mapa_shared((uint32_t)__cvta_generic_to_shared(to), peer)),
               "r"(x.x), "r"(x.y), "r"(x.z), "r"(x.w), "r"(mapa_shared(halo_bar(hb, h), peer))
               : "memory");
}

// Waits for the pushes that are still on their way to this CTA, which has made `mine`, its neighbours
// `below` and `above` (`bytes` each per push).  One thread, when no CTA of the cluster pushes any more.
// Bytes that were expected but never sent are taken off the phase, and a push this CTA never expected
// is expected now, so each wait ends with the last byte that was sent.
__device__ __forceinline__ void halo_drain(const HaloBars *hb, uint32_t mine, uint32_t below, uint32_t above, uint32_t bytes) {
  for (uint32_t back = mine < 2u ? mine : 2u;; --back) {
    const uint32_t p = mine - back;
    const uint32_t sent = bytes * (((int32_t)(below - p) > 0) + ((int32_t)(above - p) > 0));
    if (back == 0u) {
      if (sent == 0u) return;
      halo_arrive(hb, p, sent);
    } else if (sent < 2u * bytes) {
      asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(halo_bar(hb, p)), "r"(2u * bytes - sent)
                   : "memory");
    }
    if (!halo_wait(hb, p, nullptr) || back == 0u) return;
  }
}

// A wait of this CTA was given up (any thread, any number of them, before it leaves): every CTA of the cluster
// will know in halo_leave.
__device__ __forceinline__ void halo_give_up(HaloBars *hb) {
  const uint32_t flag = (uint32_t)__cvta_generic_to_shared(&hb->stopped);
  for (uint32_t q = 0; q < cluster_ctas(); ++q)
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(mapa_shared(flag, q)), "r"(1u) : "memory");
}

// End of a launch of slabs: all threads of all CTAs of the cluster call it after their last wait.  No CTA exits
// while a push to it is on its way.  What only the path after a given-up wait needs is in shared memory or read
// from the hardware again (kept in registers through the sweeps it cost 2 % at L = 40 on bytes), and the path
// of every other launch is the barrier and one load: a CTA barrier to gather the threads' flags took a call of
// two sweeps at L = 20, R = 5 on bytes from 9.4 to 10.3 us.
__device__ __forceinline__ void halo_leave(HaloBars *hb) {
  sync_slabs<2>();
  volatile HaloBars *own = hb;
  if (own->stopped == 0u) return;  // every wait of the cluster was served
  if (threadIdx.x == 0) {
    const uint32_t rank = cluster_rank(), S = cluster_ctas();
    halo_drain(hb, own->pushed, dsmem_load(&hb->pushed, (rank + S - 1) % S), dsmem_load(&hb->pushed, (rank + 1) % S), own->bytes);
  }
  __syncwarp();
  sync_slabs<2>();
}

}  // namespace rfim

// Persistent-style batched kernel: a fixed grid of CTAs pulls work items (replica groups of
// resident realizations) from a device queue and runs one exchange interval per item with the
// same device function as the single-realization launch (kernels_bits.cuh, one slab per
// replica).  The last item of each realization takes its exchange step and advances the
// realization's counters on the device.  Realizations never interact: each one's arithmetic, partial
// sums and decisions are those of a solo run with the same replica grouping.
//
// A launch takes K intervals of every realization without a barrier between them: the queue holds
// the items of interval 0, then those of interval 1, and so on, and an item of interval i waits until
// its own realization has completed i intervals.  All of that realization's items of interval i - 1
// come earlier in the queue, so they are held by running CTAs and every wait ends; with enough
// realizations they are long done.  One launch per interval instead leaves the SMs idle while the last
// items of each interval finish: 24 mixed realizations have 2.8 rounds of items per interval, and 200
// sweeps of them take 36.6 ms of device time instead of 39.5 (four intervals per launch).
#include "batch.h"
#include "batch_wait.cuh"

namespace rfim {

namespace {

template <int L, int GT>
__device__ __forceinline__ void run_item(const SlotDesc &sd, const BatchItem &bi, SlotCtl *ctl) {
  ExchArgs xa = sd.xa;
  xa.enabled = 1;
  xa.j = ctl->j;
  xa.measure_from = ctl->measure_from;
  xa.expected = (unsigned)sd.nitems;
  xa.ctl = ctl;
  const uint32_t sweep0 = ctl->sweep0;
  const int nsw = ctl->nsw;
  const PhiloxKeys keys = philox_keys(sd.v.seed, sd.v.realization);
  if (sd.kind == kBimodal)
    bits_interval<L, 1, GT, true, true>(sd.v, sd.G, bi.r0, bi.gact, 0, sweep0, nsw, sd.field4, xa, keys);
  else
    bits_interval<L, 1, GT, false, true>(sd.v, sd.G, bi.r0, bi.gact, 0, sweep0, nsw, sd.field4, xa, keys);
}

__global__ void __launch_bounds__(kBatchThreads) k_batch_bits(const SlotDesc *__restrict__ slots, SlotCtl *ctls, int nslots,
                                                              const BatchItem *__restrict__ items, BatchQueue *q,
                                                              int intervals, unsigned *err) {
  __shared__ int s_item;
  const int nitems = q->nitems;
  const unsigned total = (unsigned)nitems * (unsigned)intervals;
  for (;;) {
    if (threadIdx.x == 0) {
      const unsigned n = atomicAdd(&q->head, 1u);
      int item = -1;  // -1: the queue is empty, -2: nothing to do for this entry
      if (n < total) {
        const unsigned iv = n / (unsigned)nitems;
        item = (int)(n % (unsigned)nitems);
        const SlotCtl *ctl = ctls + items[item].slot;
        // finished realizations idle until they are retired
        if ((int)iv >= ctl->left0 || (iv > 0 && !await_interval(ctl, iv, interval_polls(*ctl, iv, items[item].gact), err))) item = -2;
      }
      s_item = item;
    }
    __syncthreads();
    const int it = s_item;
    __syncthreads();
    if (it == -1) break;
    if (it < 0) continue;
    const BatchItem bi = items[it];
    SlotCtl *ctl = ctls + bi.slot;
    const SlotDesc &sd = slots[bi.slot];
    switch (sd.L * 4 + sd.GT) {
      case 64 * 4 + 1: run_item<64, 1>(sd, bi, ctl); break;
      case 64 * 4 + 2: run_item<64, 2>(sd, bi, ctl); break;
      case 32 * 4 + 1: run_item<32, 1>(sd, bi, ctl); break;
      case 32 * 4 + 2: run_item<32, 2>(sd, bi, ctl); break;
      case 16 * 4 + 1: run_item<16, 1>(sd, bi, ctl); break;
      case 8 * 4 + 1: run_item<8, 1>(sd, bi, ctl); break;
      default: break;
    }
  }
  if (threadIdx.x == 0) {
    __threadfence();
    s_item = atomicAdd(&q->done_ctas, 1u) == gridDim.x - 1;
    __threadfence();
  }
  __syncthreads();
  if (!s_item) return;
  if (threadIdx.x == 0) {
    q->head = 0u;
    q->done_ctas = 0u;
  }
  for (int i = threadIdx.x; i < nslots; i += blockDim.x) {  // the next launch starts from here
    ctls[i].left0 = __ldcg(&ctls[i].intervals_left);
    ctls[i].done = 0u;
  }
}

}  // namespace

bool batch_supported(int L, int GT) {
  switch (L) {
    case 64: return GT == 1 || GT == 2;
    case 32: return GT == 1 || GT == 2;
    case 16: return GT == 1;
    case 8: return GT == 1;
    default: return false;
  }
}

int batch_max_gt(int L) { return (L == 64 || L == 32) ? 2 : 1; }

size_t batch_smem(int L, int G) { return (size_t)G * 2 * ((size_t)L * L * L / 64) * 4 + tab_bytes(G); }

cudaError_t batch_prepare(size_t smem) {
  return raise_smem_limit((const void *)k_batch_bits, smem);
}

cudaError_t batch_occupancy(size_t smem, int *blocks_per_sm) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_batch_bits, kBatchThreads, smem);
}

cudaError_t launch_batch(int grid, size_t smem, const SlotDesc *slots, SlotCtl *ctls, int nslots, const BatchItem *items,
                         BatchQueue *queue, int intervals, unsigned *err, cudaStream_t st) {
  k_batch_bits<<<grid, kBatchThreads, smem, st>>>(slots, ctls, nslots, items, queue, intervals, err);
  return cudaGetLastError();
}

}  // namespace rfim

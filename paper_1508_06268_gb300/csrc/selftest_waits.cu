// Device self-tests of the bounded waits inside launches (rfim_selftest_waits): one thread, one wait.
#include <cstring>

#include "rfim.h"
#include "batch_wait.cuh"
#include "exchange_records.cuh"
#include "halos.cuh"

namespace {

using namespace rfim;

struct WaitWords {
  uint4 rec;
  SlotCtl ctl;
  unsigned err;
};

__global__ void k_selftest_waits(WaitWords *w, int which, unsigned limit, int set) {
  __shared__ __align__(8) HaloBars hb;
  if (threadIdx.x != 0) return;
  if (which == 0) {
    halo_init(&hb, 0u);
    if (set) halo_expect(&hb, 0, 0);  // the only arrival, no bytes: phase 0 is complete
    mbar_wait(halo_bar(&hb, 0), 0u, limit, &w->err);
  } else if (which == 1) {
    int B, M;
    long long F;
    if (set) record_store(&w->rec, 1u, -5, 3, -7);
    if (record_await(&w->rec, 1u, &w->err, &B, &M, &F, limit) && (B != -5 || M != 3 || F != -7)) atomicOr(&w->err, 1u);
  } else {
    if (set) w->ctl.done = 1u;
    await_interval(&w->ctl, 1u, limit, &w->err);
  }
}

}  // namespace

extern "C" int rfim_selftest_waits(int32_t which, int32_t spin_limit, int32_t set_flag) {
  if (which < 0 || which > 2 || spin_limit < 1 || spin_limit > (1 << 20)) return RFIM_EINVAL;
  WaitWords *d = nullptr, h;
  memset(&h, 0, sizeof h);
  if (cudaMalloc(&d, sizeof h) != cudaSuccess) return RFIM_ECUDA;
  cudaError_t e = cudaMemcpy(d, &h, sizeof h, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_selftest_waits<<<1, 32>>>(d, which, (unsigned)spin_limit, set_flag);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(&h, d, sizeof h, cudaMemcpyDeviceToHost);
  cudaFree(d);
  if (e != cudaSuccess) return RFIM_ECUDA;
  return h.err & 2u ? RFIM_ETIMEOUT : h.err ? RFIM_EBOUNDS : RFIM_OK;
}

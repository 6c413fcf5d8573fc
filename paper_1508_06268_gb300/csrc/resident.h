// Launch shape and launcher of the resident sweep kernel (kernels_resident.cuh).
#pragma once
#include <cstdint>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "internal.h"
#include "kernels_resident.cuh"

namespace rfim {

// Exchange intervals one launch takes at most (the host regains control between launches).
constexpr int64_t kResidentIntervals = 512;

// Most sweeps (multi-hit: passes) of an interval that ends with the exchange step in the same launch.  The
// clusters run an interval independently and then wait for each other's energies, at most kRecordSpinLimit polls
// (3.4 s measured, 1.2 s at the least): a cluster of one replica beside one of twenty at L = 64 waits 0.18 ms
// per sweep.  Longer intervals are swept by a launch in which no cluster waits for another, and the exchange
// step takes a launch of its own, some 5 us more after 0.3 ms or longer.
constexpr int64_t kResidentSweeps = 2048;

struct ResidentShape {
  // slabs, replicas per cluster, Philox blocks per item (0: the kernel on bytes), threads per CTA
  int32_t S = 0, G = 0, NB = 0, threads = 0;
  bool one = true;  // one item per thread (else a thread may run several)
  int32_t T = 0;    // tile edge of the multi-hit double checkerboard (0: the plain checkerboard)
  size_t smem = 0;
};

using ResidentFn = void (*)(RealView, ResidentArgs, uint32_t, int32_t, const float4 *, ExchArgs);

struct ResidentInstance {
  int32_t L, S, NB, NT;
  bool one;  // one item per thread
  int32_t T;
  ResidentFn bim, flt;
};

template <int L, int S, int NB, int NT, bool ONE, int T = 0>
constexpr ResidentInstance resident_instance() {
  return {L, S, NB, NT, ONE, T, k_resident<L, S, NB, true, NT, ONE, T>, k_resident<L, S, NB, false, NT, ONE, T>};
}

// The instance that measures the structure factor too (kernels_resident_xi.cu), or null.
ResidentFn resident_xi_kernel(int32_t L, int32_t S, int32_t NB, bool one, bool bimodal);
// Whether launches of shape s for up to R replicas can measure it: the instance exists and its CTAs fit.
bool resident_xi_fits(int32_t L, int32_t R, bool bimodal, const ResidentShape &s);

// The multi-hit instances (kernels_resident_mh.cu).
const std::vector<ResidentInstance> &resident_multihit_instances();

// The shape with the lowest estimated half-sweep time (in cycles) for R replicas of edge L among the
// instances whose CTAs are all resident at once; false when there is none.  T: tile edge of the
// multi-hit double checkerboard (then the time of a pass), 0: plain.
bool resident_shape(int32_t L, int32_t R, bool bimodal, ResidentShape *out, double *cycles, int32_t T = 0);
// One shape per instance that fits R replicas, for the launch-shape tuner.
std::vector<ResidentShape> resident_shapes(int32_t L, int32_t R, bool bimodal);
// Whether the instance exists and all CTAs of R replicas are resident at once; fills s->smem.
bool resident_fits(int32_t L, int32_t R, bool bimodal, ResidentShape *s);
// CTAs of (kernel, clusters of S, threads, shared memory) resident at once on the current device.
int resident_ctas(const void *fn, int S, int threads, size_t smem);
constexpr size_t kOneCtaSmem = 116 * 1024;  // more than half an SM's shared memory: one CTA per SM

// Launch configuration of `clusters` clusters of shape s; cooperative when the CTAs wait for one
// another (the exchange step of more than one cluster).
struct ResidentLaunch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  ResidentLaunch(int clusters, const ResidentShape &s, bool exchange, cudaStream_t st);
  ResidentLaunch(const ResidentLaunch &) = delete;
};

// Estimated times (us) of the two ways to run a realization of the plan on bytes: a resident launch (a half-sweep,
// the launch itself with the lattice's way in and out, the tail of an interval), or a launch per half-sweep and
// two per exchange step.
struct BytesCosts {
  double half = 0.0, launch = 0.0, tail = 0.0, half_apart = 0.0, step_apart = 0.0;
};

// The same on bytes (kernels_bytes.cuh): realizations of the int8 layout at other even L.
bool bytes_shape(int32_t L, int32_t R, bool bimodal, ResidentShape *out, double *cycles);
cudaError_t launch_resident_bytes(const RealView &v, const ResidentShape &s, const ResidentArgs &args, uint32_t sweep0,
                                  int32_t n_sweeps, const ExchArgs &xa, cudaStream_t st);
cudaError_t launch_resident(const RealView &v, const ResidentShape &s, const ResidentArgs &args, uint32_t sweep0,
                            int32_t n_sweeps, const float4 *field4, const ExchArgs &xa, cudaStream_t st);

}  // namespace rfim

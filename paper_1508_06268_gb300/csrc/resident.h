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

struct ResidentShape {
  int32_t S = 0, G = 0, NB = 0, threads = 0;  // slabs, replicas per cluster, Philox blocks per item, threads per CTA
  bool one = true;  // one item per thread (else a thread may run several)
  size_t smem = 0;
};

// The shape with the lowest estimated half-sweep time (in cycles) for R replicas of edge L among the
// instances whose CTAs are all resident at once; false when there is none.
bool resident_shape(int32_t L, int32_t R, bool bimodal, ResidentShape *out, double *cycles);
// One shape per instance that fits R replicas, for the launch-shape tuner.
std::vector<ResidentShape> resident_shapes(int32_t L, int32_t R, bool bimodal);
// Whether the instance exists and all CTAs of R replicas are resident at once; fills s->smem.
bool resident_fits(int32_t L, int32_t R, bool bimodal, ResidentShape *s);
cudaError_t launch_resident(const RealView &v, const ResidentShape &s, const ResidentArgs &args, uint32_t sweep0,
                            int32_t n_sweeps, const float4 *field4, const ExchArgs &xa, cudaStream_t st);

}  // namespace rfim

// Launch plan and launcher of the bit-layout sweep kernel.
#pragma once
#include <cstdint>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "internal.h"
#include "resident.h"

namespace rfim {

struct FieldQuant;  // kernels_bits.cuh

// How one realization is mapped onto CTAs: a cluster of S CTAs (z slabs of L/S planes each)
// holds G replicas; every thread updates a word of the slab for GT of them at once (so one field
// load serves GT replicas).  Grid = ceil(R / G) clusters.  S == 0 selects the grid-wide
// cooperative kernel (kernels_grid.cuh): groups of 4 replicas, planes spread over one CTA per SM.
struct BitsPlan {
  int32_t L = 0, S = 1, G = 1, GT = 1, threads = 256;
  size_t smem = 0;
  int32_t Rcap = 0;
  float4 *field4 = nullptr;  // float path: hh as float4 per (colour, word, chunk), see kernels_bits.cu
  // float path: fixed-point field of the energy tail (flimb_index layout) and its exponent/sum
  uint4 *flimb = nullptr;
  FieldQuant *fquant = nullptr;
  // fused exchange tail: per-(replica, slab) partials and the arrival counter
  long long *partB = nullptr, *partM = nullptr, *partFi = nullptr;
  double *partF = nullptr;
  unsigned int *counter = nullptr;
  // grid-wide plan (S == 0): per-(replica, slab) partials, per-CTA progress words, SM count
  long long *gpartB = nullptr, *gpartM = nullptr, *gpartFi = nullptr;
  double *gpartF = nullptr;
  unsigned int *prog = nullptr;
  uint32_t *gbits = nullptr;  // int8 layout on the grid-wide plan: published end planes as bits
  // progress count the grid-wide kernel's words held when the next launch starts (each launch
  // adds its half-sweeps, so no launch has to zero them first)
  mutable uint32_t prog_base = 0;
  mutable uint32_t arrive_base = 0;  // the same for the arrival count of the exchange steps (counter[2])
  int32_t sms = 0;
  bool i8 = false;  // the realization is stored in the int8 layout and staged as bits (cluster shapes)
  int32_t NS = 1;   // 4: every word split over four warps, one block pair each (small lattices)
  // resident plan (kernels_resident.cuh): its shape (threads > 0 when it is the plan), the energy
  // records and the number of the last exchange interval that has been launched
  ResidentShape res;
  uint4 *rec = nullptr;
  size_t rec_slots = 0;  // records of one interval the array holds (two intervals)
  mutable uint32_t epoch = 0;
  SelftestStop stop{-1, 0};  // self-test: where the resident launches give up a wait
  ResidentShape mh_res;  // resident shape of the multi-hit sweeps in force (threads > 0 when they have one)
  bool resident() const { return res.threads > 0; }
  bool xi = false;  // plain resident launches can measure the structure factor (XiWork)
  bool measures_xi(int32_t mh) const { return xi && mh == 0; }
  // whether n sweeps and the exchange step after them are launches of their own
  bool sweeps_apart(int64_t n, int32_t mh) const {
    return (mh > 0 ? mh_res.threads > 0 : resident()) && n > kResidentSweeps / (mh > 1 ? mh : 1);
  }
  BytesCosts cost;  // plan on bytes only
  // Whether k intervals of n sweeps, each with an exchange step or without, are faster in a launch per
  // half-sweep and step than in one resident launch: short calls of large lattices, whose way into shared
  // memory and out again is not paid back, and lattices that few CTAs hold.
  bool faster_apart(int64_t n, int64_t k, bool exchange) const {
    if (cost.half <= 0.0) return false;
    const double one = cost.launch + k * (2.0 * n * cost.half + (exchange ? cost.tail : 0.0));
    // (estimates: where they are close the resident launch stands, of runs, whose tails the estimate puts too
    // high, more so)
    const double close = n > 0 && exchange ? 0.88 : n > 0 ? 0.92 : 0.95;
    return k * (2.0 * n * cost.half_apart + (exchange ? cost.step_apart : 0.0)) < close * one;
  }
  // exchange intervals one launch takes at most (mh passes per visit; 0: plain sweeps)
  int64_t max_intervals(int32_t mh) const {
    if (mh > 0) return mh_res.threads > 0 && mh < kResidentIntervals ? kResidentIntervals / mh : 1;
    return resident() ? kResidentIntervals : S == 0 ? 64 : 1;
  }
};

// Multi-hit double 3D checkerboard (Sec. 3.2, kernels_mh.cuh): mh local passes per tile visit
// (0: the plain checkerboard), tiles of edge `tile` (8, 16 or 32, dividing L / 2; the kernel is
// instantiated per tile edge).
struct MultiHit {
  int32_t mh = 0, tile = 0;
};

// Workspace of the structure factor measured inside resident launches: marginals and the replica at
// every temperature of up to `intervals` exchange intervals (0: not allocated).  A launch fills in its
// intervals `first` and later; which those are is decided once, on the host (its step numbers have 64 bits).
struct XiWork {
  int32_t *marg = nullptr, *t2r = nullptr;
  int32_t intervals = 0, first = 0;
};
// Whether tiles of edge `tile` are supported at L; the setting for (L, mh, tile).
bool multihit_tile_ok(int32_t L, int32_t tile);
MultiHit make_multihit(int32_t L, int32_t mh, int32_t tile);
// Whether the plan's shape has a multi-hit instance; sets its launch attributes.
cudaError_t prepare_multihit(const BitsPlan &plan, bool bimodal);
// Gives the plan a resident shape for multi-hit sweeps with tiles of edge `tile`, beside its shape for
// plain sweeps; *found is false when there is none or the cluster kernel is expected to be faster.
cudaError_t prepare_multihit_resident(BitsPlan &plan, bool bimodal, int32_t tile, cudaStream_t st, bool *found);

bool bits_supported(int32_t L);
// Launch-shape tuner support: a thread-local candidate shape for the next make_bits_plan, the
// remembered best shape per (L, R, field kind), and the candidates instantiated for each L.
void set_plan_override(const char *plan);
void remember_tuned_plan(int32_t L, int32_t R, bool bimodal, const std::string &plan);
std::vector<std::string> plan_candidates(int32_t L, int32_t R, bool bimodal);
int make_bits_plan(int32_t L, int32_t Rcap, bool bimodal, BitsPlan *plan, std::string *err, bool i8 = false);
// The int8-layout staging instance for a cluster shape (kernels_bits_i8.cu), or null.
void *kernel_for_i8(int L, int S, int GT, int NT, bool bim);
// The split-word instance (NS = 4, kernels_bits_split.cu) for a shape, or null.
void *kernel_for_split(int L, int S, int GT, int NT, bool bim);
// The resident plan on bytes for the int8 layout at L without a bit layout; an empty plan (counter
// null) when the lattice does not fit.
int make_bytes_plan(int32_t L, int32_t Rcap, bool bimodal, BitsPlan *plan, std::string *err);
bool bits_plan_fits(const BitsPlan &plan, int32_t R);
cudaError_t build_field4(const RealView &v, BitsPlan &plan, cudaStream_t st);
void free_bits_plan(BitsPlan &plan);
// Zeroes the words and records that launches of the plan count on across launches (after an expired
// wait they can be uneven).
cudaError_t reset_bits_plan(const BitsPlan &plan, cudaStream_t st);
// The shape in the format of rfim_get_plan.
std::string plan_name(const BitsPlan &plan);
// n_sweeps sweeps; when exchange is true the launch ends with exchange step j (energies, swap
// decisions, permutation, measurement when j >= measure_from).
// With mh set (mh->mh > 0) the sweeps are multi-hit double-checkerboard sweeps.
// n_intervals > 1 (grid-wide and resident plans with the exchange only): that many exchange intervals
// of n_sweeps sweeps each in one launch, exchange steps j, j + 1, ...
cudaError_t launch_sweeps_bits(const RealView &v, const BitsPlan &plan, uint32_t sweep0, int32_t n_sweeps,
                               bool exchange, uint32_t j, int64_t measure_from, double J, double h,
                               cudaStream_t st, const MultiHit *mh = nullptr, int32_t n_intervals = 1,
                               const XiWork *xi = nullptr);

}  // namespace rfim

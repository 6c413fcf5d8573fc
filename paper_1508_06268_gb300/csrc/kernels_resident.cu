// Instances, launch shapes and launcher of the resident sweep kernel (kernels_resident.cuh).
#include <algorithm>
#include <iterator>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "resident.h"

namespace rfim {

int resident_ctas(const void *fn, int S, int threads, size_t smem) {
  static std::mutex mu;
  static std::map<std::tuple<int, const void *, int, int, size_t>, int> known;
  int dev = 0;
  cudaGetDevice(&dev);
  const auto key = std::make_tuple(dev, fn, S, threads, smem);
  {
    std::lock_guard<std::mutex> lk(mu);
    const auto it = known.find(key);
    if (it != known.end()) return it->second;
  }
  int n = 0;
  if (raise_smem_limit(fn, smem) == cudaSuccess &&
      (S <= 8 || cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess)) {
    if (S == 1) {
      int per_sm = 0, sms = 0;
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem) == cudaSuccess &&
          cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess)
        n = per_sm * sms;
    } else {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)S);
      cfg.blockDim = dim3((unsigned)threads);
      cfg.dynamicSmemBytes = smem;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = (unsigned)S;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int clusters = 0;
      if (cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) == cudaSuccess) n = clusters * S;
    }
  }
  cudaGetLastError();
  std::lock_guard<std::mutex> lk(mu);
  known[key] = n;
  return n;
}

namespace {

using Instance = ResidentInstance;

const Instance kInstances[] = {
    resident_instance<8, 1, 1, 512, true>(),   resident_instance<8, 1, 2, 512, true>(),   resident_instance<8, 1, 4, 512, true>(),
    resident_instance<16, 1, 1, 512, true>(),  resident_instance<16, 1, 2, 512, true>(),  resident_instance<16, 1, 4, 512, true>(),
    resident_instance<16, 2, 1, 256, true>(),  resident_instance<16, 2, 2, 256, true>(),  resident_instance<32, 2, 4, 512, true>(),
    resident_instance<32, 4, 4, 256, true>(),  resident_instance<32, 8, 2, 256, true>(),  resident_instance<32, 1, 4, 512, false>(),
    resident_instance<32, 2, 4, 512, false>(), resident_instance<64, 16, 4, 512, true>(), resident_instance<64, 8, 4, 512, false>(),
    resident_instance<64, 4, 4, 512, false>(),
};

// The first instance of tile edge T for which f holds, or null.
template <class F>
const Instance *find_if(int32_t T, F f) {
  const std::vector<Instance> &mh = resident_multihit_instances();
  const Instance *first = T ? mh.data() : std::begin(kInstances), *last = T ? mh.data() + mh.size() : std::end(kInstances);
  const Instance *i = std::find_if(first, last, [&](const Instance &x) { return x.T == T && f(x); });
  return i == last ? nullptr : i;
}

const Instance *find(int32_t L, const ResidentShape &s) {
  return find_if(s.T, [&](const Instance &i) { return i.L == L && i.S == s.S && i.NB == s.NB && i.one == s.one; });
}

int slab_words(int32_t L, int32_t S) { return L / S * (L * L / 64); }

size_t resident_smem(int32_t L, int32_t S, int32_t G, int32_t R) {
  const int wc = slab_words(L, S), chunks = std::max(1, 2 * wc / 32);
  const int planes = L / S + (S > 1 ? 2 : 0);
  return (size_t)G * 2 * planes * (L * L / 64) * 4 + tab_bytes(G) + (size_t)G * chunks * sizeof(ChunkSum) + resident_state_bytes(R);
}

// With the marginals of the structure factor.
size_t resident_xi_smem(int32_t L, const ResidentShape &s) { return s.smem + (size_t)s.G * 3 * L * sizeof(int); }

// log2 of the words whose items of one part are neighbouring threads: a warp's worth, or all of a
// CTA's words when they are fewer (several parts then share a warp).
int lane_words(const Instance &i, int32_t G) {
  int lw = 5;
  while (i.one && lw > 0 && (1 << (lw - 1)) >= G * slab_words(i.L, i.S)) --lw;
  return lw;
}

int warp_items(const Instance &i, int32_t G) {
  const int lw = lane_words(i, G), groups = (G * slab_words(i.L, i.S) + (1 << lw) - 1) >> lw;
  return ((groups * ((i.T ? 4 : 8) / i.NB) << lw) + 31) / 32;
}

// Threads of a CTA: one item each up to the instance's limit, and enough to poll the records.
int cta_threads(const Instance &i, int32_t G, int32_t R) {
  const int want = std::max(32 * warp_items(i, G), std::min((R + 31) / 32 * 32, 256));
  return std::min(want, i.NT);
}

// Estimated cycles of a half-sweep (measured at L = 8 to 64, 2.07 GHz): warp instructions of the
// fullest SM (15 per attempt and 50 per item, 137 where items are decoded every time) at 2.4 per
// cycle, the dependent chain of one item, and for slabs the halo exchange, which CTAs sharing an SM
// run one after the other.  Clusters pack into the GPU's processing clusters, so the CTAs that run
// at one per SM are fewer than the SMs (144 of 152 in clusters of four, 120 in clusters of eight).
double half_sweep_cycles(const Instance &i, int32_t G, int32_t R, int spread) {
  const int ctas = (R + G - 1) / G * i.S, per_sm = (ctas + spread - 1) / spread;
  const double instr = (double)per_sm * warp_items(i, G) * (4.0 * 15.0 * i.NB + (i.one ? 50.0 : 137.0));
  // (multi-hit slabs of whole tiles exchange halos once per visit, not per pass)
  const bool halos = i.S > 1 && !(i.T && i.L / i.S % i.T == 0);
  return instr / 2.4 + 200.0 + 30.0 * i.NB + (halos ? 300.0 + 400.0 * (per_sm - 1) : 0.0);
}

struct Candidate {
  const Instance *inst;
  ResidentShape shape;
  double cycles;
};

// Every instance with every group size, the fastest by estimate first.
std::vector<Candidate> candidates(int32_t L, int32_t R, bool bimodal, int32_t T = 0) {
  std::vector<Candidate> all;
  find_if(T, [&](const Instance &i) {
    if (i.L != L) return false;
    const int spread = resident_ctas((const void *)(bimodal ? i.bim : i.flt), i.S, i.NT, kOneCtaSmem);
    for (int32_t G = 1; spread > 0 && G <= std::min(R, 64); ++G) {
      if (i.one && 32 * warp_items(i, G) > i.NT) break;
      Candidate c{&i, {}, half_sweep_cycles(i, G, R, spread)};
      c.shape.S = i.S;
      c.shape.G = G;
      c.shape.NB = i.NB;
      c.shape.one = i.one;
      c.shape.T = i.T;
      c.shape.threads = cta_threads(i, G, R);
      all.push_back(c);
    }
    return false;
  });
  std::stable_sort(all.begin(), all.end(), [](const Candidate &a, const Candidate &b) { return a.cycles < b.cycles; });
  return all;
}

}  // namespace

bool resident_fits(int32_t L, int32_t R, bool bimodal, ResidentShape *s) {
  const Instance *i = find(L, *s);
  if (!i || s->G < 1 || s->threads < 32 || s->threads > i->NT || s->threads % 32) return false;
  if (i->one && 32 * warp_items(*i, s->G) > s->threads) return false;
  s->smem = resident_smem(L, s->S, s->G, R);
  if (s->smem > 227 * 1024) return false;
  const int64_t ctas = (int64_t)((R + s->G - 1) / s->G) * s->S;
  return ctas <= resident_ctas((const void *)(bimodal ? i->bim : i->flt), s->S, s->threads, s->smem);
}

bool resident_xi_fits(int32_t L, int32_t R, bool bimodal, const ResidentShape &s) {
  const ResidentFn fn = s.T || !s.NB ? nullptr : resident_xi_kernel(L, s.S, s.NB, s.one, bimodal);
  const size_t smem = resident_xi_smem(L, s);
  if (!fn || smem > 227 * 1024) return false;
  const int64_t ctas = (int64_t)((R + s.G - 1) / s.G) * s.S;
  return ctas <= resident_ctas((const void *)fn, s.S, s.threads, smem);
}

bool resident_shape(int32_t L, int32_t R, bool bimodal, ResidentShape *out, double *cycles, int32_t T) {
  for (const Candidate &c : candidates(L, R, bimodal, T)) {
    ResidentShape s = c.shape;
    if (!resident_fits(L, R, bimodal, &s)) continue;
    *out = s;
    *cycles = c.cycles;
    return true;
  }
  return false;
}

std::vector<ResidentShape> resident_shapes(int32_t L, int32_t R, bool bimodal) {
  std::vector<ResidentShape> all;
  std::vector<const Instance *> seen;
  for (const Candidate &c : candidates(L, R, bimodal)) {
    ResidentShape s = c.shape;
    if (std::find(seen.begin(), seen.end(), c.inst) != seen.end() || !resident_fits(L, R, bimodal, &s)) continue;
    seen.push_back(c.inst);
    all.push_back(s);
  }
  return all;
}

ResidentLaunch::ResidentLaunch(int clusters, const ResidentShape &s, bool exchange, cudaStream_t st) {
  cfg.gridDim = dim3((unsigned)(clusters * s.S));
  cfg.blockDim = dim3((unsigned)s.threads);
  cfg.dynamicSmemBytes = s.smem;
  cfg.stream = st;
  if (s.S > 1) {
    at[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    at[cfg.numAttrs].val.clusterDim.x = (unsigned)s.S;
    at[cfg.numAttrs].val.clusterDim.y = 1;
    at[cfg.numAttrs++].val.clusterDim.z = 1;
  }
  if (exchange && clusters > 1) {
    at[cfg.numAttrs].id = cudaLaunchAttributeCooperative;
    at[cfg.numAttrs++].val.cooperative = 1;
  }
  cfg.attrs = at;
}

cudaError_t launch_resident(const RealView &v, const ResidentShape &s, const ResidentArgs &args, uint32_t sweep0,
                            int32_t n_sweeps, const float4 *field4, const ExchArgs &xa, cudaStream_t st) {
  const Instance *i = find(v.L, s);
  if (!i) return cudaErrorInvalidConfiguration;
  ResidentArgs ra = args;
  ra.keys = philox_keys(v.seed, v.realization);
  ra.lw = lane_words(*i, s.G);
  const int clusters = (v.R + s.G - 1) / s.G;
  const bool bim = v.kind == kBimodal;
  ResidentFn fn = bim ? i->bim : i->flt;
  ResidentShape ls = s;
  // without an exchange step no thread polls records: no more warps than have items (L = 8, R = 400, two sweeps per
  // call: 8.5 us with the warps that poll, 6.5 without)
  if (!xa.enabled && s.one) ls.threads = std::max(32, 32 * warp_items(*i, s.G));
  if (ra.xi_marg) {
    fn = resident_xi_kernel(v.L, s.S, s.NB, s.one, bim);
    if (!fn || s.T) return cudaErrorInvalidConfiguration;
    ls.smem = resident_xi_smem(v.L, s);
  }
  ResidentLaunch l(clusters, ls, xa.enabled, st);
  return cudaLaunchKernelEx(&l.cfg, fn, v, ra, sweep0, n_sweeps, field4, xa);
}

}  // namespace rfim

// Launch shapes and launcher of the resident sweep on bytes (kernels_bytes.cuh).
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "kernels_bytes.cuh"
#include "sweep_bits.h"

namespace rfim {

namespace {

using BytesFn = void (*)(RealView, BytesArgs, uint32_t, int32_t, ExchArgs);

constexpr int kBytesThreads = 512;

int row_width(int32_t L) { return L % 8 == 0 ? 4 : L % 4 == 0 ? 2 : 1; }

template <bool ONE>
BytesFn pick(int32_t L, bool bim) {
  switch (row_width(L)) {
    case 4: return bim ? (BytesFn)k_resident_bytes<4, true, ONE> : (BytesFn)k_resident_bytes<4, false, ONE>;
    case 2: return bim ? (BytesFn)k_resident_bytes<2, true, ONE> : (BytesFn)k_resident_bytes<2, false, ONE>;
    default: return bim ? (BytesFn)k_resident_bytes<1, true, ONE> : (BytesFn)k_resident_bytes<1, false, ONE>;
  }
}

BytesFn bytes_fn(int32_t L, bool bim, bool one) { return one ? pick<true>(L, bim) : pick<false>(L, bim); }

int plane_stride(int32_t L) { return (L * L / 2 + 15) / 16 * 16; }
int slab_planes(int32_t L, int32_t S) { return (L + S - 1) / S; }
int slab_blocks(int32_t L, int32_t S) { return (slab_planes(L, S) * (L * L / 2) + 3) / 4 + 1; }

size_t bytes_smem(int32_t L, int32_t S, int32_t G, int32_t R) {
  return (size_t)G * 2 * (slab_planes(L, S) + 2) * plane_stride(L) + tab_bytes(G) + resident_state_bytes(R);
}

int bytes_threads(int32_t L, int32_t S, int32_t G, int32_t R) {
  const int want = std::max((G * slab_blocks(L, S) + 31) / 32 * 32, std::min((R + 31) / 32 * 32, 256));
  return std::min(want, kBytesThreads);
}

// Whether every thread has at most one item.
bool one_item(int32_t L, const ResidentShape &s) { return s.G * slab_blocks(L, s.S) <= s.threads; }

// Estimated cycles of a half-sweep: warp instructions of the fullest SM at 2 per cycle, the chain of
// one item, and the halo exchange of slabs.
double bytes_cycles(int32_t L, const ResidentShape &s, int32_t R, int spread) {
  const int ctas = (R + s.G - 1) / s.G * s.S, per_sm = (ctas + spread - 1) / spread;
  const bool one = one_item(L, s);
  const int instr = row_width(L) == 4 ? (one ? 95 : 140) : row_width(L) == 2 ? (one ? 110 : 165) : (one ? 130 : 220);
  return (double)per_sm * ((s.G * slab_blocks(L, s.S) + 31) / 32) * instr / 2.0 + 3.0 * instr +
         (s.S > 1 ? 300.0 + 200.0 * (per_sm - 1) : 0.0);
}

// Fitted to L = 4 to 116, R = 2 to 400 (Gaussian field; calls of two sweeps, of an exchange step, runs of 5 and of
// 1 sweep per step), mostly within a fifth; bimodal ones are up to a sixth faster.  A few of the points, us per call, resident / apart: two sweeps
// L = 116, R = 2 171 / 66, L = 40, R = 250 80 / 62, L = 24, R = 40 11 / 26, L = 10, R = 24 8.6 / 21; an exchange
// step L = 40, R = 250 43 / 32, L = 50, R = 100 97 / 138, L = 24, R = 64 17 / 15.
BytesCosts bytes_costs(int32_t L, const ResidentShape &s, int32_t R, double cycles) {
  BytesCosts c;
  const int w = row_width(L);
  const double sites = 0.5 * (double)L * L * L * R * 1e-6, ksites = (double)L * L * L * 1e-3;  // per half-sweep, per replica
  const double kib = (double)s.G * 2 * (slab_planes(L, s.S) + 2) * plane_stride(L) / 1024.0;
  c.half = 0.3 + 1.12 * cycles / 2070.0;
  c.launch = 7.0 + kib * (w == 4 ? 0.045 : w == 2 ? 0.09 : 0.35);
  c.tail = 4.5 + (w == 1 ? 1.5 : 1.15) * c.half + 0.01 * R * s.S;
  c.half_apart = std::min(4.2 + 0.35 * (R - 2), w == 4 ? 6.5 : 5.2) + (w == 4 ? 1.0 : 7.1) * sites;
  const int waves = (R + 151) / 152;  // the energy kernels take a CTA per replica, several for rows of 16
  c.step_apart = L % 16 == 0 ? 21.5 + 0.01 * ksites + sites
                 : w == 4    ? 12.0 + 0.128 * ksites * waves + 0.02 * R
                             : 12.0 + ksites * (1.0 + 0.45 * (waves - 1)) + 0.02 * R;
  return c;
}

bool bytes_fits(int32_t L, int32_t R, bool bim, ResidentShape *s) {
  if (s->S < 1 || s->S > 8 || L < 2 * s->S || s->G < 1 || s->threads < 32 || s->threads > kBytesThreads || s->threads % 32)
    return false;
  s->one = one_item(L, *s);
  s->smem = bytes_smem(L, s->S, s->G, R);
  if (s->smem > 227 * 1024) return false;
  const int64_t ctas = (int64_t)((R + s->G - 1) / s->G) * s->S;
  return ctas <= resident_ctas((const void *)bytes_fn(L, bim, s->one), s->S, s->threads, s->smem);
}

}  // namespace

bool bytes_shape(int32_t L, int32_t R, bool bim, ResidentShape *out, double *cycles) {
  if (L < 4 || L % 2 || L > kBytesMaxL || bits_supported(L)) return false;
  ResidentShape s;
  s.NB = 0;
  const char *o = getenv("RFIM_BITS_PLAN");  // "S,G,4,threads,b" names a shape of this kernel
  char suffix = 0;
  int words = 0;
  if (o && sscanf(o, "%d,%d,%d,%d,%c", &s.S, &s.G, &words, &s.threads, &suffix) == 5 && suffix == 'b' && bytes_fits(L, R, bim, &s)) {
    *out = s;
    *cycles = 0.0;
    return true;
  }
  struct Candidate {
    ResidentShape s;
    double cycles;
  };
  std::vector<Candidate> all;
  for (int32_t S : {1, 2, 4, 8}) {
    if (L < 2 * S) continue;
    const int spread = resident_ctas((const void *)bytes_fn(L, bim, false), S, kBytesThreads, kOneCtaSmem);
    for (int32_t G = 1; spread > 0 && G <= std::min(R, 64) && bytes_smem(L, S, G, R) <= 227 * 1024; ++G) {
      Candidate c;
      c.s.S = S;
      c.s.G = G;
      c.s.NB = 0;
      c.s.threads = bytes_threads(L, S, G, R);
      c.cycles = bytes_cycles(L, c.s, R, spread);
      all.push_back(c);
    }
  }
  std::stable_sort(all.begin(), all.end(), [](const Candidate &a, const Candidate &b) { return a.cycles < b.cycles; });
  for (const Candidate &c : all) {
    s = c.s;
    if (!bytes_fits(L, R, bim, &s)) continue;
    *out = s;
    *cycles = c.cycles;
    return true;
  }
  return false;
}

int make_bytes_plan(int32_t L, int32_t Rcap, bool bimodal, BitsPlan *plan, std::string *err) {
  BitsPlan p;
  ResidentShape s;
  double cycles = 0.0;
  // Rows of whole blocks with many replicas (above about 8 million sites per half-sweep) are still
  // faster in one launch per half-sweep: 6.5 us + 1.15 us per million sites (measured: L = 40, R = 159
  // 12.4 against 10.4 us here, L = 56, R = 100 16.2 / 16.7, L = 48, R = 200 17.7 / 20.3); other rows take
  // twice the time here or more there at every size (L = 50, R = 150: 71.7 / 33.1).
  const double sites = 0.5 * (double)L * L * L * Rcap * 1e-6;
  if (!bytes_shape(L, Rcap, bimodal, &s, &cycles) || (row_width(L) == 4 && cycles > 2070.0 * (6.5 + 1.15 * sites))) return 0;
  p.L = L;
  p.Rcap = Rcap;
  p.S = s.S;
  p.G = s.G;
  p.threads = s.threads;
  p.smem = s.smem;
  p.res = s;
  if (cycles > 0.0) p.cost = bytes_costs(L, s, Rcap, cycles);  // a named shape is taken for every launch
  p.rec_slots = (size_t)Rcap * s.S;
  const size_t rec_bytes = 2 * p.rec_slots * sizeof(uint4);
  cudaError_t e = cudaMalloc((void **)&p.rec, rec_bytes);
  if (e == cudaSuccess) e = cudaMalloc((void **)&p.counter, 16);
  if (e == cudaSuccess) e = cudaMemset(p.rec, 0, rec_bytes);
  if (e == cudaSuccess) e = cudaMemset(p.counter, 0, 16);
  if (e != cudaSuccess) {
    cudaGetLastError();
    if (err) *err = std::string("resident plan: ") + cudaGetErrorString(e);
    free_bits_plan(p);
    return e == cudaErrorMemoryAllocation ? -2 : -3;
  }
  *plan = p;
  return 0;
}

cudaError_t launch_resident_bytes(const RealView &v, const ResidentShape &s, const ResidentArgs &ra, uint32_t sweep0,
                                  int32_t n_sweeps, const ExchArgs &xa, cudaStream_t st) {
  BytesArgs ba{};
  ba.keys = philox_keys(v.seed, v.realization);
  ba.S = s.S;
  ba.G = s.G;
  ba.rcap = ra.rcap;
  ba.n_iv = ra.n_iv;
  ba.epoch0 = ra.epoch0;
  ba.rec = ra.rec;
  ba.stop = ra.stop;
  ba.stride = plane_stride(v.L);
  ba.planes = slab_planes(v.L, s.S);
  const int clusters = (v.R + s.G - 1) / s.G;
  ResidentLaunch l(clusters, s, xa.enabled, st);
  return cudaLaunchKernelEx(&l.cfg, bytes_fn(v.L, v.kind == kBimodal, s.one), v, ba, sweep0, n_sweeps, xa);
}

}  // namespace rfim

// Number of (block, or site of a plane) quotients of the kernel's arithmetic that are wrong or outside its bound.
extern "C" int rfim_selftest_bytes(int32_t L) {
  using namespace rfim;
  if (L < 4 || L % 2 || L > kBytesMaxL) return -1;  // RFIM_EINVAL
  const int plane = L * L / 2, Lh = L / 2, blocks = plane * L / 4;
  const uint32_t m_plane = recip((uint32_t)plane / 2), m_row = recip((uint32_t)Lh);
  int bad = (uint64_t)(2 * blocks) * (plane / 2) >= 1ull << 32;
  for (int b = 0; b < blocks; ++b) bad += plane_of_block(b, m_plane) != 4 * b / plane;
  for (int rem = 0; rem < plane; ++rem) bad += quot(rem, m_row) != rem / Lh;
  return bad;
}

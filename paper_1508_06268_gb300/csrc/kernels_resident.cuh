// Resident sweep of small realizations: every lattice stays in shared memory for many exchange
// intervals of one launch.
//
// Bound: latency.  A half-sweep of a small realization (L = 8, R = 16: 1024 Philox blocks; L = 32,
// R = 70: 286720) is a few hundred cycles of work per SM, so what counts is the chain from one
// half-sweep to the next and the exchange step, not the rate of the decisions.  Therefore
//   - a cluster of S CTAs (z slabs) holds G replicas, with S and G chosen so that all CTAs are
//     resident at once and spread over the SMs (resident_shape); a launch runs up to
//     kResidentIntervals intervals;
//   - an item is NB of the 8 Philox blocks of a 32-site word of one replica; the NP = 8 / NB items of a
//     word xor their flips into it.  ONE: every thread has one item for the whole launch, and all
//     that depends on it alone (neighbour addresses, field values, the products of the first two
//     Philox rounds that hold the block index) is formed once and stays in registers;
//   - the random words do not depend on the spins: S = 1 forms those of the next half-sweep in the
//     same straight-line code as the decisions of this one, so that the two dependent chains fill
//     each other's latencies; S > 1 forms them while the halos are on their way;
//   - slabs push their end planes into the neighbours' halo planes with st.async, which counts the
//     bytes into the neighbour's mbarrier: the data is its own signal.  (A cluster barrier with
//     release semantics per half-sweep instead stalls on the memory barrier it implies: a fifth of
//     the issue slots at L = 32, R = 70.)
//   - the exchange step gathers the energies as records (exchange_records.cuh) instead of one
//     launch per interval with an arrival counter and a last CTA that takes the step alone, and
//     the measurement of temperature k is added by CTA k mod P.
//
// T > 0: the multi-hit double checkerboard (Sec. 3.2; see kernels_mh.cuh for the order of the passes)
// with tiles of edge T.  A pass updates half of the blocks of a colour, so it is even shorter, and
// the four blocks of a word in tiles of even x index and the four in odd ones are updated in turn
// by the same items: an item is NB of four.  Where slabs are whole tiles the halos a visit reads are
// frozen, so the slabs exchange both colours once per visit instead of one colour per pass.
// Per pass, against one launch per interval with a cluster barrier per pass (us): L = 16, R = 32 1.43 -> 0.32,
// L = 32, R = 40 2.06 -> 0.81 (tiles of 8) and 0.85 (of 16), R = 140 2.38 -> 1.42, L = 64, R = 14 10.0 -> 1.34.
#pragma once
#include <cstdint>

#include "exchange_records.cuh"
#include "halos.cuh"
#include "kernels_bits.cuh"
#include "philox_parts.cuh"

namespace rfim {

struct ResidentArgs {
  PhiloxKeys keys;
  int32_t G;        // replicas per cluster
  int32_t rcap;     // replica capacity
  int32_t n_iv;     // exchange intervals in this launch
  uint32_t epoch0;  // interval number of this launch's first interval
  uint4 *rec;       // [2][rcap * S] energy records
  int32_t i8;       // the realization is stored as bytes (v.spins8) and staged as bits
  int32_t lw;       // log2 of the words whose items of one part are neighbouring threads (ONE; else 5)
  int32_t mh;       // passes per tile visit (T > 0)
  SelftestStop stop;
  // structure factor (XI): of every interval iv >= xi_first, the marginals S_d[t] of every
  // replica, [iv][R][3][L], zero when the launch starts, and the replica at every temperature, [iv][R]
  int32_t *xi_marg, *xi_t2r;
  int32_t xi_first;
};

// Planes of a slab in shared memory: with S > 1 a halo plane before and after the slab's own.
template <int L, int S>
__host__ __device__ constexpr int resident_planes() { return L / S + (S > 1 ? 2 : 0); }

// 32-word chunks (L = 8: 16-word ones, a replica) the energy reduction of a slab is cut into.
template <int L, int S>
__host__ __device__ constexpr int resident_chunks() {
  return 2 * (L / S) * (L * L / 64) >= 32 ? 2 * (L / S) * (L * L / 64) / 32 : 1;
}

// Items of a word: its eight blocks, or the four that one pass of the double checkerboard updates,
// by NB.
template <int NB, int T>
__host__ __device__ constexpr int resident_parts() { return (T ? 4 : 8) / NB; }

// Block j of an item relative to its first one; with tiles of edge T the blocks of every other run of T / 8.
template <int NB, int T>
__host__ __device__ constexpr int item_block(int j) { return T == 0 ? j : j / (T / 8) * (T / 4) + j % (T / 8); }
template <int NB, int T>
__host__ __device__ constexpr uint32_t item_pattern() {
  uint32_t m = 0u;
  for (int j = 0; j < NB; ++j) m |= 1u << item_block<NB, T>(j);
  return m;
}

// 32 x 32 bits over a warp, transposed: bit k of lane i was bit i of lane k.
__device__ __forceinline__ uint32_t transpose_bits(uint32_t x, int lane) {
  uint32_t m = 0x0000FFFFu;
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, s);
    x = lane & s ? (x & ~m) | ((y & ~m) >> s) : (x & m) | ((y & m) << s);
    m ^= m << (s / 2);
  }
  return x;
}

// Marginals S_d[t] (sums of the spins with coordinate t along axis d, Sec. 7's structure factor) of
// gact replicas over the planes z0 .. of a slab, first in marg[g][3][L] (zero at the call) and then added to
// out[g][3][L] in global memory; replica g's colours are CW words each, the slab's own planes from word
// `first` of a colour on.  A warp takes 32 words: their transpose gives lane b the 32 bits of in-word
// bit b, i.e. of one x up to the row parity.
template <int L, int PZ>
__device__ __forceinline__ void slab_marginals(const uint32_t *sp, int CW, int first, int *marg, int gact, int z0, int32_t *out) {
  constexpr int P = BitsGeom<L>::P, Lh = L / 2, RW = 64 / L, WC = PZ * P, NCK = (WC + 31) / 32;
  constexpr uint32_t kRow = ((1u << (Lh / 4)) - 1u) * 0x01010101u;
  const int lane = threadIdx.x & 31, p = 4 * (lane & 7) + (lane >> 3);  // in-word position of bit `lane`
  for (int u = threadIdx.x >> 5; u < gact * 2 * NCK; u += blockDim.x >> 5) {
    const int g = u / (2 * NCK), c = u / NCK & 1, wl = u % NCK * 32 + lane;
    const bool in = wl < WC;
    const uint32_t w = in ? sp[(g * 2 + c) * CW + first + wl] : 0u;
    int *mg = marg + g * 3 * L;
    const int z = z0 + (in ? wl : 0) / P, y0 = wl % P * RW;
    if (in) {
#pragma unroll
      for (int rr = 0; rr < RW; ++rr) atomicAdd(&mg[L + y0 + rr], 2 * __popc(w & (kRow << (rr * (Lh / 4)))) - Lh);
    }
    if (P >= 32) {  // the warp's words share one plane
      const int zs = __reduce_add_sync(0xffffffffu, 2 * __popc(w) - 32);
      if (lane == 0) atomicAdd(&mg[2 * L + z], zs);
    } else if (in) {
      atomicAdd(&mg[2 * L + z], 2 * __popc(w) - 32);
    }
    const uint32_t have = __ballot_sync(0xffffffffu, in), odd0 = __ballot_sync(0xffffffffu, in && ((c + y0 + z) & 1));
    const uint32_t col = transpose_bits(w, lane), odd = (p / Lh & 1) ? have & ~odd0 : odd0, even = have & ~odd;
    atomicAdd(&mg[2 * (p % Lh)], 2 * __popc(col & even) - __popc(even));
    atomicAdd(&mg[2 * (p % Lh) + 1], 2 * __popc(col & odd) - __popc(odd));
  }
  __syncthreads();
  for (int t = threadIdx.x; t < gact * 3 * L; t += blockDim.x)
    if (marg[t] != 0) atomicAdd(out + t, marg[t]);
}

// One item: word iw of plane zl of replica g of the slab, blocks sh + item_block(0 .. NB - 1) of it (T > 0:
// sh for the tiles of even x index, T / 8 further on for the odd ones).
template <int NB>
struct ResidentItem {
  int g, z, sh;
  int odd;                        // T > 0: parity of y / T + z / T
  int64_t wq;                     // word within its colour
  int same, next, prev, up, down; // word indices in the replica's colour-0 planes
  uint32_t p0;                    // row-parity mask of colour 0 (colour 1: its complement)
};

// XI: measures the structure factor too (an instance of its own: as a run-time choice it slowed runs
// that do not measure it, L = 16, R = 32 5.7 -> 5.9 us per interval).
template <int L, int S, int NB, bool BIM, int NT, bool ONE, int T = 0, bool XI = false>
__global__ void __launch_bounds__(NT) k_resident(const RealView v, const __grid_constant__ ResidentArgs ra, uint32_t sweep0,
                                                 int32_t nsw, const float4 *__restrict__ field4, const ExchArgs xa) {
  using Gm = BitsGeom<L>;
  constexpr int P = Gm::P, W = Gm::W, PZ = L / S, WC = PZ * P, NP = resident_parts<NB, T>();
  constexpr int CW = resident_planes<L, S>() * P;  // words of one colour of one replica, halos included
  constexpr int Z1 = S > 1 ? 1 : 0;                // the slab's first own plane
  constexpr int64_t WPAD = (W + 31) / 32 * 32;
  constexpr int SEG = 2 * WC < 32 ? 2 * WC : 32, NCH = resident_chunks<L, S>();
  static_assert(2 * WC >= 16, "a slab of one replica fills at least half a warp");
  constexpr bool WHOLE_TILES = T > 0 && PZ % (T ? T : 1) == 0;  // no tile is cut by the slabs
  static_assert(S == 1 || P % 4 == 0, "halo planes are pushed 16 bytes at a time");
  static_assert(T == 0 || (T % 8 == 0 && L % (2 * T) == 0 && NB <= 4 && (NB >= T / 8 || T / 8 % NB == 0)),
                "an item's blocks lie in tiles of one x parity");
  extern __shared__ __align__(16) uint32_t sm[];
  __shared__ __align__(8) HaloBars hb;
  __shared__ volatile GaveUp gave_up;
  const int rank = S > 1 ? (int)cluster_rank() : 0;
  const int z0 = rank * PZ, r0 = (int)(blockIdx.x / S) * ra.G, gact = min(ra.G, v.R - r0);
  const int nt = blockDim.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
  const int R = v.R;

  constexpr int NC = WHOLE_TILES ? 2 : 1;                     // colours of a push
  const uint32_t push_bytes = (uint32_t)(gact * NC * P * 4);  // to each neighbour

  uint32_t *sp = sm;                            // [G][2][CW]
  uint32_t *tab = sm + (size_t)ra.G * 2 * CW;   // G decision-table slots
  const uint32_t slot0 = tab_slot0(tab);
  ChunkSum *red = reinterpret_cast<ChunkSum *>(reinterpret_cast<char *>(tab) + tab_bytes(ra.G));  // [G][NCH]
  ResidentState xs;
  xs.E = reinterpret_cast<double *>(red + (size_t)ra.G * NCH);
  xs.beta = xs.E + ra.rcap;
  xs.M = reinterpret_cast<int32_t *>(xs.beta + ra.rcap);
  xs.t2r = xs.M + ra.rcap;
  xs.r2t = xs.t2r + ra.rcap;
  xs.swapped = reinterpret_cast<uint8_t *>(xs.r2t + ra.rcap);
  int *marg = reinterpret_cast<int *>(reinterpret_cast<char *>(xs.E) + resident_state_bytes(ra.rcap) / 16 * 16);  // [G][3][L]

  // debug build: the replica range, the shared-memory plan and the cluster must be the launch's
  const bool ok = RFIM_DCHECK(xa.err, gact >= 1 && gact <= ra.G && r0 + gact <= R && R <= ra.rcap, kDbgGlobal) &&
                  RFIM_DCHECK(xa.err, xs.swapped + ra.rcap <= reinterpret_cast<uint8_t *>(marg) &&
                                          (uint32_t)__cvta_generic_to_shared(marg + (XI ? 3 * L * ra.G : 0)) <=
                                              (uint32_t)__cvta_generic_to_shared(sm) + dyn_smem_bytes(),
                              kDbgTable) &&
                  RFIM_DCHECK(xa.err, S == 1 || cluster_ctas() == (uint32_t)S, kDbgRank);
  // the slab with its halo planes (the halos of colour 0 are pushed before they are needed)
  for (int t = tid; ok && t < gact * 2 * CW; t += nt) {
    const int g = t / (2 * CW), rem = t % (2 * CW), c = rem / CW, pl = rem % CW / P, iw = rem % P;
    const int z = (z0 + pl - Z1 + L) % L;
    const int64_t gw = ((int64_t)(r0 + g) * 2 + c) * W + (int64_t)z * P + iw;
    sp[t] = ra.i8 ? pack_int8_word(v.spins8 + 32 * gw) : v.bits[gw];
  }
  if (ok) tab_fill<BIM>(v, tab, slot0, gact, [&](int g) { return r0 + g; });
  if (xa.enabled && ok)
    for (int r = tid; r < R; r += nt) {
      xs.t2r[r] = v.t2r[r];
      xs.r2t[r] = v.r2t[r];
      xs.beta[r] = v.beta_d[r];
    }
  const bool limbs = !BIM && xa.flimb != nullptr;
  const double fscale = limbs ? ldexp(1.0, xa.fquant->qe) : 1.0;
  const long long Htot = limbs ? xa.fquant->Htot : 0;
  if (tid == 0) gave_up.sweep[0] = gave_up.sweep[1] = gave_up.exchange = 0u;
  if (S > 1) {
    if (tid == 0) halo_init(&hb, push_bytes);
    sync_slabs<S>();  // every CTA's mbarriers are ready before the first push
  } else {
    __syncthreads();
  }

  const int words = ok ? gact * WC : 0;
  auto decode = [&](int item, int lw, bool *valid) {
    ResidentItem<NB> it;
    const int fw = ((item >> lw) / NP << lw) + (item & ((1 << lw) - 1));
    *valid = fw < words;
    const int f = *valid ? fw : 0;  // a thread without an item repeats the first one and drops its flips
    const int part = (item >> lw) % NP * NB;  // the item's first block (T > 0: among the four of a pass)
    it.sh = item_block<1, T>(part);
    it.g = f / WC;
    const int wl = f % WC, zl = wl / P, iw = wl % P;
    it.z = z0 + zl;
    it.wq = (int64_t)it.z * P + iw;
    const int base = it.g * 2 * CW, pl = base + (zl + Z1) * P;
    it.same = pl + iw;
    it.next = pl + (iw + 1) % P;
    it.prev = pl + (iw + P - 1) % P;
    it.up = S > 1 ? it.same + P : base + (zl + 1) % L * P + iw;
    it.down = S > 1 ? it.same - P : base + (zl + L - 1) % L * P + iw;
    it.p0 = parity0_mask<L>(0, it.z, iw);
    it.odd = T ? ((iw * (64 / L)) / (T ? T : 1) + it.z / (T ? T : 1)) & 1 : 0;
    return it;
  };
  // first block of the item in the tiles of coarse colour `coarse` (T = 0: one set of blocks)
  auto first_block = [&](const ResidentItem<NB> &it, int coarse) { return it.sh + (T ? ((coarse ^ it.odd) & 1) * (T / 8) : 0); };
  auto parts_of = [&](const ResidentItem<NB> &it, int coarse) {
    return block_parts<NB>(ra.keys, v.stage, (uint32_t)(8 * it.wq + first_block(it, coarse)), [](int j) { return item_block<NB, T>(j); });
  };
  auto field_of = [&](const ResidentItem<NB> &it, int sh, int c, float4 (&h)[NB]) {
#pragma unroll
    for (int j = 0; j < NB; ++j)
      h[j] = BIM ? make_float4(0.f, 0.f, 0.f, 0.f) : __ldg(field4 + field4_index(c, it.wq, sh + item_block<NB, T>(j), WPAD));
  };
  auto field_bits = [&](const ResidentItem<NB> &it, int c) { return BIM ? v.hbits[(int64_t)c * W + it.wq] : 0u; };
  // decisions of one item of colour c, first block sh, from its random words, xored into its word
  auto update = [&](const ResidentItem<NB> &it, int sh, int c, const Words4 (&w)[NB], const float4 (&h)[NB], uint32_t fb, bool valid) {
    const uint32_t *O = sp + (c ^ 1) * CW;
    uint32_t A, B, C, D, c0, c1, c2;
    nb_xy<L>(O[it.same], O[it.next], O[it.prev], c ? ~it.p0 : it.p0, A, B, C, D);
    count6(A, B, C, D, O[it.up], O[it.down], c0, c1, c2);
    uint32_t *self = sp + c * CW + it.same;
    const PairSlices ps = make_pairs(c0 >> sh, c1 >> sh, c2 >> sh, *self >> sh, fb >> sh);
    const uint32_t slot = slot0 + (uint32_t)it.g * kTabSlot;
    Flips<BIM> fl;
    fl.clear();
#pragma unroll
    for (int j = NB - 1; j >= 0; --j) decide_block<BIM>(w[j], ps, item_block<NB, T>(j), slot, h[j], fl);
    uint32_t flip = fl.template word<NB>();
    if (BIM && T > 0) flip = deposit_bits<item_pattern<NB, T>()>(flip);
    if (valid) atomicXor(self, flip << sh);
  };
  // After half-sweep number h of this launch (all of the CTA's updates of colour c done): the slab's
  // first and last planes into the halo planes of the slabs below and above (halos.cuh).
  // WHOLE_TILES: both colours after tile visit number h.
  auto push_halos = [&](int colour, int flag, uint32_t h) {
    constexpr int VEC = P >= 4 ? P / 4 : 1;
    if (tid >= gact * 2 * NC * VEC || !halo_may_push(&gave_up, flag)) return;
    if (tid == 0) halo_expect(&hb, h, 2 * push_bytes);
    for (int t = tid; t < gact * 2 * NC * VEC; t += nt) {
      const int g = t / (2 * NC * VEC), c = NC == 2 ? t / (2 * VEC) & 1 : colour, side = t / VEC & 1, q = t % VEC * 4;
      const uint32_t peer = (uint32_t)(rank + (side ? 1 : S - 1)) % S;
      const int from = (g * 2 + c) * CW + (side ? PZ : 1) * P + q, to = (g * 2 + c) * CW + (side ? 0 : PZ + 1) * P + q;
      halo_store(&hb, h, sp + to, peer, *reinterpret_cast<const uint4 *>(sp + from));
    }
  };
  auto wait_halos = [&](uint32_t h, int flag) {
    if (!halo_wait(&hb, h, xa.err)) gave_up.sweep[flag] = 1u;  // (the cluster hears of it at the end of the interval)
  };

  bool valid;
  const ResidentItem<NB> own = decode(tid, ONE ? ra.lw : 5, &valid);
  constexpr int SETS = T ? 2 : 1;  // sets of blocks: one per coarse colour
  BlockParts<NB> bp[SETS];
  float4 hown[SETS][2][NB];
  uint32_t fbown[2] = {0u, 0u};
  Words4 w[NB];
  if (ONE) {
#pragma unroll
    for (int k = 0; k < SETS; ++k) bp[k] = parts_of(own, k);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
#pragma unroll
      for (int k = 0; k < SETS; ++k)
        if (NB <= 2) field_of(own, first_block(own, k), c, hown[k][c]);
      fbown[c] = field_bits(own, c);
    }
    if (S == 1 && !T) philox_words<NB>(ra.keys, bp[0], 0, (uint32_t)(r0 + own.g), sweep0, w);
  }

  const int n_iv = xa.enabled ? ra.n_iv : 1;
  uint32_t h = 0, sweep = sweep0;  // half-sweeps done in this launch; current sweep
  bool gone = false;  // (all threads) this launch's results are not to be had
  for (int iv = 0; iv < n_iv; ++iv) {
    if (!ok || (kDebugBuild && stops_here(ra.stop, iv, xa.err))) {
      gone = true;
      break;
    }
#pragma unroll 1
    for (int s = 0; s < nsw && (S == 1 || !gave_up.sweep[1]); ++s, ++sweep) {
      if constexpr (T > 0) {
#pragma unroll
        for (int coarse = 0; coarse < 2; ++coarse) {
#pragma unroll 1
          for (int hit = 0; hit < ra.mh; ++hit) {
            const uint32_t ctr = sweep * (uint32_t)ra.mh + (uint32_t)hit;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
              // WHOLE_TILES: the halos of a visit arrive before its first pass and leave after its last
              const bool wait = S > 1 && h > 0 && (!WHOLE_TILES || (hit == 0 && c == 0));
              const bool push = S > 1 && (!WHOLE_TILES || (hit == ra.mh - 1 && c == 1));
              if (ONE) {
                const int sh = first_block(own, coarse);
                if (NB > 2) field_of(own, sh, c, hown[coarse][c]);
                philox_words<NB>(ra.keys, bp[coarse], c, (uint32_t)(r0 + own.g), ctr, w);
                if (wait) wait_halos(h - 1, WHOLE_TILES ? coarse : c);
                update(own, sh, c, w, hown[coarse][c], fbown[c], valid);
              } else {
#pragma unroll 1
                for (int item = tid; item < (words + 31) / 32 * 32 * NP; item += nt) {
                  bool in;
                  const ResidentItem<NB> it = decode(item, 5, &in);
                  const int sh = first_block(it, coarse);
                  float4 hf[NB];
                  field_of(it, sh, c, hf);
                  const uint32_t fb = field_bits(it, c);
                  bp[0] = parts_of(it, coarse);
                  philox_words<NB>(ra.keys, bp[0], c, (uint32_t)(r0 + it.g), ctr, w);
                  if (wait && item == tid) wait_halos(h - 1, WHOLE_TILES ? coarse : c);
                  update(it, sh, c, w, hf, fb, in);
                }
              }
              __syncthreads();
              if (push) {
                push_halos(c, WHOLE_TILES ? coarse : c, h);
                ++h;
                // the next visit updates words of both colours at once; otherwise a pass of the other colour
                // and its barrier lie between a push and the next update of the words it reads
                if (WHOLE_TILES) __syncthreads();
              }
            }
          }
        }
        continue;
      }
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        if (ONE && S == 1) {
          if (NB > 2) field_of(own, own.sh, c, hown[0][c]);
          Words4 next[NB];
          philox_words<NB>(ra.keys, bp[0], c ^ 1, (uint32_t)(r0 + own.g), sweep + (uint32_t)c, next);
          update(own, own.sh, c, w, hown[0][c], fbown[c], valid);
#pragma unroll
          for (int j = 0; j < NB; ++j) w[j] = next[j];
          __syncthreads();
        } else if (ONE) {
          if (NB > 2) field_of(own, own.sh, c, hown[0][c]);
          philox_words<NB>(ra.keys, bp[0], c, (uint32_t)(r0 + own.g), sweep, w);
          if (h > 0) wait_halos(h - 1, c);
          update(own, own.sh, c, w, hown[0][c], fbown[c], valid);
          __syncthreads();
          push_halos(c, c, h);
        } else {
          for (int item = tid; item < (words + 31) / 32 * 32 * NP; item += nt) {
            bool in;
            const ResidentItem<NB> it = decode(item, 5, &in);
            float4 hf[NB];
            field_of(it, it.sh, c, hf);
            const uint32_t fb = field_bits(it, c);
            bp[0] = parts_of(it, 0);
            philox_words<NB>(ra.keys, bp[0], c, (uint32_t)(r0 + it.g), sweep, w);
            if (S > 1 && item == tid && h > 0) wait_halos(h - 1, c);
            update(it, it.sh, c, w, hf, fb, in);
          }
          __syncthreads();
          if (S > 1) push_halos(c, c, h);
        }
        ++h;
      }
    }
    if (S > 1 && (gave_up.sweep[0] || gave_up.sweep[1] || (h > 0 && !halo_wait(&hb, h - 1, xa.err)))) {
      gave_up.exchange = 1u;
      halo_give_up(&hb);
    }
    if (!xa.enabled) break;
    const bool xi = XI && iv >= ra.xi_first;
    if (xi)
      for (int t = tid; t < gact * 3 * L; t += nt) marg[t] = 0;

    // ---- energies (Eq. 1) of this slab's replicas, one ChunkSum per SEG words --------------------
    for (int e = tid; e < (gact * 2 * WC + 31) / 32 * 32; e += nt) {
      int b = 0, m = 0;
      unsigned hu[4] = {0u, 0u, 0u, 0u};
      int hsum = 0;
      if (ok && e < gact * 2 * WC) {
        const int g = e / (2 * WC), c = e / WC & 1, wl = e % WC, zl = wl / P, iw = wl % P, z = z0 + zl;
        const int64_t wq = (int64_t)z * P + iw;
        const uint32_t *O = sp + (g * 2 + 1) * CW + Z1 * P;  // colour 1, the slab's own planes
        const uint32_t self = sp[(g * 2 + c) * CW + Z1 * P + wl];
        m = 2 * __popc(self) - 32;
        if (c == 0) {
          uint32_t A, B, C, D;
          nb_xy<L>(O[wl], O[zl * P + (iw + 1) % P], O[zl * P + (iw + P - 1) % P], parity0_mask<L>(0, z, iw), A, B, C, D);
          const uint32_t U = S > 1 ? O[wl + P] : O[(zl + 1) % L * P + iw];
          const uint32_t V = S > 1 ? O[wl - P] : O[(zl + L - 1) % L * P + iw];
          b = 192 - 2 * (__popc(self ^ A) + __popc(self ^ B) + __popc(self ^ C) + __popc(self ^ D) + __popc(self ^ U) +
                         __popc(self ^ V));
        }
        if (BIM) {
          hsum = 32 - 2 * __popc(self ^ v.hbits[(int64_t)c * W + wq]);
        } else {
          const uint4 top0 = __ldg(xa.flimb + flimb_index(c, wq, 8, WPAD));
          const uint4 top1 = __ldg(xa.flimb + flimb_index(c, wq, 9, WPAD));
          const uint32_t top[8] = {top0.x, top0.y, top0.z, top0.w, top1.x, top1.y, top1.z, top1.w};
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint4 lo = __ldg(xa.flimb + flimb_index(c, wq, j, WPAD));
            const uint32_t up = (self >> j) & 0x01010101u;
            hu[0] = __dp4a(up, lo.x, hu[0]);
            hu[1] = __dp4a(up, lo.y, hu[1]);
            hu[2] = __dp4a(up, lo.z, hu[2]);
            hu[3] = __dp4a(up, lo.w, hu[3]);
            hsum = __dp4a((int)up, (int)top[j], hsum);
          }
        }
      }
      ChunkSum s;
      if (SEG == 32) {
        s.B = __reduce_add_sync(0xffffffffu, b);
        s.M = __reduce_add_sync(0xffffffffu, m);
        s.F = __reduce_add_sync(0xffffffffu, hsum);
        if (!BIM) {
          s.F <<= 32;
#pragma unroll
          for (int l = 0; l < 4; ++l) s.F += (long long)__reduce_add_sync(0xffffffffu, hu[l]) << (8 * l);
        }
      } else {
        s.B = b;
        s.M = m;
        s.F = hsum;
        if (!BIM)
          s.F = (s.F << 32) + hu[0] + ((long long)hu[1] << 8) + ((long long)hu[2] << 16) + ((long long)hu[3] << 24);
#pragma unroll
        for (int o = SEG / 2; o > 0; o >>= 1) {
          s.B += __shfl_xor_sync(0xffffffffu, s.B, o);
          s.M += __shfl_xor_sync(0xffffffffu, s.M, o);
          s.F += __shfl_xor_sync(0xffffffffu, s.F, o);
        }
      }
      if (lane % SEG == 0 && e < gact * 2 * WC) red[e / SEG] = s;
    }
    __syncthreads();
    const uint32_t epoch = ra.epoch0 + (uint32_t)iv;
    uint4 *rec = ra.rec + (size_t)(epoch & 1u) * ra.rcap * S;
    for (int g = NCH > 4 ? wid : tid; ok && g < gact; g += NCH > 4 ? nw : nt) {
      ChunkSum s{0, 0, 0};
      if (NCH > 4) {  // a warp adds the chunks of a replica
        for (int q = lane; q < NCH; q += 32) {
          const ChunkSum p = red[g * NCH + q];
          s.B += p.B;
          s.M += p.M;
          s.F += p.F;
        }
        s.B = __reduce_add_sync(0xffffffffu, s.B);
        s.M = __reduce_add_sync(0xffffffffu, s.M);
        s.F = warp_reduce_sum(s.F);
      } else {
        for (int q = 0; q < NCH; ++q) {
          const ChunkSum p = red[g * NCH + q];
          s.B += p.B;
          s.M += p.M;
          s.F += p.F;
        }
      }
      if (NCH <= 4 || lane == 0) record_store(rec + (size_t)(r0 + g) * S + rank, epoch, s.B, s.M, s.F);
    }

    // ---- structure factor: the slab's marginals, while the records are on their way -----------------
    if (xi && ok) slab_marginals<L, PZ>(sp, CW, Z1 * P, marg, gact, z0, ra.xi_marg + ((int64_t)iv * R + r0) * 3 * L);

    // ---- exchange step, then the tables of the temperatures it assigned ------------------------------
    auto energy_of = [&](int B, long long F) {
      const double Fd = BIM ? xa.h * (double)F : (double)(2 * F - Htot) * fscale;
      return -xa.J * (double)B - Fd;
    };
    if (!exchange_from_records<false>(v, xa, xs, rec, S, epoch, xa.j + (uint32_t)iv, &gave_up.exchange, energy_of)) {
      gone = true;
      break;
    }
    if (xi && blockIdx.x == 0)
      for (int k = tid; k < R; k += nt) ra.xi_t2r[(int64_t)iv * R + k] = xs.t2r[k];
    if (iv + 1 < n_iv) tab_fill_temps<BIM>(v, tab, slot0, gact, [&](int g) { return xs.r2t[r0 + g]; });
    __syncthreads();
  }
  if (S > 1) {
    if (gone) halo_give_up(&hb);
    halo_leave(&hb);
  }

  for (int t = tid; ok && t < gact * 2 * WC; t += nt) {
    const int g = t / (2 * WC), rem = t % (2 * WC), c = rem / WC, wl = rem % WC;
    const int64_t gw = ((int64_t)(r0 + g) * 2 + c) * W + (int64_t)z0 * P + wl;
    const uint32_t word = sp[(g * 2 + c) * CW + Z1 * P + wl];
    if (ra.i8)
      unpack_int8_word(word, v.spins8 + 32 * gw);
    else
      v.bits[gw] = word;
  }
  if (xa.enabled && !gone && blockIdx.x == 0)
    for (int r = tid; r < R; r += nt) {
      v.t2r[r] = xs.t2r[r];
      v.r2t[r] = xs.r2t[r];
      v.E[r] = xs.E[r];
      v.M[r] = xs.M[r];
    }
}

}  // namespace rfim

// Resident sweep on bytes: realizations of the int8 layout whose edge L has no bit layout (any even
// L from 4 whose lattice fits the shared memory of a cluster), kept in shared memory for many
// exchange intervals of one launch like the bit-layout ones (kernels_resident.cuh).
//
// Bound: latency for small lattices (L = 10: 125 Philox blocks per replica and half-sweep), the
// shared-memory loads of the neighbours beyond.  One launch per half-sweep, with the neighbours in
// L2, took 3 us or more whatever the size.  Here a cluster of S CTAs (S z slabs of nearly equal
// numbers of planes) holds G replicas; an item is one Philox block, i.e. four consecutive sites of a
// colour.  VW sites of it always share a row and are handled as one word: 4 when rows hold whole
// blocks (L divisible by 8), 2 when rows are even (L divisible by 4), else 1.  Coordinates come from
// multiplications by reciprocals (ONE: every thread has one item for the whole launch, whose
// coordinates, field and Philox parts are formed once), planes are padded to 16 bytes so that slabs can push their end
// planes into the neighbours' halo planes with st.async, and the exchange step gathers records.
#pragma once
#include <cstdint>

#include "decide_bytes.cuh"
#include "exchange_records.cuh"
#include "halos.cuh"
#include "philox_parts.cuh"

namespace rfim {

struct BytesArgs {
  PhiloxKeys keys;
  int32_t S, G, rcap, n_iv;  // slabs, replicas per cluster, replica capacity, intervals of this launch
  uint32_t epoch0;           // interval number of the first
  uint4 *rec;                // [2][rcap * S] energy records
  int32_t stride, planes;    // padded plane (bytes), planes of the largest slab
  SelftestStop stop;
};

// floor(n / d) for n d < 2^32 and d >= 2 with m = recip(d).  The largest argument is a half-plane number in a
// colour (locate), L^5 / 16 < 2^32; rfim_selftest_bytes checks the bound and the quotients.
constexpr int32_t kBytesMaxL = 144;
__host__ __device__ __forceinline__ uint32_t recip(uint32_t d) { return 0xFFFFFFFFu / d + 1u; }
__host__ __device__ __forceinline__ int quot(int n, uint32_t m) {
#ifdef __CUDA_ARCH__
  return (int)__umulhi((uint32_t)n, m);  // (the 64-bit product instead: L = 40, R = 64 430 us per 40 sweeps, not 424)
#else
  return (int)(((uint64_t)(uint32_t)n * m) >> 32);
#endif
}

// Plane of the first site of block b (site 4 b of the colour) with m = recip(plane / 2): planes hold an even
// number of sites, and halving both sides keeps the product below 2^32 (4 b and plane pass it at L = 112).
__host__ __device__ __forceinline__ int plane_of_block(int b, uint32_t m) { return quot(2 * b, m); }

template <int VW>
struct BytesWord;
template <>
struct BytesWord<4> { using type = uint32_t; using copy = uint4; };
template <>
struct BytesWord<2> { using type = uint16_t; using copy = uint2; };
template <>
struct BytesWord<1> { using type = uint8_t; using copy = uint16_t; };

// VW sites of a Philox block that share a row: byte offsets of the word itself and of its neighbours
// within a colour of a replica.
struct RowWord {
  int at, x_odd, x_even;  // x_odd / x_even: the word after / before it in the row (row parity 1 / 0)
  int yp, ym, zp, zm;
  uint32_t flags;  // bit 0: y + z odd, bit 1: a site of this slab
};

template <int VW, bool BIM, bool ONE>
__global__ void __launch_bounds__(512, ONE && VW < 4 ? 1 : 2) k_resident_bytes(const RealView v, const __grid_constant__ BytesArgs ba, uint32_t sweep0,
                                                        int32_t nsw, const ExchArgs xa) {
  using Word = typename BytesWord<VW>::type;
  using Copy = typename BytesWord<VW>::copy;
  extern __shared__ __align__(16) uint32_t sm[];
  __shared__ __align__(8) HaloBars hb;
  __shared__ volatile GaveUp gave_up;
  __shared__ ChunkSum part[16];
  const int L = v.L, Lh = v.Lh, plane = L * Lh, S = ba.S, PS = ba.stride, R = v.R;
  const int64_t half = (int64_t)plane * L;
  const int rank = S > 1 ? (int)cluster_rank() : 0;
  const int z0 = rank * L / S, PZ = (rank + 1) * L / S - z0;
  const int r0 = (int)(blockIdx.x / S) * ba.G, gact = min(ba.G, R - r0);
  const int nt = blockDim.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
  const uint32_t push_bytes = (uint32_t)(gact * PS);  // of end planes to each neighbour
  const int CS = (ba.planes + 2) * PS;  // bytes of one colour of one replica, halo planes included

  uint8_t *lat = reinterpret_cast<uint8_t *>(sm);            // [G][2][planes + 2][PS]
  uint32_t *tab = sm + (size_t)ba.G * 2 * CS / 4;            // G decision-table slots
  const uint32_t slot0 = tab_slot0(tab);
  ResidentState xs;
  xs.E = reinterpret_cast<double *>(reinterpret_cast<char *>(tab) + tab_bytes(ba.G));
  xs.beta = xs.E + ba.rcap;
  xs.M = reinterpret_cast<int32_t *>(xs.beta + ba.rcap);
  xs.t2r = xs.M + ba.rcap;
  xs.r2t = xs.t2r + ba.rcap;
  xs.swapped = reinterpret_cast<uint8_t *>(xs.r2t + ba.rcap);
  const bool ok = RFIM_DCHECK(xa.err, gact >= 1 && gact <= ba.G && r0 + gact <= R && R <= ba.rcap && PZ <= ba.planes, kDbgGlobal) &&
                  RFIM_DCHECK(xa.err, (uint32_t)__cvta_generic_to_shared(xs.swapped + ba.rcap) <=
                                          (uint32_t)__cvta_generic_to_shared(sm) + dyn_smem_bytes(),
                              kDbgTable);

  // plane pl of the slab (0 and PZ + 1: halos) holds lattice plane z0 + pl - 1
  const int cw = plane / (int)sizeof(Copy);
  auto copy_planes = [&](int first, int count, bool in) {
    for (int t = tid; ok && t < gact * 2 * count * cw; t += nt) {
      const int q = t % cw, p = t / cw, pl = first + p % count, gc = p / count;  // gc = 2 g + colour
      Copy *s = reinterpret_cast<Copy *>(lat + (size_t)gc * CS + (size_t)pl * PS) + q;
      Copy *d = reinterpret_cast<Copy *>(v.spins8 + ((int64_t)r0 * 2 + gc) * half + (int64_t)((z0 + pl - 1 + L) % L) * plane) + q;
      if (in)
        *s = *d;
      else
        *d = *s;
    }
  };
  copy_planes(0, PZ + 2, true);
  if (ok) tab_fill<BIM, false>(v, tab, slot0, gact, [&](int g) { return r0 + g; });
  if (xa.enabled && ok)
    for (int r = tid; r < R; r += nt) {
      xs.t2r[r] = v.t2r[r];
      xs.r2t[r] = v.r2t[r];
      xs.beta[r] = v.beta_d[r];
    }
  if (tid == 0) gave_up.sweep[0] = gave_up.sweep[1] = gave_up.exchange = 0u;
  if (S > 1) {
    if (tid == 0) halo_init(&hb, push_bytes);
    sync_slabs<2>();
  } else {
    __syncthreads();
  }

  // Philox blocks that hold sites of this slab; with VW = 1 the first and last may hold others' too
  const int qa = z0 * plane, qb = qa + PZ * plane, b0 = qa >> 2, nblk = ((qb + 3) >> 2) - b0, items = ok ? gact * nblk : 0;
  const uint32_t m_blk = recip((uint32_t)nblk), m_plane = recip((uint32_t)plane / 2), m_row = recip((uint32_t)Lh);
  const int zup = S == 1 ? -(PZ - 1) * PS : PS, zdn = -zup;  // z neighbours of the slab's end planes

  constexpr int NR = 4 / VW;  // row words of a block
  // where block b's sites are (c < 0: for both colours, else with the x neighbour of colour c in both
  // places); sites outside the slab are placed on its first one and left out
  auto locate = [&](int b, int c, RowWord (&rw)[NR]) {
    int z = plane_of_block(b, m_plane);
    const int rem = 4 * b - z * plane;
    int y = quot(rem, m_row), xh = rem - y * Lh;
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      const bool in = VW > 1 || (z >= z0 && z < z0 + PZ);
      const int zl = in ? z - z0 : 0, yy = in ? y : 0, xx = in ? xh : 0;
      const int row = (zl + 1) * PS + yy * Lh, at = row + xx;
      rw[k].at = at;
      const int after = xx + VW == Lh ? 0 : xx + VW, before = xx == 0 ? Lh - VW : xx - VW;
      const int xn = row + (((c + y + z) & 1) ? after : before);
      rw[k].x_odd = c < 0 ? row + after : xn;
      rw[k].x_even = c < 0 ? row + before : xn;
      rw[k].yp = at + (yy == L - 1 ? Lh - plane : Lh);
      rw[k].ym = at + (yy == 0 ? plane - Lh : -Lh);
      rw[k].zp = at + (zl == PZ - 1 ? zup : PS);
      rw[k].zm = at + (zl == 0 ? zdn : -PS);
      rw[k].flags = (uint32_t)((y + z) & 1) | (in ? 2u : 0u);
      // the next word of the block: next in its row, or the next row or plane
      xh += VW;
      const bool row_end = xh == Lh;
      xh = row_end ? 0 : xh;
      y += row_end;
      const bool plane_end = y == L;
      y = plane_end ? 0 : y;
      z += plane_end;
    }
  };
  // The block's own spins and up-counts, one byte per site; `mine` has 0x01 in the bytes of the
  // slab's sites, the others give 0.
  auto gather = [&](const uint8_t *lat_g, int c, const RowWord (&rw)[NR], uint32_t &cur, uint32_t &up, uint32_t &mine) {
    const uint8_t *own = lat_g + c * CS, *O = lat_g + (c ^ 1) * CS;
    cur = up = mine = 0u;
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      auto ld = [&](int o) { return (uint32_t)*reinterpret_cast<const Word *>(O + o); };
      const bool odd = ((rw[k].flags ^ (uint32_t)c) & 1u) != 0;
      const uint32_t a = ld(rw[k].at), w = ld(odd ? rw[k].x_odd : rw[k].x_even);
      uint32_t x = w;
      if (VW == 4) x = odd ? __byte_perm(a, w, 0x4321u) : __byte_perm(w, a, 0x6543u);
      if (VW == 2) x = (odd ? (a >> 8) | (w << 8) : (a << 8) | (w >> 8)) & 0xFFFFu;
      uint32_t n = a + x + ld(rw[k].yp) + ld(rw[k].ym) + ld(rw[k].zp) + ld(rw[k].zm);
      uint32_t s = *reinterpret_cast<const Word *>(own + rw[k].at);
      uint32_t one = VW == 4 ? 0x01010101u : VW == 2 ? 0x0101u : 0x01u;
      if (VW == 1 && !(rw[k].flags & 2u)) n = s = one = 0u;
      up |= n << (8 * VW * k);
      cur |= s << (8 * VW * k);
      mine |= one << (8 * VW * k);
    }
  };
  auto field_bytes = [&](int c, int b) { return BIM ? *reinterpret_cast<const uint32_t *>(v.hbit_c + c * half + 4 * b) : 0u; };
  auto field_of = [&](int c, int b) {
    return BIM ? make_float4(0.f, 0.f, 0.f, 0.f) : __ldg(reinterpret_cast<const float4 *>(v.hh_c + c * half) + b);
  };
  // after half-sweep number h: the slab's end planes into the neighbours' halo planes (halos.cuh)
  auto push_halos = [&](int c, uint32_t h) {
    const int vec = PS / 16;
    if (tid >= gact * 2 * vec || !halo_may_push(&gave_up, c)) return;
    if (tid == 0) halo_expect(&hb, h, 2 * push_bytes);
    for (int t = tid; t < gact * 2 * vec; t += nt) {
      const int q = t % vec, side = t / vec & 1, g = t / (2 * vec);
      const uint32_t peer = (uint32_t)(rank + (side ? 1 : S - 1)) % S;
      const int peer_planes = ((int)peer + 1) * L / S - (int)peer * L / S;
      const size_t base = (size_t)(2 * g + c) * CS + 16 * q;
      halo_store(&hb, h, lat + base + (size_t)(side ? 0 : peer_planes + 1) * PS, peer,
                 *reinterpret_cast<const uint4 *>(lat + base + (size_t)(side ? PZ : 1) * PS));
    }
  };
  auto wait_halos = [&](uint32_t h, int c) {
    if (!halo_wait(&hb, h, xa.err)) gave_up.sweep[c] = 1u;  // (the cluster hears of it at the end of the interval)
  };

  auto update = [&](int g, int c, const RowWord (&rw)[NR], const Words4 &w, const float4 &h4, uint32_t hb, bool valid) {
    uint8_t *lat_g = lat + (size_t)(2 * g) * CS;
    uint32_t cur, up, mine;
    gather(lat_g, c, rw, cur, up, mine);
    const uint32_t nxt = cur ^ decide4<BIM>(w, cur, up, hb, h4, slot0 + (uint32_t)g * kTabSlot);
#pragma unroll
    for (int k = 0; k < NR; ++k)
      if (valid && (VW > 1 || (rw[k].flags & 2u)))
        *reinterpret_cast<Word *>(lat_g + c * CS + rw[k].at) = (Word)(nxt >> (8 * VW * k));
  };

  // ONE: this thread's item (a thread without one repeats the first and writes nothing)
  const bool valid = tid < items;
  const int own_g = valid ? quot(tid, m_blk) : 0, own_b = b0 + (valid ? tid - own_g * nblk : 0);
  RowWord own[NR];
  BlockParts<1> bp;
  float4 hown[2];
  uint32_t hbown[2];
  Words4 w[1];
  if (ONE) {
    locate(own_b, -1, own);
    bp = block_parts<1>(ba.keys, v.stage, (uint32_t)own_b);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      hown[c] = field_of(c, own_b);
      hbown[c] = field_bytes(c, own_b);
    }
    if (S == 1) philox_words<1>(ba.keys, bp, 0, (uint32_t)(r0 + own_g), sweep0, w);
  }

  const int n_iv = xa.enabled ? ba.n_iv : 1;
  uint32_t h = 0, sweep = sweep0;
  bool gone = false;  // (all threads) this launch's results are not to be had
  for (int iv = 0; iv < n_iv; ++iv) {
    if (!ok || (kDebugBuild && stops_here(ba.stop, iv, xa.err))) {
      gone = true;
      break;
    }
#pragma unroll 1
    for (int s = 0; s < nsw && (S == 1 || !gave_up.sweep[1]); ++s, ++sweep) {
      if (ONE) {
#pragma unroll
        for (int c = 0; c < 2; ++c, ++h) {
          if (S == 1) {  // the next half-sweep's words in the same straight-line code as these decisions
            Words4 next[1];
            philox_words<1>(ba.keys, bp, c ^ 1, (uint32_t)(r0 + own_g), sweep + (uint32_t)c, next);
            update(own_g, c, own, w[0], hown[c], hbown[c], valid);
            w[0] = next[0];
            __syncthreads();
          } else {  // this half-sweep's words while the halos are on their way
            philox_words<1>(ba.keys, bp, c, (uint32_t)(r0 + own_g), sweep, w);
            if (h > 0) wait_halos(h - 1, c);
            update(own_g, c, own, w[0], hown[c], hbown[c], valid);
            __syncthreads();
            push_halos(c, h);
          }
        }
      } else {
#pragma unroll 1
        for (int c = 0; c < 2; ++c, ++h) {
          const uint32_t tag = tag_word(kTagMetro, v.stage, (uint32_t)c);
#pragma unroll 1
          for (int item = tid; item < items; item += nt) {
            const int g = quot(item, m_blk), b = b0 + item - g * nblk;
            const float4 h4 = field_of(c, b);
            const uint32_t hbits = field_bytes(c, b);
            RowWord rw[NR];
            locate(b, c, rw);
            const Words4 wi = philox_keyed(ba.keys, (uint32_t)b, (uint32_t)(r0 + g), sweep, tag);
            if (S > 1 && item == tid && h > 0) wait_halos(h - 1, c);
            update(g, c, rw, wi, h4, hbits, true);
          }
          __syncthreads();
          if (S > 1) push_halos(c, h);
        }
      }
    }
    if (S > 1 && (gave_up.sweep[0] || gave_up.sweep[1] || (h > 0 && !halo_wait(&hb, h - 1, xa.err)))) {
      gave_up.exchange = 1u;
      halo_give_up(&hb);
    }
    if (!xa.enabled) break;

    // ---- energies (Eq. 1): small replicas by one warp each, others by the whole CTA ---------------
    // ONE with one replica: every thread has its block's places and field in registers, for both colours
    const uint32_t epoch = ba.epoch0 + (uint32_t)iv;
    uint4 *rec = ba.rec + (size_t)(epoch & 1u) * ba.rcap * S;
    const bool own_blocks = ONE && gact == 1, by_warp = nblk <= 256 && gact > 1;
    const int t0 = by_warp ? lane : tid, dt = by_warp ? 32 : nt;
    for (int g = by_warp ? wid : 0; ok && g < gact; g += by_warp ? nw : 1) {
      int B = 0, M = 0, Fi = 0;
      float fs = 0.f, fe = 0.f;
      auto add_block = [&](int c, const RowWord (&rw)[NR], uint32_t hb, const float4 &h4) {
        uint32_t cur, up, mine;
        gather(lat + (size_t)(2 * g) * CS, c, rw, cur, up, mine);
        const int n = __popc(mine), ups = __popc(cur);
        M += 2 * ups - n;
        // sum of s (2 up - 6) over the sites, s = 2 cur - 1 (colour 0: every bond once)
        if (c == 0) B += 4 * (int)__dp4a(cur, up, 0u) - 12 * ups - 2 * (int)__dp4a(up, 0x01010101u, 0u) + 6 * n;
        if (BIM) {
          Fi += n - 2 * __popc((cur ^ hb) & mine);
        } else {
          const float hk[4] = {h4.x, h4.y, h4.z, h4.w};
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if (!((mine >> (8 * k)) & 1u)) continue;
            const float term = ((cur >> (8 * k)) & 1u) ? hk[k] : -hk[k];
            const float sum = __fadd_rn(fs, term);
            const float bp = __fsub_rn(sum, fs);
            fe = __fadd_rn(fe, __fadd_rn(__fsub_rn(fs, __fsub_rn(sum, bp)), __fsub_rn(term, bp)));
            fs = sum;
          }
        }
      };
      if (own_blocks) {
        if (valid) {
#pragma unroll
          for (int c = 0; c < 2; ++c) add_block(c, own, hbown[c], hown[c]);
        }
      } else {
        for (int t = t0; t < 2 * nblk; t += dt) {
          const int c = t >= nblk, b = b0 + t - (c ? nblk : 0);
          RowWord rw[NR];
          locate(b, c, rw);
          add_block(c, rw, field_bytes(c, b), field_of(c, b));
        }
      }
      ChunkSum sum;
      sum.B = __reduce_add_sync(0xffffffffu, B);
      sum.M = __reduce_add_sync(0xffffffffu, M);
      sum.F = BIM ? (long long)__reduce_add_sync(0xffffffffu, Fi)
                  : __double_as_longlong(warp_reduce_sum((double)fs + (double)fe));
      if (!by_warp) {
        if (lane == 0) part[wid] = sum;
        __syncthreads();
        if (wid == 0) {
          const ChunkSum p = lane < nw ? part[lane] : ChunkSum{0, 0, 0};
          sum.B = __reduce_add_sync(0xffffffffu, p.B);
          sum.M = __reduce_add_sync(0xffffffffu, p.M);
          sum.F = BIM ? warp_reduce_sum(p.F) : __double_as_longlong(warp_reduce_sum(__longlong_as_double(p.F)));
        }
        __syncthreads();
      }
      if (lane == 0 && (by_warp || wid == 0)) record_store(rec + (size_t)(r0 + g) * S + rank, epoch, sum.B, sum.M, sum.F);
    }

    auto energy_of = [&](int B, long long F) {
      return -xa.J * (double)B - (BIM ? xa.h * (double)F : __longlong_as_double(F));
    };
    if (!exchange_from_records<!BIM, false>(v, xa, xs, rec, S, epoch, xa.j + (uint32_t)iv, &gave_up.exchange, energy_of)) {
      gone = true;
      break;
    }
    if (iv + 1 < n_iv) tab_fill_temps<BIM, false>(v, tab, slot0, gact, [&](int g) { return xs.r2t[r0 + g]; });
    __syncthreads();
  }
  if (S > 1) {
    if (gone) halo_give_up(&hb);
    halo_leave(&hb);
  }
  copy_planes(1, PZ, false);
  if (xa.enabled && !gone && blockIdx.x == 0)
    for (int r = tid; r < R; r += nt) {
      v.t2r[r] = xs.t2r[r];
      v.r2t[r] = xs.r2t[r];
      v.E[r] = xs.E[r];
      v.M[r] = xs.M[r];
    }
}

}  // namespace rfim

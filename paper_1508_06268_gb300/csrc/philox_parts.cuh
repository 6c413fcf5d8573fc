// Philox4x32-10 of the metropolis stream with the round keys in the constant bank and the parts that
// do not depend on the replica and the sweep formed ahead (philox.cuh has the generator itself).
#pragma once
#include <cstdint>

#include "philox.cuh"

namespace rfim {

// Round keys of the realization's Philox streams (operands from the constant bank: no key adds).
struct PhiloxKeys {
  uint32_t k0[10], k1[10];
};
__host__ __device__ __forceinline__ PhiloxKeys philox_keys(uint32_t seed, uint32_t realization) {
  PhiloxKeys k;
#pragma unroll
  for (uint32_t i = 0; i < 10; ++i) {
    k.k0[i] = seed + i * kPhiloxW0;
    k.k1[i] = realization + i * kPhiloxW1;
  }
  return k;
}

// philox10 of a metropolis counter with the keys of the realization.
__device__ __forceinline__ Words4 philox_keyed(const PhiloxKeys &k, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3) {
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    const uint64_t p0 = (uint64_t)kPhiloxM0 * c0, p1 = (uint64_t)kPhiloxM1 * c2;
    c0 = (uint32_t)(p1 >> 32) ^ c1 ^ k.k0[i];
    c2 = (uint32_t)(p0 >> 32) ^ c3 ^ k.k1[i];
    c1 = (uint32_t)p1;
    c3 = (uint32_t)p0;
  }
  Words4 r;
  r.w[0] = c0;
  r.w[1] = c1;
  r.w[2] = c2;
  r.w[3] = c3;
  return r;
}

// What the words of Philox blocks of one thread need besides the replica and the sweep: the products
// of the first two rounds that hold only the block index and the colour.
template <int NB>
struct BlockParts {
  uint32_t lo[NB];      // low half of M0 * block
  uint64_t q[2][NB];    // per colour: M1 * (high half of M0 * block ^ tag ^ k1[0])
};

// Words of the NB blocks for sweep and colour c: rounds 0 and 1 from the parts, then eight rounds.
template <int NB>
__device__ __forceinline__ void philox_words(const PhiloxKeys &k, const BlockParts<NB> &bp, int c, uint32_t r, uint32_t sweep,
                                             Words4 (&w)[NB]) {
  const uint64_t s = (uint64_t)kPhiloxM1 * sweep;
  const uint64_t p = (uint64_t)kPhiloxM0 * ((uint32_t)(s >> 32) ^ r ^ k.k0[0]);
#pragma unroll
  for (int j = 0; j < NB; ++j) {
    uint32_t c0 = (uint32_t)(bp.q[c][j] >> 32) ^ (uint32_t)s ^ k.k0[1], c1 = (uint32_t)bp.q[c][j];
    uint32_t c2 = (uint32_t)(p >> 32) ^ bp.lo[j] ^ k.k1[1], c3 = (uint32_t)p;
#pragma unroll
    for (int i = 2; i < 10; ++i) {
      const uint64_t p0 = (uint64_t)kPhiloxM0 * c0, p1 = (uint64_t)kPhiloxM1 * c2;
      c0 = (uint32_t)(p1 >> 32) ^ c1 ^ k.k0[i];
      c2 = (uint32_t)(p0 >> 32) ^ c3 ^ k.k1[i];
      c1 = (uint32_t)p1;
      c3 = (uint32_t)p0;
    }
    w[j].w[0] = c0;
    w[j].w[1] = c1;
    w[j].w[2] = c2;
    w[j].w[3] = c3;
  }
}

// Blocks block0 + step(j).
template <int NB, class F>
__device__ __forceinline__ BlockParts<NB> block_parts(const PhiloxKeys &k, uint32_t stage, uint32_t block0, F step) {
  BlockParts<NB> bp;
#pragma unroll
  for (int j = 0; j < NB; ++j) {
    const uint64_t p = (uint64_t)kPhiloxM0 * (block0 + (uint32_t)step(j));
    bp.lo[j] = (uint32_t)p;
#pragma unroll
    for (int c = 0; c < 2; ++c)
      bp.q[c][j] = (uint64_t)kPhiloxM1 * ((uint32_t)(p >> 32) ^ tag_word(kTagMetro, stage, (uint32_t)c) ^ k.k1[0]);
  }
  return bp;
}

template <int NB>
__device__ __forceinline__ BlockParts<NB> block_parts(const PhiloxKeys &k, uint32_t stage, uint32_t block0) {
  return block_parts<NB>(k, stage, block0, [](int j) { return j; });
}

}  // namespace rfim

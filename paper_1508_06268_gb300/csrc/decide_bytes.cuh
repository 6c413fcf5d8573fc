// Decisions of the four sites of one Philox block from 0/1 bytes, shared by the int8-layout kernels.
#pragma once
#include <cstdint>

#include "decide.cuh"
#include "philox.cuh"

namespace rfim {

// Decisions of the four sites of one Philox block: 0/1 spin bytes `cur`, up-count bytes `up`,
// field bits `hb` (bimodal) or values `h4` (float), table slot `slot`.  Returns 0x01 in the byte
// of every accepted site.
template <bool kBimodalField>
__device__ __forceinline__ uint32_t decide4(const Words4 &w, uint32_t cur, uint32_t up, uint32_t hb, const float4 &h4,
                                            uint32_t slot) {
  if (kBimodalField) {
    const uint32_t offs = ((hb << 4) | (cur << 3) | up) << 2;  // per byte: table index x 4
    uint32_t flips = 0u;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint32_t t;
      asm volatile("ld.shared.u32 %0, [%1];" : "=r"(t) : "r"(__byte_perm(offs, slot, 0x7650u | (uint32_t)j)));
      if (accept_table(w.w[j], t)) flips |= 1u << (8 * j);
    }
    return flips;
  }
  const float hk[4] = {h4.x, h4.y, h4.z, h4.w};
  const uint32_t offs = ((cur << 3) | up) << 3;  // per byte: table index x 8
  float2 e[4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];"
                 : "=f"(e[j].x), "=f"(e[j].y)
                 : "r"(__byte_perm(offs, slot, 0x7650u | (uint32_t)j)));
  const uint2 a = accept_float_signs(w.w[0], w.w[1], e[0], e[1], hk[0], hk[1]);
  const uint2 b = accept_float_signs(w.w[2], w.w[3], e[2], e[3], hk[2], hk[3]);
  // byte j = 0xFF where site j is accepted (its sign bit), then one bit per byte
  const uint32_t m01 = prmt(a.x, a.y, 0x00FBu), m23 = prmt(b.x, b.y, 0xFB00u);
  return ((m01 & 0x0000FFFFu) | (m23 & 0xFFFF0000u)) & 0x01010101u;
}

}  // namespace rfim

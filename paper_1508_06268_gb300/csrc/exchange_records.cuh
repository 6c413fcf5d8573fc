// All-gather of the replicas' energy partials between the CTAs of one launch, and the exchange step
// every CTA then takes on its own copy of the temperature assignment.
//
// A (replica, slab) partial is one 16-byte record: the field sum (64 bits) and, in the other 64
// bits, the bond sum, the magnetisation and the number of the exchange interval it belongs to.  It
// is stored and polled with single 128-bit accesses, which are one memory operation each, so a
// record that carries the awaited interval number is complete: the step needs no fence, no
// arrival counter and no second round trip to read the sums.  Records alternate between two
// buffers by interval; a CTA can only reach interval i + 2 after every CTA has published i + 1 and
// hence finished reading i, so nothing awaited is overwritten.
#pragma once
#include <cstdint>

#include "exchange.cuh"
#include "kernels_bits.cuh"

namespace rfim {

constexpr unsigned kRecordSpinLimit = 1u << 22;
constexpr uint32_t kRecordEpochs = 1u << 22;  // interval numbers 1 .. kRecordEpochs - 1; 0: never written

__device__ __forceinline__ void record_store(uint4 *rec, uint32_t epoch, int B, int M, long long F) {
  const unsigned long long hi = ((unsigned long long)epoch << 42) |
                                ((unsigned long long)(uint32_t)(B + (1 << 21)) << 20) | (uint32_t)(M + (1 << 19));
  asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(rec),
               "l"(F), "l"(hi)
               : "memory");
}

__device__ __forceinline__ void record_load(const uint4 *rec, long long *F, unsigned long long *hi) {
  asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
               : "=l"(*F), "=l"(*hi)
               : "l"(rec)
               : "memory");
}

__device__ __forceinline__ int record_bonds(unsigned long long hi) { return (int)((hi >> 20) & 0x3FFFFFu) - (1 << 21); }
__device__ __forceinline__ int record_spin(unsigned long long hi) { return (int)(hi & 0xFFFFFu) - (1 << 19); }

// Sums of n consecutive records of interval `epoch`, polled at most kRecordSpinLimit times; false
// when they did not all arrive (recorded in *err) or an earlier wait of this launch expired.
__device__ __forceinline__ bool records_sum(const uint4 *rec, int n, uint32_t epoch, unsigned *err, int *B, int *M,
                                            long long *F) {
  for (unsigned it = 0; it < kRecordSpinLimit; ++it) {
    int b = 0, m = 0;
    long long f = 0;
    bool all = true;
#pragma unroll 4
    for (int q = 0; q < n; ++q) {
      long long fq;
      unsigned long long hi;
      record_load(rec + q, &fq, &hi);
      all = all && (uint32_t)(hi >> 42) == epoch;
      b += record_bonds(hi);
      m += record_spin(hi);
      f += fq;
    }
    if (all) {
      *B = b;
      *M = m;
      *F = f;
      return true;
    }
    if ((it & 63u) == 63u && *(volatile unsigned *)err) break;
  }
  atomicOr(err, 2u);
  *B = *M = 0;
  *F = 0;
  return false;
}

// exchange_accept's decision (u < exp(delta) or delta >= 0) for a given u.  The double exponential
// is only evaluated when a single-precision one leaves the decision open: ex2.approx of the float
// delta * log2 e is within 1e-4 relative of exp(delta) for delta > -80 (its argument is rounded
// twice, |delta log2 e| 2^-23 < 2e-5, and ex2.approx adds 2^-22), and exp(delta) < 2e-35 below,
// where u = 0 alone can accept; u is a multiple of 2^-32.
__device__ __forceinline__ bool accept_delta(double delta, double u) {
  if (delta >= 0.0) return true;
  const float d = (float)delta, uf = (float)u;
  if (d > -80.0f) {
    const float p = ex2_approx(__fmul_rn(d, 1.4426950409f));
    if (uf < p * 0.9999f) return true;
    if (uf > p * 1.0001f) return false;
  } else if (uf > 0.0f) {
    return false;
  }
  return u < exp(delta);
}

// measure_add with each sum added in memory: the adds of one temperature come from one thread in
// interval order, each rounded to nearest as measure_add rounds it, and nothing waits for them.
// inv_N: 1 / N when N is a power of two (the products below are then the quotients), else 0.
__device__ __forceinline__ void measure_red(double *acc, double E, long long M, double Nd, double inv_N) {
  const double e = inv_N != 0.0 ? E * inv_N : E / Nd;
  const double m = inv_N != 0.0 ? (double)M * inv_N : (double)M / Nd;
  const double m2 = __dmul_rn(m, m);
  atomicAdd(acc + 0, e);
  atomicAdd(acc + 1, __dmul_rn(e, e));
  atomicAdd(acc + 2, fabs(m));
  atomicAdd(acc + 3, m2);
  atomicAdd(acc + 4, __dmul_rn(__dmul_rn(m2, m), m));
}

}  // namespace rfim

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

// Copy of the exchange state each CTA keeps, one entry per replica or temperature.
struct ResidentState {
  double *E, *beta;
  int32_t *M, *t2r, *r2t;
  uint8_t *swapped;
};

__host__ __device__ constexpr size_t resident_state_bytes(int rcap) { return ((size_t)rcap * 29 + 32 + 15) / 16 * 16; }

struct alignas(16) ChunkSum {
  int B, M;
  long long F;
};

// Self-test of waits that are given up, in the debug build (in the release build it cost up to 3 %, by the
// registers): CTA `cta` of a launch acts as if it had given up a wait when it starts interval `iv` of the
// launch (-1: no CTA does).
struct SelftestStop {
  int32_t cta, iv;
};
__device__ __forceinline__ bool stops_here(const SelftestStop &s, int iv, unsigned *err) {
  if ((int)blockIdx.x != s.cta || iv != s.iv) return false;
  if (threadIdx.x == 0) atomicOr(err, 2u);
  return true;
}

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

// The record of interval `epoch`, polled at most `polls` times; false when it did not arrive
// (recorded in *err) or an earlier wait of this launch expired.
__device__ __forceinline__ bool record_await(const uint4 *rec, uint32_t epoch, unsigned *err, int *B, int *M, long long *F,
                                             unsigned polls = kRecordSpinLimit) {
  for (unsigned it = 0; it < polls; ++it) {
    unsigned long long hi;
    record_load(rec, F, &hi);
    if ((uint32_t)(hi >> 42) == epoch) {
      *B = record_bonds(hi);
      *M = record_spin(hi);
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
// POW2: N is a power of two, so that the products with 1 / N are the quotients.
template <bool POW2>
__device__ __forceinline__ void measure_red(double *acc, double E, long long M, double Nd) {
  const double e = POW2 ? E * (1.0 / Nd) : E / Nd;
  const double m = POW2 ? (double)M * (1.0 / Nd) : (double)M / Nd;
  const double m2 = __dmul_rn(m, m);
  atomicAdd(acc + 0, e);
  atomicAdd(acc + 1, __dmul_rn(e, e));
  atomicAdd(acc + 2, fabs(m));
  atomicAdd(acc + 3, m2);
  atomicAdd(acc + 4, __dmul_rn(__dmul_rn(m2, m), m));
}

// Exchange step j over the records of interval `epoch` (slabs per replica: S), taken by every CTA of
// the launch on its own copy xs of the temperature assignment: energies E = energy_of(bonds, field
// sum), the swap decisions of the disjoint pairs (Eq. 2, Sec. 3.3), and, for the temperatures
// k = CTA mod number of CTAs, the pair counts and the measurement (Sec. 7).  All threads of the CTA
// call it; the assignment is complete when it returns.  False, and nothing is exchanged, when a thread of the
// CTA has given up a wait: for a record here, or before with *gave_up set (in shared memory).
template <bool REAL, bool POW2 = !REAL, class F>
__device__ __forceinline__ bool exchange_from_records(const RealView &v, const ExchArgs &xa, const ResidentState &xs,
                                                      const uint4 *rec, int S, uint32_t epoch, uint32_t j,
                                                      volatile uint32_t *gave_up, F energy_of) {
  const int nt = blockDim.x, tid = threadIdx.x, R = v.R;
  const int p0 = (int)(j & 1u) + 2 * tid;  // this thread's first pair
  auto random_of = [&](int k) {
    return philox10(v.seed, v.realization, (uint32_t)k, 0u, j, tag_word(kTagExch, v.stage, 0)).w[0];
  };
  // the random number of the first pair does not depend on the energies
  const uint32_t u0 = p0 + 1 < R ? random_of(p0) : 0u;
  // One lane per record, the S lanes of a replica (a power of two up to 16) then add theirs in a tree;
  // REAL: the 64-bit field sums are doubles.  Every CTA polls every record, so the lines they lie in
  // are what the step waits for: a warp's load takes each line once (a lane per replica that read
  // its S records one after another took it S times; L = 24, R = 40, eight slabs: 8.7 us for the
  // whole tail of an interval, 6.4 so, and 6.0 with the energies on bytes from registers as well).
  if (S == 1 || (S & (S - 1)) != 0) {  // one slab, or a number of slabs that no default shape has
    for (int r = tid; r < R; r += nt) {
      int B = 0, M = 0;
      long long F = 0;
      for (int q = 0; q < S; ++q) {
        int b, m;
        long long f;
        if (!record_await(rec + (size_t)r * S + q, epoch, xa.err, &b, &m, &f)) *gave_up = 1u;
        B += b;
        M += m;
        F = REAL && q > 0 ? __double_as_longlong(__dadd_rn(__longlong_as_double(F), __longlong_as_double(f))) : F + f;
      }
      xs.E[r] = energy_of(B, F);
      xs.M[r] = M;
    }
  } else {
    for (int n0 = (tid >> 5) * 32; n0 < R * S; n0 += nt & ~31) {
      const int n = n0 + (tid & 31), r = n / S;
      int B = 0, M = 0;
      long long F = 0;
      if (n < R * S && !record_await(rec + n, epoch, xa.err, &B, &M, &F)) *gave_up = 1u;
      __syncwarp();
      for (int o = S / 2; o > 0; o >>= 1) {
        B += __shfl_xor_sync(0xffffffffu, B, o);
        M += __shfl_xor_sync(0xffffffffu, M, o);
        const long long G = __shfl_xor_sync(0xffffffffu, F, o);
        F = REAL ? __double_as_longlong(__dadd_rn(__longlong_as_double(F), __longlong_as_double(G))) : F + G;
      }
      if (n < R * S && n % S == 0) {
        xs.E[r] = energy_of(B, F);
        xs.M[r] = M;
      }
    }
  }
  __syncthreads();
  if (*gave_up) return false;
  for (int k = p0; k + 1 < R; k += 2 * nt) {
    const int a = xs.t2r[k], b = xs.t2r[k + 1];
    const uint32_t u = k == p0 ? u0 : random_of(k);
    const bool acc = accept_delta((xs.beta[k] - xs.beta[k + 1]) * (xs.E[a] - xs.E[b]), (double)u * 0x1p-32);
    xs.swapped[k] = acc;
    if (acc) {
      xs.t2r[k] = b;
      xs.t2r[k + 1] = a;
      xs.r2t[b] = k;
      xs.r2t[a] = k + 1;
    }
  }
  __syncthreads();
  const bool measure = (int64_t)j >= xa.measure_from;
  for (int k = (int)blockIdx.x + (nt - 1 - tid) * (int)gridDim.x; k < R; k += nt * (int)gridDim.x) {
    if (((uint32_t)k & 1u) == (j & 1u) && k + 1 < R) {
      atomicAdd(reinterpret_cast<unsigned long long *>(v.att) + k, 1ull);
      if (xs.swapped[k]) atomicAdd(reinterpret_cast<unsigned long long *>(v.acc) + k, 1ull);
    }
    const int a = xs.t2r[k];
    if (measure) measure_red<POW2>(v.obs + (int64_t)k * 5, xs.E[a], xs.M[a], (double)v.N);
    if (k == 0 && measure) atomicAdd(reinterpret_cast<unsigned long long *>(v.n_meas), 1ull);
  }
  return true;
}

}  // namespace rfim

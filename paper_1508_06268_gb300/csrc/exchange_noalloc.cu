// rfim_exchange_noalloc: the energy reduction and exchange step on caller-owned device buffers,
// with its scratch (per-(replica, slab) partial sums and the arrival counter) in a file-scope
// device array instead of memory the library allocates.  For callers that cannot allocate
// device memory: a framework or arena that owns all of it, or a latency-critical loop where
// cudaMalloc / cudaFree would synchronise the device.
//
// The array is shared by every call on a device and keeps the last call's contents; calls that
// overlap on the GPU (different streams, or host threads without ordering) race on it.  The
// arrival counter starts at zero (a file-scope device array is zero when the module loads) and
// the last CTA of each call sets it back to zero.
#include <algorithm>
#include <cstdint>
#include <string>

#include "rfim.h"
#include "bits_layout.cuh"
#include "debug_check.cuh"
#include "exchange.cuh"
#include "exchange_records.cuh"
#include "internal.h"
#include "lattice.cuh"

namespace rfim {

namespace {

// Scratch capacity: R * slabs partial slots of 16 bytes plus the counter: 256 KiB + 256.
constexpr int kNoAllocSlots = 16384;
constexpr size_t kCounterOffset = (size_t)kNoAllocSlots * 16;
constexpr size_t kScratchBytes = kCounterOffset + 256;
// Replicas whose exchange state the last CTA keeps in shared memory (16 bytes each).
constexpr int kNoAllocShared = 1024;
constexpr int kNoAllocThreads = 256;

static __device__ __align__(256) unsigned char g_exchange_scratch[kScratchBytes];

// Partial of one (replica, slab): field term (bimodal: integer sum of h s, else double sum of hh s),
// bond sum, magnetisation.
struct alignas(16) NoAllocPart {
  long long F;
  int B, M;
};

struct NoAllocArgs {
  RealView v;
  const float *field;  // unscaled h_i, natural order
  float h;
  double J;
  int32_t slabs;
};

// s + e += s2 + e2 with the rounding error of the sum kept in e (Knuth's TwoSum).
__device__ __forceinline__ void sum2_add(float &s, float &e, float s2, float e2) {
  const float t = __fadd_rn(s, s2), bp = __fsub_rn(t, s);
  e = __fadd_rn(__fadd_rn(e, e2), __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(s2, bp)));
  s = t;
}

// One CTA per (RG replicas, slab of words); the last CTA to arrive adds the partials in slab order,
// forms E = -J B - F and takes exchange step j and the measurement.
//
// Bound: latency (at L = 32, R = 70 the call reads 0.4 MB), so every phase is spread over many
// lanes and loads do not wait for one another.
//   - Field term: word wq of the two colours holds the sites 64 wq .. 64 wq + 63 of the natural
//     order, so a warp takes one pair of words at a time, lane l the sites l and l + 32: two
//     coalesced field loads serve RG replicas, whose words every lane reads (broadcast).  With
//     one thread per word, 32 strided loads and a chain of 32 error-free sums, and the last CTA
//     reading its state and adding the sums through L2, a call at L = 32, R = 70 took 17.2 us
//     from the host's call to the result; it takes 11.9 us.
//   - RG = 4 shares the field loads between replicas where that leaves at least a CTA per SM;
//     RG = 1 keeps more CTAs where the realization is small (L = 8, R = 16: 16 CTAs instead of 4).
//   - The error-free float sums (running sum and the sum of its rounding errors) are joined across
//     the warp as such; doubles, of which an SM adds two per cycle, only add the warps' sums.
//   - While the last arrival is counted, every CTA has the temperature assignment and the random
//     number of its threads' first pair; the last one decides from shared memory, and the
//     counts and measurement sums are added in memory without waiting.
template <int L, int RG, bool BIM>
__global__ void __launch_bounds__(kNoAllocThreads) k_exchange_noalloc(NoAllocArgs a, uint32_t j, int64_t measure_from,
                                                                      unsigned char *scratch) {
  using Gm = BitsGeom<L>;
  constexpr int P = Gm::P, W = Gm::W, NW = kNoAllocThreads / 32;
  const RealView &v = a.v;
  NoAllocPart *part = reinterpret_cast<NoAllocPart *>(scratch);
  unsigned int *counter = reinterpret_cast<unsigned int *>(scratch + kCounterOffset);
  __shared__ int sB[RG], sM[RG];
  __shared__ int si[NW][RG];
  __shared__ double sd[NW][RG];
  __shared__ int last;
  __shared__ double E_s[kNoAllocShared];
  __shared__ int32_t M_s[kNoAllocShared], t2r_s[kNoAllocShared];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, R = v.R;
  const bool shared_state = R <= kNoAllocShared;
  const int grp = blockIdx.x / a.slabs, slab = blockIdx.x % a.slabs;
  const int r0 = grp * RG, gact = min(RG, R - r0);
  // debug build: this CTA's partial slots must lie inside the static array (else it writes none)
  const bool slot_ok = RFIM_DCHECK(counter + 1, gact >= 1 && (r0 + gact) * a.slabs <= kNoAllocSlots, kDbgScratch);
  const int w0 = slab * W / a.slabs, nwd = (slab + 1) * W / a.slabs - w0;
  if (tid < RG) sB[tid] = sM[tid] = 0;
  const int p0 = (int)(j & 1u) + 2 * tid;  // this thread's first pair
  double db0 = 0.0;
  uint32_t u0 = 0u;
  auto random_of = [&](int k) {
    return philox10(v.seed, v.realization, (uint32_t)k, 0u, j, tag_word(kTagExch, v.stage, 0)).w[0];
  };
  if (shared_state)
    for (int k = tid; k < R; k += kNoAllocThreads) t2r_s[k] = v.t2r[k];
  if (p0 + 1 < R) {
    db0 = v.beta_d[p0] - v.beta_d[p0 + 1];
    u0 = random_of(p0);
  }
  __syncthreads();

  // bond sum over the colour-0 words (six neighbour words each) and magnetisation over all words
  const int chunks = (2 * nwd + 31) / 32;
  for (int u = wid; u < gact * chunks; u += NW) {
    const int g = u / chunks, e = u % chunks * 32 + lane;
    int b = 0, m = 0;
    if (e < 2 * nwd) {
      const int c = e / nwd, wq = w0 + e % nwd, z = wq / P, iw = wq % P;
      const uint32_t *S0 = v.bits + (int64_t)(r0 + g) * 2 * W, *O = S0 + W;
      const uint32_t self = S0[c * W + wq];
      m = 2 * __popc(self) - 32;
      if (c == 0) {
        uint32_t A, B, C, D;
        nb_xy<L>(O[wq], O[z * P + (iw + 1) % P], O[z * P + (iw + P - 1) % P], parity0_mask<L>(0, z, iw), A, B, C, D);
        const uint32_t U = O[((z + 1) % L) * P + iw], V = O[((z + L - 1) % L) * P + iw];
        b = 6 * 32 - 2 * (__popc(self ^ A) + __popc(self ^ B) + __popc(self ^ C) + __popc(self ^ D) + __popc(self ^ U) +
                          __popc(self ^ V));
      }
    }
    b = __reduce_add_sync(0xffffffffu, b);
    m = __reduce_add_sync(0xffffffffu, m);
    if (lane == 0) {
      atomicAdd(&sB[g], b);
      atomicAdd(&sM[g], m);
    }
  }

  // field term: sites n = lane and lane + 32 of a word pair, in-word position n / 2, colour
  // (x + y + z) mod 2 with x = n mod L, y = (first row of the word) + n / L
  int fi[RG];
  float fs[RG], fe[RG];
#pragma unroll
  for (int g = 0; g < RG; ++g) {
    fi[g] = 0;
    fs[g] = fe[g] = 0.f;
  }
#pragma unroll 2
  for (int w = wid; w < nwd; w += NW) {
    const int wq = w0 + w, z = wq / P, iw = wq % P;
    const int y0 = L == 64 ? iw : iw * (64 / L);
    const float hv[2] = {a.field[64 * (int64_t)wq + lane], a.field[64 * (int64_t)wq + lane + 32]};
    uint32_t s[RG][2];
#pragma unroll
    for (int g = 0; g < RG; ++g) {
      const uint32_t *S = v.bits + (int64_t)(r0 + min(g, gact - 1)) * 2 * W + wq;
      s[g][0] = S[0];
      s[g][1] = S[W];
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int n = lane + 32 * q, bit = (int)bit_of(n >> 1);
      const int c = (n % L + y0 + n / L + z) & 1;
#pragma unroll
      for (int g = 0; g < RG; ++g) {
        const uint32_t down = (~(c ? s[g][1] : s[g][0]) >> bit) & 1u;
        if (BIM) {
          fi[g] += (down != 0u) == (hv[q] > 0.0f) ? -1 : 1;
        } else {
          const float hh = __fmul_rn(a.h, hv[q]);
          sum2_add(fs[g], fe[g], __uint_as_float(__float_as_uint(hh) ^ (down << 31)), 0.f);
        }
      }
    }
  }
  if (BIM) {
#pragma unroll
    for (int g = 0; g < RG; ++g) {
      const int t = __reduce_add_sync(0xffffffffu, fi[g]);
      if (lane == 0) si[wid][g] = t;
    }
  } else {
    // RG sums over 32 lanes: each halving step hands half of the sums still held to the partner
    int g = 0;
#pragma unroll
    for (int n = RG, o = 16; o > 0; o >>= 1) {
      if (n > 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < n / 2; ++i) {
          const float ss = up ? fs[i] : fs[i + n / 2], se = up ? fe[i] : fe[i + n / 2];
          const float ks = up ? fs[i + n / 2] : fs[i], ke = up ? fe[i + n / 2] : fe[i];
          fs[i] = ks;
          fe[i] = ke;
          sum2_add(fs[i], fe[i], __shfl_xor_sync(0xffffffffu, ss, o), __shfl_xor_sync(0xffffffffu, se, o));
        }
        n /= 2;
        g += up ? n : 0;
      } else {
        sum2_add(fs[0], fe[0], __shfl_xor_sync(0xffffffffu, fs[0], o), __shfl_xor_sync(0xffffffffu, fe[0], o));
      }
    }
    if (lane % (32 / RG) == 0) sd[wid][g] = (double)fs[0] + (double)fe[0];
  }
  __syncthreads();
  if (tid < 8 * RG) {  // the warps' sums of replica g: eight lanes each
    static_assert(NW == 8, "eight lanes add the warps' sums of a replica");
    const unsigned mask = RG * 8 == 32 ? 0xffffffffu : (1u << (RG * 8)) - 1u;
    const int g = tid / 8;
    long long F = 0;
    if (BIM) {
      int t = si[tid % 8][g];
      for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(mask, t, o);
      F = t;
    } else {
      double t = sd[tid % 8][g];
      for (int o = 4; o > 0; o >>= 1) t = __dadd_rn(t, __shfl_xor_sync(mask, t, o));
      F = __double_as_longlong(t);
    }
    if (tid % 8 == 0 && g < gact && slot_ok) part[(int64_t)(r0 + g) * a.slabs + slab] = NoAllocPart{F, sB[g], sM[g]};
  }
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  // four lanes per replica add its slabs' partials
  for (int base = 0; base < R; base += kNoAllocThreads / 4) {
    const int r = base + tid / 4;
    int tb = 0, tm = 0;
    long long tf = 0;
    double td = 0.0;
    if (r < R) {
#pragma unroll 4
      for (int q = tid % 4; q < a.slabs; q += 4) {
        const int4 x = __ldcg(reinterpret_cast<const int4 *>(part) + (int64_t)r * a.slabs + q);
        const long long F = (long long)(((unsigned long long)(uint32_t)x.y << 32) | (uint32_t)x.x);
        if (BIM)
          tf += F;
        else
          td += __longlong_as_double(F);
        tb += x.z;
        tm += x.w;
      }
    }
#pragma unroll
    for (int o = 2; o > 0; o >>= 1) {
      tb += __shfl_xor_sync(0xffffffffu, tb, o);
      tm += __shfl_xor_sync(0xffffffffu, tm, o);
      if (BIM)
        tf += __shfl_xor_sync(0xffffffffu, tf, o);
      else
        td += __shfl_xor_sync(0xffffffffu, td, o);
    }
    if (r < R && tid % 4 == 0) {
      const double E = -a.J * (double)tb - (BIM ? (double)a.h * (double)tf : td);
      v.E[r] = E;
      v.M[r] = tm;
      if (shared_state) {
        E_s[r] = E;
        M_s[r] = tm;
      }
    }
  }
  if (tid == 0) *counter = 0u;
  __syncthreads();
  if (!shared_state) {
    exchange_and_measure(v, j, measure_from);
    return;
  }
  for (int k = p0; k + 1 < R; k += 2 * kNoAllocThreads) {
    const int ra = t2r_s[k], rb = t2r_s[k + 1];
    const double db = k == p0 ? db0 : v.beta_d[k] - v.beta_d[k + 1];
    const uint32_t u = k == p0 ? u0 : random_of(k);
    atomicAdd(reinterpret_cast<unsigned long long *>(v.att) + k, 1ull);
    if (accept_delta(db * (E_s[ra] - E_s[rb]), (double)u * 0x1p-32)) {
      atomicAdd(reinterpret_cast<unsigned long long *>(v.acc) + k, 1ull);
      t2r_s[k] = v.t2r[k] = rb;
      t2r_s[k + 1] = v.t2r[k + 1] = ra;
      v.r2t[rb] = k;
      v.r2t[ra] = k + 1;
    }
  }
  if ((int64_t)j < measure_from) return;
  __syncthreads();
  for (int k = tid; k < R; k += kNoAllocThreads) {
    const int r = t2r_s[k];
    measure_red<true>(v.obs + (int64_t)k * 5, E_s[r], M_s[r], (double)v.N);
  }
  if (tid == 0) atomicAdd(reinterpret_cast<unsigned long long *>(v.n_meas), 1ull);
}

using NoAllocFn = void (*)(NoAllocArgs, uint32_t, int64_t, unsigned char *);

template <int L>
NoAllocFn noalloc_kernel(int RG, bool bim) {
  if (RG == 4) return bim ? k_exchange_noalloc<L, 4, true> : k_exchange_noalloc<L, 4, false>;
  return bim ? k_exchange_noalloc<L, 1, true> : k_exchange_noalloc<L, 1, false>;
}

}  // namespace

}  // namespace rfim

using namespace rfim;

extern "C" int rfim_exchange_noalloc(const rfim_exchange_buffers *b, uint32_t j, int64_t measure_from, void *stream) {
  if (!b) return set_thread_error(RFIM_EINVAL, "rfim_exchange_noalloc: null buffers");
  const int32_t L = b->L, R = b->R;
  if (!(L == 8 || L == 16 || L == 32 || L == 64))
    return set_thread_error(RFIM_EINVAL, "rfim_exchange_noalloc: L must be 8, 16, 32 or 64");
  if (R < 2) return set_thread_error(RFIM_EINVAL, "rfim_exchange_noalloc: R must be >= 2");
  if (!b->spins || !b->field || !b->beta || !b->t2r || !b->r2t || !b->att || !b->acc || !b->obs || !b->n_meas || !b->E ||
      !b->M)
    return set_thread_error(RFIM_EINVAL, "rfim_exchange_noalloc: a buffer pointer is null");
  // Four replicas per CTA where slabs of 32 word pairs then still give every SM a CTA, else one.
  // Slabs: up to four CTAs per SM, none below eight word pairs (one per warp; 32 with four replicas,
  // whose sums cost more to join), bounded by the scratch capacity.
  const int words = L * L * L / 64;
  const int RG = (int64_t)((R + 3) / 4) * (words / 32) >= 152 ? 4 : 1, groups = (R + RG - 1) / RG;
  int slabs = std::max(1, std::min(words / (RG == 4 ? 32 : 8), 608 / groups));
  if ((int64_t)R * slabs > kNoAllocSlots) slabs = kNoAllocSlots / R;
  if (slabs < 1)
    return set_thread_error(RFIM_EINVAL, "rfim_exchange_noalloc: R exceeds the static scratch capacity (16384 replicas)");
  cudaStream_t st = (cudaStream_t)stream;
  // In host code g_exchange_scratch names a host-side stand-in, not device memory: the kernel
  // gets the array's device address on the current device, looked up on every call (no stream
  // work; a cached address would go stale after cudaDeviceReset).
  unsigned char *scratch = nullptr;
  cudaError_t e = cudaGetSymbolAddress((void **)&scratch, g_exchange_scratch);
  if (e != cudaSuccess || !scratch)
    return set_thread_error(RFIM_ECUDA, std::string("rfim_exchange_noalloc: cudaGetSymbolAddress: ") +
                                            cudaGetErrorString(e));
  NoAllocArgs a{};
  a.v.L = L;
  a.v.Lh = L / 2;
  a.v.N = L * L * L;
  a.v.R = R;
  a.v.kind = b->field_kind == RFIM_FIELD_BIMODAL ? kBimodal : kGaussian;
  a.v.seed = b->seed;
  a.v.realization = b->realization;
  a.v.stage = b->stage;
  a.v.bits = const_cast<uint32_t *>(b->spins);
  a.v.beta_d = b->beta;
  a.v.t2r = b->t2r;
  a.v.r2t = b->r2t;
  a.v.E = b->E;
  a.v.M = b->M;
  a.v.att = b->att;
  a.v.acc = b->acc;
  a.v.obs = b->obs;
  a.v.n_meas = b->n_meas;
  a.field = b->field;
  a.h = b->h;
  a.J = (double)b->J;
  a.slabs = slabs;
  const bool bim = a.v.kind == kBimodal;
  const NoAllocFn fn = L == 8    ? noalloc_kernel<8>(RG, bim)
                       : L == 16 ? noalloc_kernel<16>(RG, bim)
                       : L == 32 ? noalloc_kernel<32>(RG, bim)
                                 : noalloc_kernel<64>(RG, bim);
  fn<<<groups * slabs, kNoAllocThreads, 0, st>>>(a, j, measure_from, scratch);
  e = cudaGetLastError();
  if (e != cudaSuccess)
    return set_thread_error(RFIM_ECUDA, std::string("rfim_exchange_noalloc: launch: ") + cudaGetErrorString(e));
  if (kDebugBuild) {  // debug build only: wait for the launch and report its bounds checks
    unsigned int word = 0, zero = 0;
    unsigned int *err = reinterpret_cast<unsigned int *>(scratch + kCounterOffset) + 1;
    e = cudaMemcpyAsync(&word, err, 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess && word) e = cudaMemcpyAsync(err, &zero, 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess)
      return set_thread_error(RFIM_ECUDA, std::string("rfim_exchange_noalloc: ") + cudaGetErrorString(e));
    if (word) return set_thread_error(RFIM_EBOUNDS, "rfim_exchange_noalloc: a bounds check of the debug build failed");
  }
  return RFIM_OK;
}

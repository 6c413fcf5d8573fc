// Instances of the resident sweep kernel that measure the structure factor too (kernels_resident.cuh, XI): those
// of kernels_resident.cu.
#include "resident.h"

namespace rfim {

namespace {

struct XiInstance {
  int32_t L, S, NB;
  bool one;
  ResidentFn bim, flt;
};

template <int L, int S, int NB, int NT, bool ONE>
constexpr XiInstance xi_instance() {
  return {L, S, NB, ONE, k_resident<L, S, NB, true, NT, ONE, 0, true>, k_resident<L, S, NB, false, NT, ONE, 0, true>};
}

const XiInstance kXiInstances[] = {
    xi_instance<8, 1, 1, 512, true>(),   xi_instance<8, 1, 2, 512, true>(),   xi_instance<8, 1, 4, 512, true>(),
    xi_instance<16, 1, 1, 512, true>(),  xi_instance<16, 1, 2, 512, true>(),  xi_instance<16, 1, 4, 512, true>(),
    xi_instance<16, 2, 1, 256, true>(),  xi_instance<16, 2, 2, 256, true>(),  xi_instance<32, 2, 4, 512, true>(),
    xi_instance<32, 4, 4, 256, true>(),  xi_instance<32, 8, 2, 256, true>(),  xi_instance<32, 1, 4, 512, false>(),
    xi_instance<32, 2, 4, 512, false>(), xi_instance<64, 16, 4, 512, true>(), xi_instance<64, 8, 4, 512, false>(),
    xi_instance<64, 4, 4, 512, false>(),
};

}  // namespace

ResidentFn resident_xi_kernel(int32_t L, int32_t S, int32_t NB, bool one, bool bimodal) {
  for (const XiInstance &i : kXiInstances)
    if (i.L == L && i.S == S && i.NB == NB && i.one == one) return bimodal ? i.bim : i.flt;
  return nullptr;
}

}  // namespace rfim

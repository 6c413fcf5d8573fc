// Instances of the resident sweep kernel for the multi-hit double checkerboard (kernels_resident.cuh, T > 0).
#include "resident.h"

namespace rfim {

const std::vector<ResidentInstance> &resident_multihit_instances() {
  static const std::vector<ResidentInstance> all = {
      resident_instance<16, 1, 1, 512, true, 8>(),   resident_instance<16, 1, 2, 512, true, 8>(),
      resident_instance<16, 1, 4, 512, true, 8>(),   resident_instance<32, 4, 1, 512, true, 8>(),
      resident_instance<32, 4, 2, 512, true, 8>(),   resident_instance<32, 2, 2, 512, true, 8>(),
      resident_instance<32, 2, 4, 512, true, 8>(),   resident_instance<32, 4, 1, 512, true, 16>(),
      resident_instance<32, 2, 2, 512, true, 16>(),  resident_instance<32, 2, 4, 512, true, 16>(),
      resident_instance<64, 16, 2, 512, true, 8>(),  resident_instance<64, 8, 4, 512, true, 8>(),
      resident_instance<64, 4, 4, 512, false, 8>(),  resident_instance<64, 16, 2, 512, true, 16>(),
      resident_instance<64, 8, 4, 512, true, 16>(),  resident_instance<64, 4, 4, 512, false, 16>(),
      resident_instance<64, 16, 2, 512, true, 32>(), resident_instance<64, 8, 4, 512, true, 32>(),
      resident_instance<64, 4, 4, 512, false, 32>(),
  };
  return all;
}

}  // namespace rfim

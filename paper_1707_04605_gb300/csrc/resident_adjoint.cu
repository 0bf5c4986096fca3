// Instances of the resident reverse steps.
#include "resident_adjoint.cuh"

namespace mg {

int launch_resident_adjoint(const ResidentAdjArgs& a, const ResidentShape& s, cudaStream_t st) {
  switch (s.lpr) {
    case 1: return launch_adj<1>(a, s, st);
    case 2: return launch_adj<2>(a, s, st);
    case 4: return launch_adj<4>(a, s, st);
    case 8: return launch_adj<8>(a, s, st);
    case 16: return launch_adj<16>(a, s, st);
    case 32: return launch_adj<32>(a, s, st);
  }
  return MG_ERR_ARG;
}

}  // namespace mg

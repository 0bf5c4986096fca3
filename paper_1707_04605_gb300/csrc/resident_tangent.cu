// Instances of the resident forward + tangent kernel.
#include "resident_step.cuh"

namespace mg {

int launch_resident_tangent(const ResidentArgs& a, const ResidentShape& s, cudaStream_t st) {
  switch (s.lpr) {
    case 2: return launch_lpr<2, true>(a, s, st);
    case 4: return launch_lpr<4, true>(a, s, st);
    case 8: return launch_lpr<8, true>(a, s, st);
    case 16: return launch_lpr<16, true>(a, s, st);
    case 32: return launch_lpr<32, true>(a, s, st);
  }
  return MG_ERR_ARG;
}

}  // namespace mg

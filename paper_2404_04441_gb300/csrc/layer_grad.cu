// The CPML layer's unrolled line ends for the gradient: the recompute (which
// also updates D) and the adjoint.
#include "layer_lines.cuh"

namespace gbw {

template void cpml_launch_lines<float, true>(const CpmlPlan &, const CpmlTiles &, const CpmlPass &,
                                             bool, cudaStream_t);

void cpml_launch_adjoint_lines(const CpmlPlan &p, const CpmlTiles &t, const CpmlPass &a,
                               cudaStream_t st) {
  switch (p.variant) {
    case 0: return cpml_launch<CpmlAdjoint<8>>(p, t, a, false, st);
    case 1: return cpml_launch<CpmlAdjoint<10>>(p, t, a, false, st);
    case 2: return cpml_launch<CpmlAdjoint<16>>(p, t, a, false, st);
    default: return cpml_launch<CpmlAdjoint<20>>(p, t, a, false, st);
  }
}

}  // namespace gbw

// The CPML layer's unrolled line ends for BF16 wavefields.
#include "layer_lines.cuh"

namespace gbw {

template void cpml_launch_lines<__nv_bfloat16, false>(const CpmlPlan &, const CpmlTiles &, const CpmlPass &,
                                           bool, cudaStream_t);
template void cpml_launch_batched_lines<__nv_bfloat16>(int, int, const CpmlBatchShot *, int, int, long long,
                                            cudaStream_t);

}  // namespace gbw

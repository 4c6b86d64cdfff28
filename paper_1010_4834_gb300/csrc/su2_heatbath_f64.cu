// The heat-bath substep (su2_heatbath.cuh) for FP64 links.
#include "su2_heatbath.cuh"

namespace su2 {

template cudaError_t launch_heatbath_prec<kF64>(const LatticeView&, int, int, const uint32_t*, uint32_t, const HBParams&, cudaStream_t, double*, int*);

}  // namespace su2

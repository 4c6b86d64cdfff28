// The heat-bath substep's launcher: one instantiation of su2_heatbath.cuh per
// link precision.
#include "su2_internal.h"
#include "su2_kernel_util.cuh"

namespace su2 {

template <int P>
cudaError_t launch_heatbath_prec(const LatticeView& v, int mu, int parity, const uint32_t* sweep_base,
                                 uint32_t sweep_off, const HBParams& hp, cudaStream_t st,
                                 double* meas, int* meas_blocks);

cudaError_t launch_heatbath(const LatticeView& v, int mu, int parity, const uint32_t* sweep_base,
                            uint32_t sweep_off, const HBParams& hp,
                            cudaStream_t st, double* meas, int* meas_blocks) {
  SU2_DISPATCH(v.prec, return launch_heatbath_prec<P>(v, mu, parity, sweep_base, sweep_off, hp, st, meas, meas_blocks));
  return cudaErrorInvalidValue;
}

}  // namespace su2

#define SU2_COMPILER_FUSES
#include "su2_batch_kernel.cuh"

namespace su2 {

template cudaError_t launch_batch_groups<kF32, false>(int, int, const BatchArgs&, cudaStream_t);
template int batch_blocks_per_sm<kF32, false>(int);

}  // namespace su2

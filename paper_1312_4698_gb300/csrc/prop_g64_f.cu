// Instantiations of the FP64 lane-group propagation kernel (split for parallel builds).
#include "propagate_g64.cuh"

namespace scivr {

template cudaError_t launch_group_fp64<9>(const PropLaunch &, cudaStream_t);

}  // namespace scivr

// FP32 stage solves of the mixed-precision mode.
#include "gmres_kernels.cuh"

namespace pp {

template cudaError_t launch_stage_gmres<float>(const DevMesh&, int, const StageGmres<float>&, cudaStream_t);

}  // namespace pp

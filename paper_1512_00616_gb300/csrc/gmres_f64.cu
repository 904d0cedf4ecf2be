// FP64 stage solves (a translation unit of their own, so that the two precisions compile in parallel).
#include "gmres_kernels.cuh"

namespace pp {

size_t stage_gmres_partial_words() { return (size_t)2 * GLD * GCTAS; }
int stage_gmres_barrier_words() { return BAR_WORDS; }

template cudaError_t launch_stage_gmres<double>(const DevMesh&, int, const StageGmres<double>&, cudaStream_t);

}  // namespace pp

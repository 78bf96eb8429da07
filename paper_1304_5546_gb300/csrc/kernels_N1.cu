// Order-1 instantiations of the node-thread FP32 stage kernel (uniform
// medium and per-element permittivity).
#include "kernels.cuh"

namespace dgw {
template cudaError_t launch_stage<1>(const StageArgs<float>&, int, int, cudaStream_t);
template cudaError_t launch_stage_media<1>(const StageArgs<float>&, int, int, cudaStream_t);
}  // namespace dgw

// Order-4 instantiations of the element-row FP32 stage kernel (uniform
// medium and per-element permittivity).
#include "kernels_er.cuh"

namespace dgw {
template cudaError_t launch_stage_er<4>(const StageArgs<float>&, const float*, bool, int, int,
                                        cudaStream_t);
}  // namespace dgw

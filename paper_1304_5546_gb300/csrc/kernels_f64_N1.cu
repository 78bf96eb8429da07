// Order-1 instantiations of the FP64 stage kernel (uniform medium and
// per-element permittivity).
#include "kernels_f64.cuh"

namespace dgw {
template cudaError_t launch_stage_f64<1>(const StageArgs<double>&, bool, int, int, cudaStream_t);
}  // namespace dgw

// Order-1 instantiations of the FP32 tensor-core stage kernel with 3xTF32
// products: uniform medium, per-element permittivity (each with its
// alternative element-block size where there is one), and the order's
// kernels of the concurrent batched launch.
#include "kernels_tc.cuh"

namespace dgw {
template cudaError_t launch_stage_tc<1, kTcTf32x3>(const StageArgs<float>&, int, int, cudaStream_t);
template cudaError_t launch_stage_tc_media<1>(const StageArgs<float>&, int, int, cudaStream_t);
template cudaError_t launch_batch_order<1, kModeFirstStage>(const StageArgs<float>&, int, bool,
                                                      cudaStream_t);
template cudaError_t launch_batch_order<1, kModeStage>(const StageArgs<float>&, int, bool,
                                                      cudaStream_t);
template cudaError_t launch_batch_order<1, kModeFirstStage, true>(const StageArgs<float>&, int, bool,
                                                                   cudaStream_t);
template cudaError_t launch_batch_order<1, kModeStage, true>(const StageArgs<float>&, int, bool,
                                                              cudaStream_t);
}  // namespace dgw

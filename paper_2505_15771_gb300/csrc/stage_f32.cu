// FP32 stage kernels (batched shots, the FP32 adjoint).
#include "stage_kernels.cuh"

namespace hho_stage {

#define HHO_INSTANTIATE(K) \
    template void launch_stage<float, K, MODE_TRACES>(const StageArgsT<float>&, int, cudaStream_t); \
    template void launch_stage<float, K, MODE_STAGE>(const StageArgsT<float>&, int, cudaStream_t); \
    template void launch_stage<float, K, MODE_APPLY>(const StageArgsT<float>&, int, cudaStream_t); \
    template void launch_grad<float, K>(const StageArgsT<float>&, const GradArgsT<float>&, cudaStream_t);

HHO_INSTANTIATE(1)
HHO_INSTANTIATE(2)
HHO_INSTANTIATE(3)

}  // namespace hho_stage

// FP64 stage kernels.
#include "stage_kernels.cuh"

namespace hho_stage {

#define HHO_INSTANTIATE(K) \
    template void launch_stage<double, K, MODE_TRACES>(const StageArgsT<double>&, int, cudaStream_t); \
    template void launch_stage<double, K, MODE_STAGE>(const StageArgsT<double>&, int, cudaStream_t); \
    template void launch_stage<double, K, MODE_APPLY>(const StageArgsT<double>&, int, cudaStream_t); \
    template void launch_grad<double, K>(const StageArgsT<double>&, const GradArgsT<double>&, cudaStream_t);

HHO_INSTANTIATE(1)
HHO_INSTANTIATE(2)
HHO_INSTANTIATE(3)

}  // namespace hho_stage

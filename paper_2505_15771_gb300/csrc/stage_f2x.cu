// Double-float stage kernels.
#include "stage_kernels.cuh"

namespace hho_stage {

#define HHO_INSTANTIATE(K) \
    template void launch_stage<f2x, K, MODE_TRACES>(const StageArgsT<f2x>&, int, cudaStream_t); \
    template void launch_stage<f2x, K, MODE_STAGE>(const StageArgsT<f2x>&, int, cudaStream_t); \
    template void launch_stage<f2x, K, MODE_APPLY>(const StageArgsT<f2x>&, int, cudaStream_t);

HHO_INSTANTIATE(1)
HHO_INSTANTIATE(2)
HHO_INSTANTIATE(3)

}  // namespace hho_stage

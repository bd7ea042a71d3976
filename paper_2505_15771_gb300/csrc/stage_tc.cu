// Tensor-core stage kernels (HHO_BF16X3) and their launcher.
#include "stage_kernels.cuh"
#include "tc.cuh"

namespace {
#include "stage_tc.cuh"
}  // namespace

namespace {
template <int K, int MODE>
struct TcTag {};
}  // namespace

namespace hho_stage {

// The tensor-core stage (HHO_BF16X3): 32 consecutive cells of one class
// (a class run is padded to 32 cells) times 4 shots per block, so that each
// warp reads 32 consecutive cells of one shot, as the FP32 kernel does.
template <int K, int MODE>
void launch_tc(const hho_ops* ops, const StageArgsT<float>& a, int n_shots, cudaStream_t s) {
    const int C = 32, S_blk = 128 / C;
    const dim3 grid((unsigned)((ops->dev.Nf + ops->dev.Ns) / C), (unsigned)((n_shots + S_blk - 1) / S_blk));
    if (grid.x == 0) return;
    TcArgs T;
    T.tiles = (const uint4*)ops->d_tc_b;
    T.meta = ops->d_tc_meta;
    T.C = C;
    T.S_blk = S_blk;
    T.n_shots = n_shots;
    T.kmax = ops->tc_kmax;
    T.cols = ops->tc_cols;
    T.error = ops->d_tc_err;
    const size_t smem = (size_t)2 * 2 * 128 * ops->tc_kmax + (size_t)ops->tc_bmax;
    stage_smem_attributes<TcTag<K, MODE>>(stage_tc_kernel<K, MODE>, smem, false);
    stage_tc_kernel<K, MODE><<<grid, 128, smem, s>>>(a, T);
}

#define HHO_INSTANTIATE(K) \
    template void launch_tc<K, MODE_TRACES>(const hho_ops*, const StageArgsT<float>&, int, cudaStream_t); \
    template void launch_tc<K, MODE_STAGE>(const hho_ops*, const StageArgsT<float>&, int, cudaStream_t);

HHO_INSTANTIATE(1)
HHO_INSTANTIATE(2)
HHO_INSTANTIATE(3)

}  // namespace hho_stage

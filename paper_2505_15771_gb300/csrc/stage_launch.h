// Launchers of the stage kernels, defined in stage_kernels.cuh and instantiated
// in one translation unit per arithmetic.
#pragma once

#include <cuda_runtime.h>

#include "hho_internal.h"

namespace hho_stage {

// One stage-kernel launch over the cells of both domains and n_shots shots.
template <class T, int K, int MODE>
void launch_stage(const StageArgsT<T>& a, int n_shots, cudaStream_t s);

// One backward stage's gradients (MODE_GRAD; FP64 and FP32).
template <class T, int K>
void launch_grad(const StageArgsT<T>& a, const GradArgsT<T>& g, cudaStream_t s);

// The tensor-core stage (HHO_BF16X3).
template <int K, int MODE>
void launch_tc(const hho_ops* ops, const StageArgsT<float>& a, int n_shots, cudaStream_t s);

}  // namespace hho_stage

// Launch parameters of the ERK stage kernels, per arithmetic and polynomial
// degree k (array index k - 1):
//   min_blocks  resident 128-thread blocks per SM asked of the register
//               allocator (__launch_bounds__): 8 allow 64 registers a
//               thread, 6 allow 80, 5 allow 96, 4 allow 128;
//   acc_smem    1: the cell's rate accumulators live in dynamic shared
//               memory instead of registers;
//   prefetch    mask of L2 prefetch hints (bits in
//               stage_kernels.cuh, L2Prefetch);
//   rect_loop   1: a rectangle's faces are traced by one body per
//               orientation looped over its two faces (compact code, fewer
//               live registers); 0: four unrolled bodies with constant signs.
// tune.py (beside the package) rewrites these tables from timings of
// candidate builds on the target GPU, over values that include all of these.
// The values here are the fastest found on GB300 for the 1024 x 512 bilayer
// (FP64, double-float), 16 shots of the 680 x 340 hybrid mesh (FP32, k = 3) and 21
// shots of the 331 x 167 hanging mesh (FP32, k = 2); the figures stand at
// MinBlocks, L2Prefetch and AccSmem in stage_kernels.cuh.
#pragma once

struct StageTuning {
    int min_blocks[3];
    int acc_smem[3];
    int prefetch[3];
    int rect_loop[3];
};

// tune.py: begin tables
constexpr StageTuning TUNED_F64 = {{8, 6, 4}, {0, 1, 0}, {0, 0, 0}, {0, 0, 0}};
constexpr StageTuning TUNED_F32 = {{8, 8, 6}, {0, 1, 1}, {50, 51, 51}, {0, 0, 0}};
constexpr StageTuning TUNED_F2X = {{8, 5, 5}, {0, 1, 0}, {0, 34, 0}, {1, 1, 1}};
// tune.py: end tables

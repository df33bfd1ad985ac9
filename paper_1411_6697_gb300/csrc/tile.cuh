// tile.cuh -- launch interface of the 2-D tile step (tile.cu).
#pragma once
#include <cuda_runtime.h>

#include "kernels.cuh"

namespace lbk {

// Blocks of a launch on this grid, and whether an FP32 grid steps with it (FP64 always does).
int tile_grid(int precision, int recovery, int nx, int ny, bool tne);
bool tile_takes_f32(int recovery, int nx, int ny);
cudaError_t launch_tile(int precision, int recovery, const void* K, const StepLaunch& a, cudaStream_t s);

} // namespace lbk

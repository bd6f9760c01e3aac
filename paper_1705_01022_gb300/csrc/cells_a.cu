// Coarse-cell device-step kernels (cells.cuh) for the cell shapes 4x8, 4x16, 8x4, 8x8.
#include "cells_lanes.cuh"

namespace oct {

template cudaError_t launch_cells_shape<4, 8>(const StepArgs &, bool, cudaStream_t);
template cudaError_t launch_cells_shape<4, 16>(const StepArgs &, bool, cudaStream_t);
template cudaError_t launch_cells_shape<8, 4>(const StepArgs &, bool, cudaStream_t);
template cudaError_t launch_cells_shape<8, 8>(const StepArgs &, bool, cudaStream_t);

}  // namespace oct

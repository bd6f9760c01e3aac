// Coarse-cell device-step kernels (cells.cuh) for the cell shapes 32x4, 32x8, 32x16.
#include "cells_lanes.cuh"

namespace oct {

template cudaError_t launch_cells_shape<32, 4>(const StepArgs &, bool, cudaStream_t);
template cudaError_t launch_cells_shape<32, 8>(const StepArgs &, bool, cudaStream_t);
template cudaError_t launch_cells_shape<32, 16>(const StepArgs &, bool, cudaStream_t);

}  // namespace oct

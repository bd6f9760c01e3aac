// Device step of DTrDT with thread cells coarser than 4x4 sites (cells.cuh):
// the shapes with a kernel and the dispatch of one device step to them.
#include "oct_internal.h"

namespace oct {

template <int CX, int CY>
cudaError_t launch_cells_shape(const StepArgs &a, bool any_random, cudaStream_t st);

bool cells_shape_supported(int cx, int cy) {
    switch (cx * 100 + cy) {
        case 804: case 408: case 808: case 1604: case 1608: case 816: case 1616:
        case 3204: case 3208: case 3216: case 416:
            return true;
        default:
            return false;
    }
}

cudaError_t launch_cells_step(const StepArgs &a, bool any_random, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    switch (a.cx * 100 + a.cy) {
        case 804: e = launch_cells_shape<8, 4>(a, any_random, st); break;
        case 408: e = launch_cells_shape<4, 8>(a, any_random, st); break;
        case 808: e = launch_cells_shape<8, 8>(a, any_random, st); break;
        case 1604: e = launch_cells_shape<16, 4>(a, any_random, st); break;
        case 1608: e = launch_cells_shape<16, 8>(a, any_random, st); break;
        case 816: e = launch_cells_shape<8, 16>(a, any_random, st); break;
        case 1616: e = launch_cells_shape<16, 16>(a, any_random, st); break;
        case 3204: e = launch_cells_shape<32, 4>(a, any_random, st); break;
        case 3208: e = launch_cells_shape<32, 8>(a, any_random, st); break;
        case 3216: e = launch_cells_shape<32, 16>(a, any_random, st); break;
        case 416: e = launch_cells_shape<4, 16>(a, any_random, st); break;
        default: return cudaErrorInvalidValue;
    }
    return e == cudaSuccess ? cudaGetLastError() : e;
}

}  // namespace oct

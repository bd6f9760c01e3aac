// Where a warp's sub-tile lies: the device layer of one MCS (Sec. 3, DTr).
//
// The origin (ox, oy) and the set permutation come from Philox(t, 0, 0,
// MCS<<28) once per MCS; device tile (tx, ty) has index T = ty*tiles_x + tx
// (the tile index of the random streams) and its sub-tile of set sigma =
// perm[k] starts at (ox + 2Bx tx + Bx (sigma&1), oy + 2By ty + By (sigma>>1))
// mod L.  A handle may hold only a row strip of the lattice (multi-GPU strip
// partition): its buffer then starts at global row row0, and it updates the
// strip_tiles_y device-tile rows whose first row (oy + 2By ty) mod L lies in
// [row0, row0 + 2By strip_tiles_y).  Work index w counts the sub-tiles the
// launch updates; y0 is returned in buffer rows.
#pragma once
#include <cstdint>

#include "oct_internal.h"
#include "philox.cuh"
#include "subtile.cuh"

namespace oct {

struct TilePlace {
    uint32_t T;       // device-tile index (random streams)
    uint32_t x0, y0;  // sub-tile origin: global column, buffer row
};

__host__ __device__ __forceinline__ uint32_t work_tiles(const StepArgs &a) {
    return a.tiles_x * (a.strip_tiles_y ? a.strip_tiles_y : a.tiles_y);
}

// Work index w in device step k of MCS t.  Sums of an offset and a place stay
// below 2L, so they are folded into [0, L) by one subtraction.
__device__ __forceinline__ TilePlace place_tile(const StepArgs &a, uint32_t w, uint32_t t, uint32_t k) {
    const uint32_t L = a.L;
    const uint4 M = philox4x32_10(t, 0u, 0u, kTagMcs << 28, a.k0, a.k1);
    const uint32_t ox = __umulhi(M.x, L), oy = __umulhi(M.y, L);
    const uint32_t sigma = static_cast<uint32_t>(perm_element(__umulhi(M.z, 24u), k));
    const uint32_t j = w / a.tiles_x, tx = w - j * a.tiles_x;
    uint32_t ty = j;
    if (a.strip_tiles_y) {
        // tile rows whose first row lies in the strip: ty = (j - q) mod tiles_y,
        // q = ((oy - row0) mod L) div 2By
        const uint32_t d = (oy + L - a.row0) % L;
        const uint32_t q = (d / (2u * a.By)) % a.tiles_y;
        ty = (j + a.tiles_y - q) % a.tiles_y;
    }
    TilePlace p;
    p.T = ty * a.tiles_x + tx;
    p.x0 = ox + a.Bx * (2u * tx + (sigma & 1u));
    if (p.x0 >= L) p.x0 -= L;
    p.y0 = oy + a.By * (2u * ty + (sigma >> 1));
    if (p.y0 >= L) p.y0 -= L;
    p.y0 += p.y0 >= a.row0 ? 0u - a.row0 : L - a.row0;  // buffer row
    return p;
}

}  // namespace oct

// Index arithmetic and size rules in plain C++, with host and device forms, so
// that both are tested on the CPU.
#pragma once

#include <stdint.h>

#include "awpm_fixed.h"

namespace awpm {

// Nonzeros handled by one warp per tile of the edge-parallel kernels; tiles
// start at multiples of kTile, so tile t owns word t of the column-start
// bitmap.
constexpr int kTile = 32;

// Largest nnz: the positions of all tiles' lanes, and of those of one tile past
// the last, stay in int32.
constexpr int32_t kMaxEntries = 0x7fffffff - 63;

// Position of a lane's entry in tile t.  A kernel that looks ahead asks for
// tiles past the last one: they get the positions of tile ntiles, which are at
// or past nnz and never wrap (the product t * kTile does, close to kMaxEntries).
AWPM_HD int32_t tile_pos(int32_t t, int32_t ntiles, int lane)
{
    return (t < ntiles ? t : ntiles) * kTile + lane;
}

}  // namespace awpm

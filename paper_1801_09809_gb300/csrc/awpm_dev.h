// Device helpers shared by the kernel files.
#pragma once

#include "awpm_internal.h"

namespace awpm {

#define FULL_MASK 0xffffffffu

constexpr int kThreads = 256;

__device__ __forceinline__ int64_t gtid()
{
    return blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
}

__device__ __forceinline__ int64_t gstride()
{
    return (int64_t)gridDim.x * blockDim.x;
}

__device__ __forceinline__ void raise_err(Ctl *ctl, unsigned bits)
{
    atomicOr(&ctl->err, bits);
}

// Column of the lane's nonzero: c0 (column of the tile's first nonzero) plus
// the columns starting after the tile's first nonzero and up to this lane.
// Exact when no column is empty (guaranteed once the matching validated).
__device__ __forceinline__ int32_t lane_column(int32_t c0, uint32_t mask, int lane)
{
    return c0 + __popc(mask & ((2u << lane) - 1u) & ~1u);
}

// The segment of a column that starts at `lane` covers the whole column when
// the column starts here and ends inside the tile: a later start bit, the
// end of the matrix, or a column starting the next tile.
__device__ __forceinline__ bool segment_complete(uint32_t mask, int lane, int32_t base,
                                                 int32_t nnz, const uint32_t *starts, int64_t t)
{
    const bool starts_here = (mask >> lane) & 1u;
    if (!starts_here)
        return false;
    const uint32_t later = lane == 31 ? 0u : (mask >> (lane + 1));
    return later != 0u || base + kTile >= nnz || (__ldg(starts + t + 1) & 1u);
}

}  // namespace awpm

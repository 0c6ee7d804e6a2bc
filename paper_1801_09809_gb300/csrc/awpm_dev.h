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

// Bounded retries for the lock-free arg-max updates (each failed
// compare-and-swap means another thread stored a strictly better record, so
// the loop ends long before this; the bound only turns a broken invariant
// into an error bit instead of a hang).
constexpr int kCasRetryCap = 1 << 20;

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_down_sync(FULL_MASK, v, o);
    return v;
}

// Sum v over the block and add it to *dst with one atomic.  All threads call.
__device__ __forceinline__ void block_add_u64(unsigned long long v, unsigned long long *dst)
{
    __shared__ unsigned long long sm[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    v = warp_sum_u64(v);
    __syncthreads();
    if (lane == 0)
        sm[wid] = v;
    __syncthreads();
    if (wid == 0) {
        v = (lane < (int)(blockDim.x >> 5)) ? sm[lane] : 0ull;
        v = warp_sum_u64(v);
        if (lane == 0 && v)
            atomicAdd(dst, v);
    }
}

__device__ __forceinline__ void warp_add_i32(int v, int32_t *dst)
{
    v = __reduce_add_sync(FULL_MASK, v);
    if ((threadIdx.x & 31) == 0 && v)
        atomicAdd(dst, v);
}

constexpr long long kKeyNone = (long long)0x8000000000000000ull;

// Integer ordered like the weight (-0 taken as +0; finite weights only).
__device__ __forceinline__ long long order_key(double x)
{
    long long b = __double_as_longlong(x);
    if (b == kKeyNone)
        b = 0;
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

// End of a pass (Algorithm 2): count it, stop when nothing was flipped or
// the pass cap is reached.  An incremental pass counted differences from the
// pass before.
__device__ __forceinline__ int control_step(Ctl *ctl, bool inc)
{
    if (ctl->err) {
        ctl->active = 0;
        return 0;
    }
    if (!ctl->active)
        return 0;
    const unsigned long long f = ctl->pass_flips;
    ctl->pass_flips = 0;
    if (inc) {
        if (ctl->iterations == 0) {
            ctl->cur_candidates = ctl->candidates;
            ctl->cur_found = ctl->found;
            ctl->cur_positive = ctl->positive;
        } else {
            ctl->candidates += ctl->cur_candidates += ctl->d_candidates;
            ctl->found += ctl->cur_found += ctl->d_found;
            ctl->positive += ctl->cur_positive += ctl->d_positive;
            ctl->d_candidates = ctl->d_found = ctl->d_positive = 0;
        }
        ctl->last_flips = f;
    }
    ctl->iterations += 1;
    ctl->cycles += f;
    if (f == 0) {
        ctl->converged = 1;
        ctl->active = 0;
    } else if (ctl->iterations >= ctl->max_passes) {
        ctl->active = 0;
    }
    return ctl->active;
}

}  // namespace awpm

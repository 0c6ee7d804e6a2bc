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
#ifndef AWPM_CAS_RETRY_CAP
#define AWPM_CAS_RETRY_CAP (1 << 20)
#endif
constexpr int kCasRetryCap = AWPM_CAS_RETRY_CAP;

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
    }
    ctl->last_flips = f;
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

// ---- gains as integers ----------------------------------------------------------
// FP64 instructions are scarce on this GPU, so gains are compared through
// their IEEE bit patterns.  For values in [+0, +inf] the order of the bit
// patterns read as signed 64-bit integers is the numeric order, and equal
// patterns are equal values; every stored or compared gain is either +0.0
// ("none") or a positive gain.

__device__ __forceinline__ long long gbits(double g)
{
    return __double_as_longlong(g);
}

// g > 0.0 exactly as IEEE compares it: sign clear, not zero, not NaN.
__device__ __forceinline__ bool gain_positive(double g)
{
    const long long b = gbits(g);
    return b > 0ll && b <= 0x7ff0000000000000ll;
}

// ---- lock-free arg-max records ----------------------------------------------

// (g, p) beats (cg, cp): larger gain, then lower position (gains >= +0).
__device__ __forceinline__ bool rec_better(double g, int32_t p, double cg, int32_t cp)
{
    const long long a = gbits(g), b = gbits(cg);
    return a > b || (a == b && p < cp);
}

// A 16-byte record read in one piece, from L2, as other threads' exchanges leave
// it: two reads of eight bytes, or a vector load, which promises no more, may
// see halves of two records.
template <typename T>
__device__ __forceinline__ T ld_record(const T *addr)
{
    static_assert(sizeof(T) == 16 && alignof(T) == 16, "one 128-bit access");
    union {
        unsigned long long h[2];
        T rec;
    } v;
    asm volatile("{\n\t"
                 ".reg .b128 t;\n\t"
                 "ld.relaxed.gpu.global.b128 t, [%2];\n\t"
                 "mov.b128 {%0, %1}, t;\n\t"
                 "}"
                 : "=l"(v.h[0]), "=l"(v.h[1])
                 : "l"(addr)
                 : "memory");
    return v.rec;
}

// Maximum of (g, lowest p) into a Step-C record.
__device__ __forceinline__ void rec_combine(Rec *addr, Rec mine, Ctl *ctl)
{
    Rec cur = *addr;
    for (int it = 0; it < kCasRetryCap; ++it) {
        if (!rec_better(mine.g, mine.p, cur.g, cur.p))
            return;
        Rec old = atomicCAS(addr, cur, mine);
        if (__double_as_longlong(old.g) == __double_as_longlong(cur.g) && old.p == cur.p &&
            old.q == cur.q)
            return;
        cur = old;
    }
    raise_err(ctl, kErrTimeout);
}

// (g, j) beats (cg, cj): larger gain, then lower root (gains >= +0).
__device__ __forceinline__ bool sel_better(double g, int32_t j, double cg, int32_t cj)
{
    const long long a = gbits(g), b = gbits(cg);
    return a > b || (a == b && j < cj);
}

// Maximum of (g, lowest root j) into a Step-D selection (a record of another
// epoch counts as empty).
__device__ __forceinline__ void sel_combine(Sel *addr, Sel mine, Ctl *ctl)
{
    Sel cur = ld_record(addr);
    for (int it = 0; it < kCasRetryCap; ++it) {
        if (cur.epoch == mine.epoch && !sel_better(mine.g, mine.j, cur.g, cur.j))
            return;
        Sel old = atomicCAS(addr, cur, mine);
        if (__double_as_longlong(old.g) == __double_as_longlong(cur.g) && old.j == cur.j &&
            old.epoch == cur.epoch)
            return;
        cur = old;
    }
    raise_err(ctl, kErrTimeout);
}

// Bitmap words a warp takes at a time when `words` of them are spread over
// `nwarps` warps: 32 (one per lane) when there are enough, fewer, down to 1,
// when that keeps more warps busy (the winners' accesses are scattered, so
// the time goes with the winners that one warp takes in turn: the flips of
// a solve of the 27-point stencil of 96^3 went from 2.5 to 0.85 ms in all).
__device__ __forceinline__ int words_per_warp(int64_t words, int64_t nwarps)
{
    int k = 1;
    while (k < 32 && k * nwarps < words)
        k *= 2;
    return k;
}

// The winners (set bits) of the bitmap words [x0, x0 + count), count <= 32,
// 32 winners at a time with every lane busy: the words' bit counts are
// scanned across the warp, and in each round lane l takes the winner of rank
// round * 32 + l (found by a binary search over the scan and the word's
// rank-th set bit).  Calls f(j) on every lane each round, j = -1 for lanes
// past the last winner.  Called by the whole warp; `clear` zeroes the words
// as they are read.
template <typename F>
__device__ __forceinline__ void for_winners(uint32_t *winbits, int64_t x0, int count,
                                            int64_t words, int lane, bool clear, F f)
{
    const uint32_t mine = lane < count && x0 + lane < words ? winbits[x0 + lane] : 0u;
    if (clear && mine)
        winbits[x0 + lane] = 0u;
    __syncwarp();  // f may set a bit of a cleared word again
    const int cnt = __popc(mine);
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL_MASK, incl, o);
        if (lane >= o)
            incl += y;
    }
    const int excl = incl - cnt;
    const int total = __shfl_sync(FULL_MASK, incl, 31);
    for (int base = 0; base < total; base += 32) {
        const int want = base + lane;
        // the last word whose first rank is <= want
        int src = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1) {
            const int e = __shfl_sync(FULL_MASK, excl, src + step);
            if (e <= want)
                src += step;
        }
        const int first = __shfl_sync(FULL_MASK, excl, src);
        const uint32_t word = __shfl_sync(FULL_MASK, mine, src);
        int32_t j = -1;
        if (want < total) {
            const int bit = (int)__fns(word, 0u, want - first + 1);
            j = (int32_t)((x0 + src) * 32 + bit);
        }
        f(j);
    }
}

// Barrier of the cluster's threads, ordering their memory accesses.
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
                 "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

}  // namespace awpm

// Maximum cardinality matching with the heavy-weight tie-break (Section 5.2):
// kernels (sm_103a).
//
// Phases of breadth-first augmenting-path searches from every free column.
// Per level, every frontier column offers its rows not reached yet (through
// unmatched edges); a row goes to the offer with the heaviest edge, then the
// lowest column (order key and column in one 128-bit record).  A free row so
// reached ends a path of its tree (the tree keeps the heaviest last edge, then
// the lowest row, and stops growing); a matched row brings its matched column
// into the next frontier.  The trees are vertex-disjoint, so all paths found
// in a phase are augmented at once.  A phase that augments nothing ends the
// search: the matching is maximum.
//
// A level is three steps (offer, join, advance), each over what the level
// touches only: the listed 32-entry tiles holding an entry of a frontier
// column, the rows offered something, and the columns matched to them.  In the
// graph form one cluster of blocks runs levels of few tiles one after another
// (a level of the grid is three launches, whatever its size).
//
// Bound by the dependent accesses of a level (tile, row, record, mate, column),
// hundreds of levels of which most are small, not by bytes.  Measured: R-MAT
// graph of scale 22 from a greedy matching, 386 levels, 25 -> 19.5 ms; a
// random matrix of 250,000 columns, 54 levels, 2.15 -> 1.76 ms.  Levels in one
// cluster up to 512, 2,048, 4,096, 8,192 and 16,384 tiles: 27.5, 27.5, 27.7,
// 28.5 and 29.8 ms for the whole chain of greedy, matching and improvement.
#include "awpm.h"
#include "awpm_dev.h"
#include "awpm_internal.h"

namespace awpm {

namespace {

// Small levels run in one cluster of kSmallBlocks blocks, while they have at
// most kSmallTiles tiles and 32 times as many columns.
constexpr int kSmallThreads = 1024;
constexpr int kSmallBlocks = 8;
#ifndef AWPM_MC_SMALL
#define AWPM_MC_SMALL 2048
#endif
constexpr int32_t kSmallTiles = AWPM_MC_SMALL;

// Clear the per-solve state; mr = -1; every offer record empty; no row
// reached, no column in the frontier, no tile listed.
__global__ void k_mc_reset(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (gtid() == 0) {
        Ctl *c = w.ctl;
        c->err = 0u;
        c->active = 1;
        c->iterations = 0;
        c->converged = 0;
        c->live = 0;
        c->levels = 0ull;
        c->pass_flips = 0ull;
        c->cycles = 0ull;
        c->front_next = 0;
        c->level_tiles = 0;
        c->front_n = 0;
        c->level_done = 0u;
        c->touched = 0;
    }
    for (int64_t x = gtid(); x < w.n; x += gstride()) {
        w.mr[x] = -1;
        w.mroff[x] = Off{kKeyNone, 0x7fffffff, 0};
    }
    const int64_t words = ((int64_t)w.nnz + 31) / 32 + 1;
    for (int64_t x = gtid(); x < words; x += gstride())
        w.starts[x] = 0u;
    for (int64_t x = gtid(); x < w.n / 32 + 2; x += gstride())
        w.mfront[x] = 0u;
    for (int64_t x = gtid(); x < w.ntiles / 32 + 1; x += gstride())
        w.mtmark[x] = 0u;
}

// A column without entries is no error for the maximum matching (it stays
// unmatched): drop that report of the column-pointer check.
__global__ void k_mc_allow_empty(const Work *__restrict__ W)
{
    Ctl *c = W->ctl;
    c->nonempty = (c->err & kErrNotPerfect) ? 0 : 1;
    atomicAnd(&c->err, ~kErrNotPerfect);
}

// The starting matching: row of every column or -1, each row once, every
// pair a stored entry (binary search in the sorted column); its size.
__global__ void k_mc_load(const Work *__restrict__ W)
{
    const Work &w = *W;
    unsigned long long have = 0;
    if (!w.ctl->err) {
        for (int64_t j = gtid(); j < w.n; j += gstride()) {
            const int32_t r = w.mmate[j];
            w.mc[j] = r < 0 ? -1 : r;
            if (r < 0)
                continue;
            if (r >= w.n || atomicCAS(&w.mr[r], -1, (int32_t)j) != -1) {
                raise_err(w.ctl, kErrNotPerfect);
                continue;
            }
            int32_t lo = w.colptr[j], len = w.colptr[j + 1] - lo;
            while (len > 0) {
                const int32_t half = len >> 1;
                if (w.rowidx[lo + half] < r) {
                    lo += half + 1;
                    len -= half + 1;
                } else {
                    len = half;
                }
            }
            if (lo >= w.colptr[j + 1] || w.rowidx[lo] != r)
                raise_err(w.ctl, kErrNotPerfect);
            ++have;
        }
    }
    block_add_u64(have, &w.ctl->cycles);
}

// Column of every entry (a warp per column), for the levels' offers when a
// column is empty.
__global__ void k_mc_colof(const Work *__restrict__ W)
{
    const Work &w = *W;
    if ((w.ctl->err & kErrInvalid) || w.ctl->nonempty)
        return;
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = gstride() >> 5;
    for (int64_t j = gtid() >> 5; j < w.n; j += nwarps)
        for (int32_t p = w.colptr[j] + lane; p < w.colptr[j + 1]; p += 32)
            w.mcolof[p] = (int32_t)j;
}

// Append frontier columns (lane l of the warp: column c[u], -1 for none, u <
// kU) to the frontier list and the tiles that their entries span to the tile
// list of the next level; one 64-bit atomic per call reserves both.  A tile
// shared by several columns is listed once: the first to set its bit lists it
// (a tile inside one column needs no bit).  So the list has room for every
// tile once; an append past that is refused with an internal error.
// Called by a whole warp.
template <int kU>
__device__ __forceinline__ void mc_append(const Work &w, const int32_t (&c)[kU], int lane)
{
    int32_t first[kU], count[kU];  // tiles first .. first + count - 1
    int32_t tiles = 0, cols = 0;
#pragma unroll
    for (int u = 0; u < kU; ++u) {
        first[u] = count[u] = 0;
        if (c[u] < 0)
            continue;
        ++cols;
        const int32_t s = __ldg(w.colptr + c[u]), e = __ldg(w.colptr + c[u] + 1);
        if (e <= s)
            continue;
        int32_t t0 = s >> 5, t1 = (e - 1) >> 5;
        auto taken = [&](int32_t t) {
            const uint32_t bit = 1u << (t & 31);
            return (atomicOr(w.mtmark + (t >> 5), bit) & bit) != 0u;
        };
        const bool last_whole = e - (t1 << 5) >= 32, first_whole = (s & 31) == 0;
        if (t0 == t1) {
            if (!(first_whole && last_whole) && taken(t0))
                ++t0;
        } else {
            if (!first_whole && taken(t0))
                ++t0;
            if (!last_whole && taken(t1))
                --t1;
        }
        first[u] = t0;
        count[u] = t1 - t0 + 1;
        tiles += count[u];
    }
    int32_t it = tiles, ic = cols;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t a = __shfl_up_sync(FULL_MASK, it, o), b = __shfl_up_sync(FULL_MASK, ic, o);
        if (lane >= o) {
            it += a;
            ic += b;
        }
    }
    const int32_t all_t = __shfl_sync(FULL_MASK, it, 31), all_c = __shfl_sync(FULL_MASK, ic, 31);
    if (all_c == 0)
        return;
    unsigned long long base = 0;
    if (lane == 0)
        base = atomicAdd(reinterpret_cast<unsigned long long *>(&w.ctl->level_tiles),
                         ((unsigned long long)(uint32_t)all_c << 32) | (uint32_t)all_t);
    base = __shfl_sync(FULL_MASK, base, 0);
    int64_t at = (int64_t)(uint32_t)base + it - tiles;
    int64_t ac = (int64_t)(base >> 32) + ic - cols;
    if ((int64_t)(uint32_t)base + all_t > w.mtiles_cap || (int64_t)(base >> 32) + all_c > w.n) {
        if (lane == 0)
            raise_err(w.ctl, kErrInternal);
        return;
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
        if (c[u] >= 0)
            w.mfl[ac++] = c[u];
        // a long column's tiles: the warp together
        unsigned longm = __ballot_sync(FULL_MASK, count[u] > 32);
        while (longm) {
            const int src = __ffs(longm) - 1;
            longm &= longm - 1;
            const int32_t f = __shfl_sync(FULL_MASK, first[u], src);
            const int32_t k = __shfl_sync(FULL_MASK, count[u], src);
            const int64_t a = __shfl_sync(FULL_MASK, at, src);
            for (int32_t y = lane; y < k; y += 32)
                w.mtiles[a + y] = f + y;
        }
        if (count[u] <= 32)
            for (int32_t y = 0; y < count[u]; ++y)
                w.mtiles[at + y] = first[u] + y;
        at += count[u];
    }
}

// The end of a step that made a frontier: its size, for the loops, and the
// counters for the next level.  (level_tiles is emptied by the join.)
__device__ __forceinline__ void mc_frontier_made(Ctl *c)
{
    c->front_n = c->front_next;
    c->live = c->front_next;
    c->front_next = 0;
    c->touched = 0;
}

// True in thread 0 of the block that finishes last (its count of finished
// blocks orders it after every other block's writes).
__device__ __forceinline__ bool mc_last_block(Ctl *c)
{
    __syncthreads();
    if (threadIdx.x != 0)
        return false;
    __threadfence();
    if (atomicAdd(&c->level_done, 1u) != gridDim.x - 1)
        return false;
    __threadfence();
    c->level_done = 0u;
    return true;
}

// A phase: every free column roots a tree (its end record cleared) and forms
// the frontier; no row is reached.  (A row's offer record was cleared by the
// join that reached it.  End records are read only for the roots of the
// running phase.)
__device__ __forceinline__ void mc_phase(const Work &w)
{
    if (!w.ctl->err) {
        // four words at a time: with one, the list's counter held the phase up
        // where most columns are free (of 4 M: about 120 us, now 52)
        constexpr int kU = 4;
        const int lane = threadIdx.x & 31;
        const int64_t words = (int64_t)w.n / 32 + 1, nwarps = gstride() >> 5;
        for (int64_t x0 = gtid() >> 5; x0 < words; x0 += kU * nwarps) {
            int32_t c[kU];
            unsigned any = 0u;
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int64_t j = (x0 + u * nwarps) * 32 + lane;
                c[u] = j < w.n && w.mc[j] < 0 ? (int32_t)j : -1;
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int64_t x = x0 + u * nwarps;
                const unsigned bits = __ballot_sync(FULL_MASK, c[u] >= 0);
                any |= bits;
                if (lane == 0 && x < words) {
                    w.mfront[x] = bits;
                    w.mreach[x] = 0u;
                }
                if (c[u] >= 0) {
                    w.mroot[c[u]] = c[u];
                    w.mtend[c[u]] = Off{kKeyNone, 0x7fffffff, 0};
                }
            }
            if (any)
                mc_append<kU>(w, c, lane);
        }
    }
    if (gtid() == 0)
        w.ctl->phase_levels = 0;
}

__global__ void k_mc_phase(const Work *__restrict__ W)
{
    mc_phase(*W);
    if (mc_last_block(W->ctl))
        mc_frontier_made(W->ctl);
}

// (key, who) beats the record cur: heavier key, then lower index.
__device__ __forceinline__ bool off_better(long long key, int32_t who, const Off &cur)
{
    return key > cur.key || (key == cur.key && who < cur.who);
}

// Fold (key, who) into the record at addr, last seen as cur (128-bit
// compare-and-swap; a failed exchange means another thread stored a better
// record, so the loop is short; its bound only turns a broken invariant into
// an error bit).  True for the exchange that replaced the empty record.
__device__ __forceinline__ bool off_combine(Off *addr, Off cur, long long key, int32_t who, Ctl *ctl)
{
    const Off mine{key, who, 0};
    for (int k = 0; k < kCasRetryCap; ++k) {
        if (!off_better(key, who, cur))
            return false;
        const Off old = atomicCAS(addr, cur, mine);
        if (old.key == cur.key && old.who == cur.who && old.pad == cur.pad)
            return old.who == 0x7fffffff;
        cur = old;
    }
    raise_err(ctl, kErrTimeout);
    return false;
}

// Level, step 1: per unreached row the best offer of the level: the heaviest
// edge from a frontier column, then the lowest column.  A warp takes four
// listed tiles per round, their reads side by side (tile, then its row
// indices and words, then the rows' and columns' bits, then weights and
// records), the next round's tile numbers read ahead.  The rows offered
// something for the first time are collected per warp and listed 64 or more
// at a time: with an atomic per tile the list's counter alone held the level
// up.
constexpr int kRowBuf = 64 + 4 * 32;

__device__ __forceinline__ void mc_offer(const Work &w, int32_t *buf)
{
    constexpr int kU = 4;
    const int lane = threadIdx.x & 31;
    const unsigned lanes_below = (1u << lane) - 1u;
    const int64_t nwarps = gstride() >> 5;
    const bool exact = w.ctl->nonempty != 0;
    const int32_t listed = w.ctl->level_tiles;
    const int32_t nnz = w.nnz;
    int have = 0;  // rows in buf (warp-uniform)
    auto put = [&]() {
        __syncwarp();
        int32_t base = 0;
        if (lane == 0)
            base = atomicAdd(&w.ctl->touched, have);
        base = __shfl_sync(FULL_MASK, base, 0);
        for (int x = lane; x < have; x += 32)
            w.mtouch[base + x] = buf[x];
        __syncwarp();
        have = 0;
    };
    int32_t nt[kU];
    const int64_t x00 = gtid() >> 5;
#pragma unroll
    for (int u = 0; u < kU; ++u)
        nt[u] = x00 + u * nwarps < listed ? w.mtiles[x00 + u * nwarps] : -1;
    for (int64_t x0 = x00; x0 < listed; x0 += kU * nwarps) {
        int32_t t[kU], c0[kU], r[kU], c[kU];
        uint32_t mask[kU];
        bool go[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u)
            t[u] = nt[u];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int64_t x = x0 + (kU + u) * nwarps;
            nt[u] = x < listed ? w.mtiles[x] : -1;
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int32_t p = t[u] * kTile + lane;
            const bool valid = t[u] >= 0 && p < nnz;
            c0[u] = t[u] >= 0 ? __ldg(w.tile_col + t[u]) : 0;
            mask[u] = t[u] >= 0 ? __ldg(w.starts + t[u]) : 1u;
            r[u] = valid ? __ldg(w.rowidx + p) : -1;
            c[u] = exact ? lane_column(c0[u], mask[u], lane)
                         : valid ? __ldg(w.mcolof + p) : 0;
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            go[u] = r[u] >= 0;
            uint32_t front = 0u, reached = 0u;
            if (go[u]) {
                front = w.mfront[c[u] >> 5];
                reached = w.mreach[r[u] >> 5];
            }
            // (a frontier column's own matched row was reached before it)
            go[u] = go[u] && ((front >> (c[u] & 31)) & 1u) && !((reached >> (r[u] & 31)) & 1u);
        }
        long long key[kU];
        Off cur[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            key[u] = 0;
            cur[u] = Off{0, 0, 0};
            if (go[u]) {
                key[u] = order_key(__ldg(w.w + (int64_t)t[u] * kTile + lane));
                cur[u] = ld_record(w.mroff + r[u]);
            }
            // the tile leaves the list (its next listing is by the advance)
            if (lane == 0 && t[u] >= 0)
                atomicAnd(w.mtmark + (t[u] >> 5), ~(1u << (t[u] & 31)));
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            bool first = false;
            if (go[u])
                first = off_combine(w.mroff + r[u], cur[u], key[u], c[u], w.ctl);
            const unsigned m = __ballot_sync(FULL_MASK, first);
            if (first)
                buf[have + __popc(m & lanes_below)] = r[u];
            have += __popc(m);
        }
        if (have >= 64)
            put();
    }
    if (have > 0)
        put();
}

// Level, step 2: every row offered something at this level joins the tree of
// its best offer's column.  A free row is a candidate end of the tree: the
// tree keeps the heaviest last edge, then the lowest row.  A matched row's
// column takes its place in the list, for step 3.  The level's frontier and
// tile list are emptied.
__device__ __forceinline__ void mc_join(const Work &w)
{
    const int64_t first = gtid(), step = gstride();
    if (first == 0)
        w.ctl->level_tiles = 0;  // (read by the offer only)
    const int32_t front = w.ctl->front_n;
    for (int64_t x = first; x < front; x += step)
        w.mfront[w.mfl[x] >> 5] = 0u;  // (only this frontier's bits are set)
    const int32_t touched = w.ctl->touched;
    for (int64_t x = first; x < touched; x += step) {
        const int32_t r = w.mtouch[x];
        const Off o = ld_record(w.mroff + r);
        const int32_t c = o.who;
        const int32_t c2 = w.mr[r];
        const int32_t t_root = w.mroot[c];
        w.mroff[r] = Off{kKeyNone, 0x7fffffff, 0};
        w.mrpar[r] = c;
        atomicOr(w.mreach + (r >> 5), 1u << (r & 31));
        w.mtouch[x] = c2;
        if (c2 < 0)
            off_combine(w.mtend + t_root, ld_record(w.mtend + t_root), o.key, r, w.ctl);
        else
            w.mroot[c2] = t_root;
    }
}

// Level, step 3: the next frontier: the columns found, without the trees that
// have an end.
__device__ __forceinline__ void mc_advance(const Work &w)
{
    constexpr int kU = 4;
    const int lane = threadIdx.x & 31;
    const int64_t step = gstride();
    const int32_t touched = w.ctl->touched;
    for (int64_t x0 = gtid() - lane; x0 < touched; x0 += kU * step) {
        int32_t c[kU], root[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int64_t x = x0 + u * step + lane;
            c[u] = x < touched ? w.mtouch[x] : -1;
        }
#pragma unroll
        for (int u = 0; u < kU; ++u)
            root[u] = c[u] >= 0 ? w.mroot[c[u]] : -1;
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            if (root[u] >= 0 && ld_record(w.mtend + root[u]).who != 0x7fffffff)
                c[u] = -1;
            if (c[u] >= 0)
                atomicOr(w.mfront + (c[u] >> 5), 1u << (c[u] & 31));
        }
        mc_append<kU>(w, c, lane);
    }
}

__global__ void __launch_bounds__(kThreads) k_mc_offer(const Work *__restrict__ W)
{
    __shared__ int32_t s_buf[kThreads / 32][kRowBuf];
    if (!W->ctl->err)
        mc_offer(*W, s_buf[threadIdx.x >> 5]);
}

__global__ void k_mc_join(const Work *__restrict__ W)
{
    if (!W->ctl->err)
        mc_join(*W);
}

__global__ void k_mc_advance(const Work *__restrict__ W)
{
    if (!W->ctl->err)
        mc_advance(*W);
    if (mc_last_block(W->ctl))
        mc_frontier_made(W->ctl);
}

// Count the level that the frontier will run; cap the levels of a phase (every
// level adds a row to the search forest, so n + 1 levels mean a broken
// invariant).  False when there is nothing to run.
__device__ __forceinline__ bool mc_count_level(const Work &w)
{
    Ctl *c = w.ctl;
    if (c->live <= 0)
        return false;
    c->levels += 1;
    if (++c->phase_levels > w.n + 1)
        raise_err(c, kErrTimeout);
    return *(volatile unsigned *)&c->err == 0u;
}

// The two together, with their reads side by side: in a level of one cluster
// everyone waits for them (2 % of a small problem's search).
__device__ __forceinline__ bool mc_level_made(const Work &w)
{
    Ctl *c = w.ctl;
    const int32_t next = c->front_next, done = c->phase_levels;
    const unsigned long long levels = c->levels;
    const unsigned err = *(volatile unsigned *)&c->err;
    c->front_n = next;
    c->live = next;
    c->front_next = 0;
    c->touched = 0;
    if (next <= 0)
        return false;
    c->levels = levels + 1;
    c->phase_levels = done + 1;
    if (done >= w.n + 1) {
        raise_err(c, kErrTimeout);
        return false;
    }
    return err == 0u;
}

// Whether the next level, if there is one, is k_mc_small's, into Ctl::active:
// decided by one thread, before the threads that act on it start, so that all
// of them agree (an error bit may be set while they are reading).
__device__ __forceinline__ void mc_next_small(const Work &w, bool go)
{
    // (a frontier of many more columns than tiles is of empty ones)
    w.ctl->active =
        go && w.ctl->level_tiles <= kSmallTiles && w.ctl->front_n / 32 <= kSmallTiles ? 1 : 0;
}

// Graph form of step 3: the block that finishes last also sets the level
// loop's condition.
__global__ void k_mc_advance_graph(const Work *__restrict__ W, cudaGraphConditionalHandle h)
{
    const Work &w = *W;
    // (after k_mc_small's levels ended the phase there is nothing left)
    const bool run = w.ctl->front_n > 0;
    if (run && !w.ctl->err)
        mc_advance(w);
    if (mc_last_block(w.ctl)) {
        const bool go = run && mc_level_made(w);
        mc_next_small(w, go);
        cudaGraphSetConditional(h, go ? 1u : 0u);
    }
}

// Graph form, before a level's grid-wide steps: while the frontier is small,
// one cluster of blocks runs its levels, with cluster barriers between the
// steps.
__global__ void __cluster_dims__(kSmallBlocks, 1, 1) __launch_bounds__(kSmallThreads)
    k_mc_small(const Work *__restrict__ W)
{
    __shared__ int32_t s_buf[kSmallThreads / 32][kRowBuf];
    const Work &w = *W;
    Ctl *c = w.ctl;
    while (*(volatile int32_t *)&c->active) {
        mc_offer(w, s_buf[threadIdx.x >> 5]);
        cluster_sync();
        mc_join(w);
        cluster_sync();
        mc_advance(w);
        cluster_sync();
        if (gtid() == 0)
            mc_next_small(w, mc_level_made(w));
        cluster_sync();
    }
}

// Graph form of the level loop's condition before a phase's first level.
__global__ void k_mc_cond_level(const Work *__restrict__ W, cudaGraphConditionalHandle h)
{
    const bool go = mc_count_level(*W);
    mc_next_small(*W, go);
    cudaGraphSetConditional(h, go ? 1u : 0u);
}

// The end of a phase: count it and the paths it augmented; continue while it
// augmented something.
__device__ __forceinline__ bool mc_count_phase(const Work &w)
{
    Ctl *c = w.ctl;
    const unsigned long long aug = c->pass_flips;
    c->pass_flips = 0ull;
    c->cycles += aug;
    c->iterations += 1;
    return aug > 0 && *(volatile unsigned *)&c->err == 0u && c->iterations <= w.n;
}

__global__ void k_mc_cond_phase(const Work *__restrict__ W, cudaGraphConditionalHandle h)
{
    cudaGraphSetConditional(h, mc_count_phase(*W) ? 1u : 0u);
}

// Every tree with an end flips its path; their number into Ctl::pass_flips.
__device__ __forceinline__ void mc_augment(const Work &w)
{
    unsigned long long aug = 0;
    if (!w.ctl->err) {
        for (int64_t t = gtid(); t < w.n; t += gstride()) {
            if (w.mc[t] >= 0 || w.mtend[t].who == 0x7fffffff)
                continue;
            int32_t r = w.mtend[t].who;
            for (int32_t guard = 0; guard <= w.n; ++guard) {
                const int32_t c = w.mrpar[r];
                if (c < 0) {  // a broken tree: report instead of walking on
                    raise_err(w.ctl, kErrInternal);
                    break;
                }
                const int32_t old = w.mc[c];
                w.mc[c] = r;
                w.mr[r] = c;
                if (old < 0)
                    break;
                r = old;
            }
            ++aug;
        }
    }
    block_add_u64(aug, &w.ctl->pass_flips);
}

__global__ void k_mc_augment(const Work *__restrict__ W)
{
    mc_augment(*W);
}

// The whole search of a small problem in one cluster: the phases and their
// levels with cluster barriers, no launch per step (a phase of the graph is at
// least eight launches).
__global__ void __cluster_dims__(kSmallBlocks, 1, 1) __launch_bounds__(kSmallThreads)
    k_mc_cluster(const Work *__restrict__ W)
{
    __shared__ int32_t s_buf[kSmallThreads / 32][kRowBuf];
    const Work &w = *W;
    Ctl *c = w.ctl;
    for (;;) {
        mc_phase(w);
        cluster_sync();
        // (one thread decides whether a level runs, between two barriers:
        // threads that read the error bits for themselves could disagree, and
        // wait at different barriers)
        if (gtid() == 0)
            c->active = mc_level_made(w) ? 1 : 0;
        cluster_sync();
        while (*(volatile int32_t *)&c->active) {
            mc_offer(w, s_buf[threadIdx.x >> 5]);
            cluster_sync();
            mc_join(w);
            cluster_sync();
            mc_advance(w);
            cluster_sync();
            if (gtid() == 0)
                c->active = mc_level_made(w) ? 1 : 0;
            cluster_sync();
        }
        mc_augment(w);
        cluster_sync();
        if (gtid() == 0)
            c->active = mc_count_phase(w) ? 1 : 0;
        cluster_sync();
        if (!*(volatile int32_t *)&c->active)
            return;
    }
}

// The result back into the caller's matching array.
__global__ void k_mc_store(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (w.ctl->err)
        return;
    for (int64_t j = gtid(); j < w.n; j += gstride())
        w.mmate[j] = w.mc[j];
}

unsigned wave(const Shape &sh, int blocks)
{
    return (unsigned)(sh.num_sms * blocks);
}

}  // namespace

void launch_mcm_load(const Work *d, const Shape &sh, Sink &k)
{
    void *a[] = {(void *)&d};
    k.launch((const void *)k_mc_reset, wave(sh, 4), kThreads, a);
    launch_check_colptr(d, sh, k);
    k.launch((const void *)k_mc_allow_empty, 1, 1, a);
    launch_mark_starts(d, sh, k);
    launch_check_entries(d, sh, k);
    k.launch((const void *)k_mc_load, wave(sh, 16), kThreads, a);
    k.launch((const void *)k_mc_colof, wave(sh, 16), kThreads, a);
}

void launch_mcm_phase(const Work *d, const Shape &sh, Sink &k)
{
    void *a[] = {(void *)&d};
    k.launch((const void *)k_mc_phase, wave(sh, 8), kThreads, a);
}

// One wave of blocks: a level's work follows its frontier, and a small
// frontier should not pay for launching idle blocks.
void launch_mcm_level(const Work *d, const Shape &sh, Sink &k)
{
    void *a[] = {(void *)&d};
    k.launch((const void *)k_mc_offer, wave(sh, 4), kThreads, a);
    k.launch((const void *)k_mc_join, wave(sh, 8), kThreads, a);
    k.launch((const void *)k_mc_advance, wave(sh, 4), kThreads, a);
}

void launch_mcm_level_graph(const Work *d, const Shape &sh, cudaGraphConditionalHandle h,
                            Sink &k)
{
    void *a[] = {(void *)&d};
    void *ah[] = {(void *)&d, (void *)&h};
    k.launch((const void *)k_mc_small, kSmallBlocks, kSmallThreads, a);
    k.launch((const void *)k_mc_offer, wave(sh, 4), kThreads, a);
    k.launch((const void *)k_mc_join, wave(sh, 8), kThreads, a);
    k.launch((const void *)k_mc_advance_graph, wave(sh, 4), kThreads, ah);
}

void launch_mcm_cluster(const Work *d, const Shape &, Sink &k)
{
    void *a[] = {(void *)&d};
    k.launch((const void *)k_mc_cluster, kSmallBlocks, kSmallThreads, a);
}

void launch_mcm_augment(const Work *d, const Shape &sh, Sink &k)
{
    void *a[] = {(void *)&d};
    k.launch((const void *)k_mc_augment, wave(sh, 4), kThreads, a);
}

void launch_mcm_cond_level(const Work *d, const Shape &, cudaGraphConditionalHandle h, Sink &k)
{
    void *ah[] = {(void *)&d, (void *)&h};
    k.launch((const void *)k_mc_cond_level, 1, 1, ah);
}

void launch_mcm_cond_phase(const Work *d, const Shape &, cudaGraphConditionalHandle h, Sink &k)
{
    void *ah[] = {(void *)&d, (void *)&h};
    k.launch((const void *)k_mc_cond_phase, 1, 1, ah);
}

void launch_mcm_store(const Work *d, const Shape &sh, Sink &k)
{
    void *a[] = {(void *)&d};
    k.launch((const void *)k_mc_store, wave(sh, 4), kThreads, a);
}

}  // namespace awpm

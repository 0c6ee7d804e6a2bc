// Heavy-weight greedy maximal matching (Section 5.1): kernels (sm_103a).
//
// The matching that greedy builds when it takes the stored entries from
// heaviest to lightest (equal weights: lower row, then lower column) and
// keeps each entry whose row and column are both free.  Computed in rounds:
// every free column names its first free entry in that order (largest
// weight, then lowest row), every free row names its first free entry
// (largest weight, then lowest column), and the entries named by both ends
// are matched.
//
// A round is two kernels.  The first passes over the entries once and keeps,
// per free row and per free column, the best entry as one 128-bit record
// (order key of the weight, index, round), so that equal weights are settled
// in the same pass; a record of another round counts as empty, so none is
// cleared, and a matched row's record says so, so that the row's state and
// its best entry are one read.  The second matches the columns.  (With 64-bit
// maxima first, the lowest indices among their holders in a second pass and a
// third kernel clearing the rows, a round read the entries and the rows'
// records twice: 1.73 ms for a random matrix of 1 M columns, now 1.36 ms.)
//
// Bound by the rate of the 128-bit compare-and-swaps in L2: with four tiles'
// swaps in flight at once the time did not change (1.39 ms); without any on
// the rows, by proposals of the columns' best in two more kernels per round,
// it was 1.49 ms.
#include "awpm.h"
#include "awpm_dev.h"
#include "awpm_internal.h"

namespace awpm {

namespace {

// Off::pad of a row record once the row is matched.
constexpr int32_t kMatched = -1;

// Tiles of a group: a warp takes one group at a time, and a byte says which
// of its tiles are dead (no free entry left; none ever comes back).
constexpr int kGroup = 8;

// Fold (key, who) of this round into the record at addr, last seen as cur:
// the larger key, then the lower index (128-bit compare-and-swap; a failed
// exchange means another thread stored a better record, so the loop is short;
// its bound only turns a broken invariant into an error bit).
__device__ __forceinline__ void rec_fold(Off *addr, Off cur, long long key, int32_t who,
                                         int32_t round, Ctl *ctl)
{
    const Off mine{key, who, round};
    for (int k = 0; k < kCasRetryCap; ++k) {
        if (cur.pad == round && (cur.key > key || (cur.key == key && cur.who <= who)))
            return;
        const Off old = atomicCAS(addr, cur, mine);
        if (old.key == cur.key && old.who == cur.who && old.pad == cur.pad)
            return;
        cur = old;
    }
    raise_err(ctl, kErrTimeout);
}

// Clear the matching, the records and the control block.
__global__ void k_gm_reset(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (gtid() == 0) {
        Ctl *c = w.ctl;
        c->err = 0u;
        c->active = 1;
        c->iterations = 0;
        c->converged = 0;
        c->live = 0;
        c->max_passes = w.max_passes;
        c->pass_flips = 0ull;
        c->flip_done = 0u;
        c->cycles = 0ull;
        c->candidates = 0ull;
        c->found = 0ull;
        c->positive = 0ull;
        c->weight_in = 0.0;
        c->weight_out = 0.0;
    }
    for (int64_t x = gtid(); x < w.n; x += gstride()) {
        w.mc[x] = -1;
        w.grow[x] = Off{0, 0, 0};
        w.gcol[x] = Off{0, 0, 0};
    }
    const int64_t words = ((int64_t)w.nnz + 31) / 32 + 1;
    for (int64_t x = gtid(); x < words; x += gstride())
        w.starts[x] = 0u;
    for (int64_t x = gtid(); x < (w.ntiles + kGroup - 1) / kGroup; x += gstride())
        w.gdead[x] = 0;
}

// Round, step 1: the best free entry of every free row and free column.  Four
// tiles side by side: their rows, weights and columns' state, then the rows'
// records.  A column's entries are combined in the warp; the first lane of a
// column that lies in the tile whole stores its record, a column cut by a
// tile's end is merged by compare-and-swap.
__device__ __forceinline__ void gm_best(const Work &w)
{
    if (w.ctl->err || !w.ctl->active)
        return;
    constexpr int kU = 4;
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = gstride() >> 5;
    const int32_t nnz = w.nnz, ntiles = w.ntiles;
    const int32_t groups = (ntiles + kGroup - 1) / kGroup;
    const int32_t round = w.ctl->iterations + 1;
    Ctl *ctl = w.ctl;
    for (int64_t g = gtid() >> 5; g < groups; g += nwarps) {
        const int32_t tg = (int32_t)g * kGroup;
        const unsigned was = w.gdead[g];
        const int left = ntiles - tg;
        const unsigned all = left >= kGroup ? (1u << kGroup) - 1u : (1u << left) - 1u;
        const unsigned alive = all & ~was;
        if (!alive)
            continue;
        int32_t c0 = 0;
        uint32_t mask = 1u;
        if ((alive >> lane) & 1u) {  // (lanes past the group have no bit)
            c0 = __ldg(w.tile_col + tg + lane);
            mask = __ldg(w.starts + tg + lane);
        }
        unsigned dead = 0u;
#pragma unroll
        for (int h = 0; h < kGroup; h += kU) {
            if (!((alive >> h) & ((1u << kU) - 1u)))
                continue;
            int32_t r[kU], j[kU];
            long long key[kU];
            uint32_t mk[kU];
            Off cur[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const bool on = (alive >> (h + u)) & 1u;
                const int32_t p = (tg + h + u) * kTile + lane;
                mk[u] = __shfl_sync(FULL_MASK, mask, h + u);
                const bool valid = on && p < nnz;
                j[u] = lane_column(__shfl_sync(FULL_MASK, c0, h + u), mk[u], lane);
                r[u] = valid ? __ldcs(w.rowidx + p) : -1;
                key[u] = valid ? order_key(__ldcs(w.w + p)) : kKeyNone;
            }
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (r[u] >= 0 && w.mc[j[u]] >= 0)
                    r[u] = -1;
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                cur[u] = Off{0, 0, kMatched};
                if (r[u] >= 0)
                    cur[u] = ld_record(w.grow + r[u]);
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const bool fr = cur[u].pad != kMatched;
                if (!__any_sync(FULL_MASK, fr)) {
                    dead |= 1u << (h + u);
                    continue;
                }
                if (fr)
                    rec_fold(w.grow + r[u], cur[u], key[u], j[u], round, ctl);
                // the columns' best: largest key, then lowest position
                const int32_t base = (tg + h + u) * kTile;
                long long k = fr ? key[u] : kKeyNone;
                int32_t at = lane;
                if (mk[u] <= 1u) {
                    const unsigned long long o = (unsigned long long)k ^ 0x8000000000000000ull;
                    const unsigned hi = (unsigned)(o >> 32);
                    const unsigned mh = __reduce_max_sync(FULL_MASK, hi);
                    const unsigned lo = hi == mh ? (unsigned)o : 0u;
                    const unsigned ml = __reduce_max_sync(FULL_MASK, lo);
                    const unsigned eq = __ballot_sync(FULL_MASK, hi == mh && lo == ml && fr);
                    at = eq ? __ffs(eq) - 1 : 0;
                    k = (long long)((((unsigned long long)mh << 32) | ml) ^ 0x8000000000000000ull);
                } else {
                    const uint32_t after = __funnelshift_rc(mk[u], 0u, lane + 1);
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const long long k2 = __shfl_down_sync(FULL_MASK, k, off);
                        const int32_t a2 = __shfl_down_sync(FULL_MASK, at, off);
                        // (equal keys: the lower lane's, this one; past lane 31
                        // the shuffle returns the lane's own values)
                        if ((after & ((1u << off) - 1u)) == 0u && k2 > k) {
                            k = k2;
                            at = a2;
                        }
                    }
                }
                const bool head = base + lane < nnz && (lane == 0 || ((mk[u] >> lane) & 1u));
                if (head && k != kKeyNone) {
                    Off *c = w.gcol + j[u];
                    if (segment_complete(mk[u], lane, base, nnz, w.starts, tg + h + u))
                        *c = Off{k, base + at, round};
                    else
                        rec_fold(c, ld_record(c), k, base + at, round, ctl);
                }
            }
        }
        if (lane == 0 && dead)
            w.gdead[g] = (uint8_t)(was | dead);
    }
}

__global__ void __launch_bounds__(kThreads, 4) k_gm_best(const Work *__restrict__ W)
{
    gm_best(*W);
}

// Round, step 2: a free column whose entry is also its row's is matched.
__device__ __forceinline__ void gm_match(const Work &w)
{
    unsigned long long matched = 0;
    if (!w.ctl->err && w.ctl->active) {
        const int32_t round = w.ctl->iterations + 1;
        for (int64_t j = gtid(); j < w.n; j += gstride()) {
            if (w.mc[j] >= 0)
                continue;
            const Off c = w.gcol[j];
            if (c.pad != round)
                continue;
            const int32_t i = w.rowidx[c.who];
            if (w.grow[i].who != (int32_t)j || w.grow[i].pad != round)
                continue;
            w.mc[j] = i;
            // (a matched column's record is not looked at again: it keeps the
            // weight for the sum)
            w.gcol[j].key = __double_as_longlong(w.w[c.who]);
            w.grow[i].pad = kMatched;  // (only this column's thread gets here for row i)
            ++matched;
        }
    }
    block_add_u64(matched, &w.ctl->pass_flips);
}

__global__ void k_gm_match(const Work *__restrict__ W)
{
    gm_match(*W);
}

// Graph form: the block that finishes last ends the round (its count of
// finished blocks orders it after every other block's matches).
__global__ void k_gm_match_graph(const Work *__restrict__ W, cudaGraphConditionalHandle h)
{
    const Work &w = *W;
    gm_match(w);
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&w.ctl->flip_done, 1u) == gridDim.x - 1) {
            __threadfence();
            w.ctl->flip_done = 0u;
            cudaGraphSetConditional(h, control_step(w.ctl, false) ? 1u : 0u);
        }
    }
}

// All rounds of a small problem in one cluster, with cluster barriers between
// the steps and no launch per round.
__global__ void __cluster_dims__(8, 1, 1) __launch_bounds__(1024)
    k_gm_cluster(const Work *__restrict__ W)
{
    const Work &w = *W;
    for (;;) {
        gm_best(w);
        cluster_sync();
        gm_match(w);
        cluster_sync();
        if (gtid() == 0)
            control_step(w.ctl, false);
        cluster_sync();
        // (last written before the barrier)
        if (!*(volatile int32_t *)&w.ctl->active)
            return;
    }
}

}  // namespace

void launch_greedy_cluster(const Work *d, const Shape &, Sink &k)
{
    void *a[] = {(void *)&d};
    k.launch((const void *)k_gm_cluster, 8, 1024, a);
}

void launch_greedy_init(const Work *d, const Shape &sh, Sink &k)
{
    void *a[] = {(void *)&d};
    k.launch((const void *)k_gm_reset, (unsigned)sh.num_sms * 8, kThreads, a);
    launch_check_colptr(d, sh, k);
    launch_mark_starts(d, sh, k);
    launch_check_entries(d, sh, k);
}

void launch_greedy_round(const Work *d, const Shape &sh, bool graph, cudaGraphConditionalHandle h,
                         Sink &k)
{
    void *a[] = {(void *)&d};
    void *ah[] = {(void *)&d, (void *)&h};
    k.launch((const void *)k_gm_best, (unsigned)sh.num_sms * 4, kThreads, a);
    if (graph) {
        k.launch((const void *)k_gm_match_graph, (unsigned)sh.num_sms * 8, kThreads, ah);
    } else {
        k.launch((const void *)k_gm_match, (unsigned)sh.num_sms * 8, kThreads, a);
        launch_control(d, sh, false, h, k);
    }
}

}  // namespace awpm

// CUDA kernels (sm_103a) of the weight-increasing alternating 4-cycle phase
// (arXiv 1801.09809, Section 5.3, Algorithms 2-6).
//
// The paper's message exchanges become arrays indexed by column in device
// memory: the A- and B-requests of Steps A and B never leave registers (one
// fused edge-parallel kernel does the lookup and the gain), Step C is a
// segmented arg-max inside each warp plus a 128-bit compare-and-swap for the
// columns that straddle a tile boundary, and Step D is one compare-and-swap
// selection per key column followed by an in-place flip.
//
// Every kernel reads the problem from a device-resident descriptor (Work) and
// runs a fixed, GPU-sized grid with grid-stride loops, so one instantiated
// CUDA graph serves every problem of a context.
#include <math.h>
#include <stdlib.h>

#include "awpm.h"
#include "awpm_dev.h"
#include "awpm_internal.h"

namespace awpm {

// Closing-edge ranges longer than this go to the warp-cooperative search
// (shorter ones to a binary search per lane).  On an R-MAT graph of scale 22
// (n = 4.2 M, 69 M nonzeros) 64 measured 4.5 us per search launch faster
// than 32, and 16 was 18 us slower.
constexpr int32_t kCoopMin = 64;
// Quiet NaN: wm[j] before the entry pass finds the matched entry of column j.
constexpr unsigned long long kNaNBits = 0x7ff8000000000000ull;

// ---------------------------------------------------------------------------
// small device helpers
// ---------------------------------------------------------------------------

// Index checks of builds with AWPM_DEBUG_BOUNDS: an index derived from data
// (a row, a mate, a position) outside [0, lim) sets kErrBounds (reported as
// AWPM_ERR_INTERNAL) and the access is skipped; nothing traps.  Other builds
// compile the checks away.
#ifdef AWPM_DEBUG_BOUNDS
__device__ __noinline__ bool in_bounds(Ctl *ctl, long long i, long long lim)
{
    if (i >= 0 && i < lim)
        return true;
    atomicOr(&ctl->err, kErrBounds);
    return false;
}
#define AWPM_IN(ctl, i, lim) in_bounds((ctl), (long long)(i), (long long)(lim))
#else
#define AWPM_IN(ctl, i, lim) true
#endif

__device__ __forceinline__ bool gate(const Ctl *ctl)
{
    return *(volatile const unsigned *)&ctl->err == 0u &&
           *(volatile const int32_t *)&ctl->active != 0;
}

// Deterministic block sum (fixed tree).  All threads call.
__device__ double block_sum_f64(double v)
{
    __shared__ double sm[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_down_sync(FULL_MASK, v, o);
    __syncthreads();
    if (lane == 0)
        sm[wid] = v;
    __syncthreads();
    v = 0.0;
    if (wid == 0) {
        v = (lane < (int)(blockDim.x >> 5)) ? sm[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            v += __shfl_down_sync(FULL_MASK, v, o);
    }
    return v;
}

// Column signatures: a partitioned Bloom filter of the column's rows in 64
// bits, one bit per row in each 32-bit half, both positions taken from one
// multiplicative hash of the row (bits 27..31 select the bit of the low
// half, bits 22..26 that of the high half).  A row with either bit clear is
// not stored in the column.  With 32-bit halves the test needs no 64-bit
// shifts.
__device__ __forceinline__ unsigned long long sig_mask(int32_t r)
{
    const uint32_t h = (uint32_t)r * 0x9E3779B1u;
    return ((unsigned long long)(1u << ((h >> 22) & 31u)) << 32) | (1u << (h >> 27));
}

__device__ __forceinline__ bool sig_has(unsigned long long sig, int32_t r)
{
    const uint32_t h = (uint32_t)r * 0x9E3779B1u;
    return (((uint32_t)sig >> (h >> 27)) & ((uint32_t)(sig >> 32) >> ((h >> 22) & 31u)) & 1u) !=
           0u;
}

// ---- per-column open-addressing tables -------------------------------------
// Column c owns the 2 * deg(c) slots [2 colptr[c], 2 colptr[c+1]) of htab;
// a slot holds (position << 32 | row), all ones when empty.  Linear probing
// from slot_start(); the table is at most half full, so every probe sequence
// meets an empty slot or the row.

constexpr unsigned long long kSlotEmpty = ~0ull;

__device__ __forceinline__ uint32_t row_mix(int32_t r)
{
    uint32_t h = (uint32_t)r;
    h ^= h >> 16;
    h *= 0x85ebca6bu;
    h ^= h >> 13;
    h *= 0xc2b2ae35u;
    h ^= h >> 16;
    return h;
}

__device__ __forceinline__ int32_t slot_start(int32_t r, int32_t base, int32_t size)
{
    return base + (int32_t)__umulhi(row_mix(r), (uint32_t)size);
}

// ---- blocked Bloom filters of long columns (binary-search lookup) -------------
// A column with more than Work::bloom_min rows, stored at positions [s, e), owns
// the words [s/4, (e-1)/4] of the bloom array: one 32-bit word per 4 nonzeros (a
// word at a boundary may be shared with the neighbouring column, which only
// adds false positives).  Each row sets three bits of one word, word and bits
// picked by a hash of the row; a row with a clear bit is not in the column.
// Long columns are where the 64-bit signature fills up, so this filter keeps
// most of their absent closing entries away from the search.

// Rows above which a column has a Bloom filter (binary-search lookup).  A filter
// entry costs the entry pass an atomic (135 of 387 us on the R-MAT graph of scale
// 22 from 32 rows up), and only the first pass's lookups use many of them.
// Whole solves of that graph: 1.447 ms from 32 rows up, 1.435 from 64, 1.439 from
// 128, 1.53 from 512.  Where the average column is that long the lookups are the
// larger part: from 64 and from 32 rows up, random with 55 entries a column, n =
// 400,000: a search 453 / 411 us, a solve 607 / 557; with 41, n = 1 M, 724 / 660
// and 854 / 793; with 37, n = 600,000, 395 / 376 and 484 / 469; against that,
// banded with 41, n = 500,000, 639 / 669 and 7,183 / 7,333.
constexpr int32_t kBloomMin = 64, kBloomMinLong = 32;
int32_t bloom_min(int32_t n, int32_t nnz)
{
    return nnz / 40 >= n ? kBloomMinLong : kBloomMin;
}

__device__ __forceinline__ void bloom_key(int32_t r, int32_t s, int32_t e, uint32_t &word,
                                          uint32_t &bits)
{
    // multiplicative hashes (top bits), with constants other than the
    // column signature's so the two filters reject different rows
    const uint32_t h = (uint32_t)r * 0x85EBCA6Bu;
    const uint32_t w0 = (uint32_t)s >> 2;
    const uint32_t nw = (((uint32_t)e - 1u) >> 2) - w0 + 1u;
    word = w0 + __umulhi(h, nw);
    const uint32_t h2 = (uint32_t)r * 0xC2B2AE35u;
    bits = (1u << (h2 >> 27)) | (1u << ((h2 >> 22) & 31u)) | (1u << ((h2 >> 17) & 31u));
}

// ---- cache-policy loads -------------------------------------------------------

__device__ __forceinline__ unsigned long long policy_evict_last()
{
    unsigned long long pol;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

// Row record of `row`: the signature, range and matched weight of the column
// matched to it (two arrays, so that the signature test gathers 8 bytes per
// candidate).
__device__ __forceinline__ void put_rowrec(const Work &w, int32_t row, int32_t s, int32_t e,
                                           unsigned long long sig, double wmatch)
{
    w.rsig[row] = sig;
    // one 16-byte store
    *reinterpret_cast<int4 *>(w.rrange + row) =
        make_int4(s, e, __double2loint(wmatch), __double2hiint(wmatch));
}

__device__ __forceinline__ RowRange ld_range(const RowRange *p)
{
    const int4 v = __ldg(reinterpret_cast<const int4 *>(p));
    RowRange g;
    g.s = v.x;
    g.e = v.y;
    g.w = __hiloint2double(v.w, v.z);
    return g;
}

__device__ __forceinline__ unsigned long long ld_u64_last(const unsigned long long *ptr,
                                                          unsigned long long pol)
{
    unsigned long long v;
    asm volatile("ld.global.nc.L2::cache_hint.b64 %0, [%1], %2;" : "=l"(v) : "l"(ptr), "l"(pol));
    return v;
}

__device__ __forceinline__ int32_t ld_i32_last(const int32_t *ptr, unsigned long long pol)
{
    int32_t v;
    asm volatile("ld.global.nc.L2::cache_hint.b32 %0, [%1], %2;" : "=r"(v) : "l"(ptr), "l"(pol));
    return v;
}

// Warp-cooperative search of row `key` among the sorted rows rowidx[s, s+len)
// for one lane's request, all 32 lanes taking part: each round every lane
// reads one pivot, a ballot picks the chunk that can hold the key and the
// range shrinks 32-fold (a 100,000-row column takes 4 rounds instead of 17
// dependent probes).  Returns the position or -1.  Called by the whole warp.
__device__ __forceinline__ int32_t coop_find(const int32_t *__restrict__ rowidx, int32_t s,
                                             int32_t len, int32_t key, int lane)
{
    while (len > 32) {
        const int32_t step = (len + 31) >> 5;
        const int32_t off = lane * step;
        const int32_t v = off < len ? __ldg(rowidx + s + off) : 0x7fffffff;
        const unsigned le = __ballot_sync(FULL_MASK, v <= key);
        if (le == 0)
            return -1;
        const int c = 31 - __clz(le);
        s += c * step;
        const int32_t rest = len - c * step;
        len = rest < step ? rest : step;
    }
    const int32_t v = lane < len ? __ldg(rowidx + s + lane) : -1;
    const unsigned eq = __ballot_sync(FULL_MASK, v == key);
    return eq ? s + __ffs(eq) - 1 : -1;
}

// ---------------------------------------------------------------------------
// Initialisation and validation (before the loop of Algorithm 2)
// ---------------------------------------------------------------------------

// Clear one set of the incremental passes' bitmaps.
__device__ __forceinline__ void inc_clear(const Work &w, int set)
{
    for (int64_t x = gtid(); x < kMapSmallBits / 32; x += gstride())
        w.map_small[set][x] = 0u;
    for (int64_t x = gtid(); x < w.map_bits / 32; x += gstride())
        w.map_large[set][x] = 0u;
    for (int64_t x = gtid(); x < w.n / 32 + 2; x += gstride()) {
        w.colfull[set][x] = 0u;
        w.colpos[set][x] = 0u;
    }
    for (int64_t x = gtid(); x < w.ntiles / 32 + 1; x += gstride())
        w.tilemark[set][x] = 0u;
}

// Clear everything a solve expects to start at zero (or empty).
__global__ void k_reset(const Work *__restrict__ W)
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
        c->d_candidates = c->d_found = c->d_positive = 0ull;
        c->weight_in = 0.0;
        c->weight_out = 0.0;
        if (w.bw.count > 0) {
            *w.bw.active = 0;
            *w.bw.tlist_n = 0;
        }
    }
    const bool rec = !w.rec_clean;
    for (int64_t j = gtid(); j < w.n; j += gstride()) {
        w.mr[j] = -1;
        if (rec) {
            w.best[j] = Rec{0.0, 0, 0};
            w.dsel[j] = Sel{0.0, 0, 0};
        }
        w.colsig[j] = 0ull;
        w.wm[j] = __longlong_as_double(kNaNBits);  // "no matched entry seen"
    }
    const int64_t words = ((int64_t)w.nnz + 31) / 32 + 1;
    for (int64_t x = gtid(); x < words; x += gstride())
        w.starts[x] = 0u;
    for (int64_t x = gtid(); x <= w.n / 32; x += gstride())
        w.winbits[x] = 0u;
    if (w.lookup == AWPM_LOOKUP_HASH && w.htab)
        for (int64_t x = gtid(); x < 2 * (int64_t)w.nnz; x += gstride())
            w.htab[x] = kSlotEmpty;
    if (w.bloom)
        for (int64_t x = gtid(); x <= (int64_t)w.nnz / 4; x += gstride())
            w.bloom[x] = 0u;
    if (w.inc) {
        for (int64_t x = gtid(); x < w.ntiles; x += gstride()) {
            w.foundbits[x] = 0u;
            w.posbits[x] = 0u;
        }
        inc_clear(w, 0);
        inc_clear(w, 1);
    }
    if (w.rowsig)
        for (int64_t x = gtid(); x < w.n; x += gstride())
            w.rowsig[x] = 0ull;
    if (w.psel) {
        for (int64_t j = gtid(); j < w.n; j += gstride())
            w.psel[j] = Sel{0.0, 0, 0};
        for (int64_t x = gtid(); x <= w.n / 32; x += gstride()) {
            w.pslive[x] = 0u;
            w.pstaken[x] = 0u;
            w.psused[x] = 0u;
        }
    }
    for (int64_t b = gtid(); b < w.bw.count; b += gstride()) {
        w.bw.mdone[b] = 0;
        w.bw.miter[b] = 0;
        w.bw.mconv[b] = 0;
        w.bw.mflips[b] = 0ull;
        w.bw.mcycles[b] = 0ull;
    }
}

// colptr[0] = 0, non-decreasing, colptr[n] = nnz.  An empty column cannot
// hold a matched entry, so it already rules out a perfect matching.
__global__ void k_check_colptr(const Work *__restrict__ W)
{
    const Work &w = *W;
    for (int64_t j = gtid(); j <= w.n; j += gstride()) {
        const int32_t c = w.colptr[j];
        const bool bad = (j == 0 && c != 0) || (j < w.n && w.colptr[j + 1] < c) ||
                         (j == w.n && c != w.nnz);
        if (bad)
            raise_err(w.ctl, kErrInvalid);
        else if (j < w.n && w.colptr[j + 1] == c)
            raise_err(w.ctl, kErrNotPerfect);
    }
}

// The column-pointer check and the start marks in one pass over colptr (the
// solve's initialisation): a column's start bit and tile entries are written
// only when its range lies inside [0, nnz], so a bad colptr (reported as
// AWPM_ERR_INVALID_ARG, which gates every later kernel) writes nothing out
// of range.
__global__ void k_check_mark(const Work *__restrict__ W)
{
    const Work &w = *W;
    for (int64_t j = gtid(); j <= w.n; j += gstride()) {
        const int32_t c = w.colptr[j];
        const int32_t e = j < w.n ? w.colptr[j + 1] : c;
        const bool bad = (j == 0 && c != 0) || (j < w.n && e < c) || (j == w.n && c != w.nnz);
        if (bad) {
            raise_err(w.ctl, kErrInvalid);
            continue;
        }
        if (j == w.n)
            continue;
        if (e == c) {
            raise_err(w.ctl, kErrNotPerfect);
            continue;
        }
        if (c < 0 || e > w.nnz)
            continue;  // (reported by the check of the last pointer)
        atomicOr(&w.starts[c >> 5], 1u << (c & 31));
        for (int64_t t = ((int64_t)c + kTile - 1) / kTile; t * kTile < e; ++t)
            w.tile_col[t] = (int32_t)j;
    }
}

// Column-start bitmap and the first column of every tile.
__global__ void k_mark_starts(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (w.ctl->err & kErrInvalid)
        return;
    for (int64_t j = gtid(); j < w.n; j += gstride()) {
        const int32_t s = w.colptr[j], e = w.colptr[j + 1];
        if (s < e) {
            atomicOr(&w.starts[s >> 5], 1u << (s & 31));
            for (int64_t t = ((int64_t)s + kTile - 1) / kTile; t * kTile < e; ++t)
                w.tile_col[t] = (int32_t)j;
        }
    }
}

// One pass over the entries: row range, sortedness inside columns, finite
// weights, the column signatures (OR of sig_mask(row) over each column) and the
// matched weight of every column: the entry (mate_in[j], j) stores its weight
// as wm[j]; with the binary-search lookup also the Bloom filters of the long
// columns.  Column numbers come from the start bitmap, exact once no column is
// empty (empty columns were reported by the column-pointer check and always
// stay below n).
//
// The kernel is bound by its instructions, not by its 12 bytes per entry, so a
// lane takes four consecutive entries (a warp 128, with 16-byte loads where the
// arrays are aligned): rows of one column are OR-ed in the lane, and one
// segmented ladder over the warp serves four tiles.  A column that lies in the
// 128 entries whole is stored, one cut by their end merged with atomics.
// Measured on the R-MAT graph of scale 22: 445 us with a lane per entry (two
// tiles per round, a ladder each), 387 us so, 252 of them without the
// filters (three, four and six blocks per SM: 400, 395 and 408 us).
__global__ void __launch_bounds__(kThreads, 5) k_entries(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (w.ctl->err & kErrInvalid)
        return;
    const int lane = threadIdx.x & 31;
    const int32_t nwarps = (int32_t)(gstride() >> 5);
    const int32_t n = w.n, nnz = w.nnz, ntiles = w.ntiles;
    const int32_t *__restrict__ rowidx = w.rowidx;
    const double *__restrict__ wv = w.w;
    const bool aligned = ((((uintptr_t)rowidx) | ((uintptr_t)wv)) & 15u) == 0u;
    const int32_t blocks = (ntiles + 3) >> 2;
    unsigned bits = 0;
    for (int32_t blk = (int32_t)(gtid() >> 5); blk < blocks; blk += nwarps) {
        const int32_t base = blk * 128;
        const int32_t p = base + 4 * lane;  // (used where entries are left)
        int32_t r[4];
        double x[4];
        const int32_t left = nnz - base - 4 * lane;
        const int nv = left >= 4 ? 4 : left;  // entries of this lane (may be <= 0)
        if (aligned && nnz - base >= 128) {
            const int4 v = __ldcs(reinterpret_cast<const int4 *>(rowidx + p));
            const double2 xa = __ldcs(reinterpret_cast<const double2 *>(wv + p));
            const double2 xb = __ldcs(reinterpret_cast<const double2 *>(wv + p) + 1);
            r[0] = v.x, r[1] = v.y, r[2] = v.z, r[3] = v.w;
            x[0] = xa.x, x[1] = xa.y, x[2] = xb.x, x[3] = xb.y;
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                r[u] = u < nv ? __ldcs(rowidx + p + u) : 0;
                x[u] = u < nv ? __ldcs(wv + p + u) : 0.0;
            }
        }
        // the lane's tile, its start bits and first column
        const int32_t t = blk * 4 + (lane >> 3);
        const int sh = (lane & 7) * 4;
        const uint32_t word = t < ntiles ? __ldg(w.starts + t) : 0u;
        const int32_t c0 = t < ntiles ? __ldg(w.tile_col + t) : 0;
        const int32_t first = lane == 0 && base > 0 ? __ldg(rowidx + base - 1) : 0;
        // does a column start after the block (or the matrix end there)?
        const bool ends = nnz - base <= 128 || (__ldg(w.starts + blk * 4 + 4) & 1u);
        const uint32_t nib = (word >> sh) & 15u;
        const uint32_t inner = nib & 14u;  // columns starting inside the lane
        int32_t j[4];
        j[0] = c0 + __popc(word & ((2u << sh) - 1u) & ~1u);
        j[1] = j[0] + ((nib >> 1) & 1);
        j[2] = j[1] + ((nib >> 2) & 1);
        j[3] = j[2] + ((nib >> 3) & 1);
        int32_t mate[4];
        mate[0] = nv > 0 ? __ldg(w.mate_in + j[0]) : -1;
#pragma unroll
        for (int u = 1; u < 4; ++u)
            mate[u] = u < nv && ((nib >> u) & 1u) ? __ldg(w.mate_in + j[u]) : -1;
        // only the lane's first and last columns can be long
        int32_t s0 = 0, e0 = 0, s3 = 0, e3 = 0;
        if (w.bloom && nv > 0) {
            s0 = s3 = __ldg(w.colptr + j[0]);
            e0 = e3 = __ldg(w.colptr + j[0] + 1);
            if (inner && nv == 4) {
                s3 = __ldg(w.colptr + j[3]);
                e3 = __ldg(w.colptr + j[3] + 1);
            }
        }
        int32_t before = __shfl_up_sync(FULL_MASK, r[3], 1);
        if (lane == 0)
            before = first;
        // the lane's OR up to the first inner start (head), from the last one
        // on (tail), and the columns between
        uint32_t hl = 0u, hh = 0u, tl = 0u, th = 0u;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (u > 0 && !((nib >> u) & 1u))
                mate[u] = mate[u - 1];
            if (u > 0 && ((nib >> u) & 1u)) {
                // a column starts here: the one before ends in this lane
                if (inner & ((1u << u) - 1u)) {  // and began in it
                    if (j[u - 1] < n)
                        w.colsig[j[u - 1]] = ((unsigned long long)th << 32) | tl;
                } else {
                    hl = tl;
                    hh = th;
                }
                tl = th = 0u;
            }
            if (u < nv) {
                const bool in_range = r[u] >= 0 && r[u] < n;
                if (!in_range)
                    bits |= kErrInvalid;
                if ((__double2hiint(x[u]) & 0x7ff00000) == 0x7ff00000)  // inf or NaN
                    bits |= kErrNonfinite;
                if (p + u > 0 && !((nib >> u) & 1u) && (u == 0 ? before : r[u - 1]) >= r[u])
                    bits |= kErrUnsorted;
                if (mate[u] == r[u])
                    w.wm[j[u]] = x[u];
                if (in_range) {
                    const uint32_t h = (uint32_t)r[u] * 0x9E3779B1u;  // (sig_mask)
                    tl |= 1u << (h >> 27);
                    th |= 1u << ((h >> 22) & 31u);
                    const bool head = !(inner & ((2u << u) - 1u));
                    const bool tail = !(inner >> (u + 1));
                    const int32_t s = head ? s0 : s3, e = head ? e0 : e3;
                    if ((head || tail) && e - s > w.bloom_min) {
                        uint32_t word_b, b;
                        bloom_key(r[u], s, e, word_b, b);
                        atomicOr(w.bloom + word_b, b);
                    }
                }
            }
        }
        if (!inner) {
            hl = tl;
            hh = th;
        }
        if (!__any_sync(FULL_MASK, lane == 0 ? inner : nib)) {
            // one column: one warp-wide OR
            const unsigned lo = __reduce_or_sync(FULL_MASK, hl);
            const unsigned hi = __reduce_or_sync(FULL_MASK, hh);
            if (lane == 0 && j[0] < n) {
                const unsigned long long v = ((unsigned long long)hi << 32) | lo;
                if ((nib & 1u) && ends)
                    w.colsig[j[0]] = v;
                else if (v)
                    atomicOr(w.colsig + j[0], v);
            }
            continue;
        }
        // head parts of the lanes to the right, as far as the column reaches:
        // the part of lane l continues in lane l + 1 when no column starts
        // inside l or at l + 1 (the last lane's after the block)
        bool next_starts = __shfl_down_sync(FULL_MASK, nib, 1) & 1u;
        if (lane == 31)
            next_starts = ends;
        bool open = !inner && !next_starts;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t l2 = __shfl_down_sync(FULL_MASK, hl, off);
            const uint32_t h2 = __shfl_down_sync(FULL_MASK, hh, off);
            const bool o2 = __shfl_down_sync(FULL_MASK, (int)open, off) != 0;
            if (open && lane + off < 32) {
                hl |= l2;
                hh |= h2;
                open = o2;
            }
        }
        const uint32_t nl = __shfl_down_sync(FULL_MASK, hl, 1);
        const uint32_t nh = __shfl_down_sync(FULL_MASK, hh, 1);
        const bool nopen = __shfl_down_sync(FULL_MASK, (int)open, 1) != 0;
        if (nv > 0 && (lane == 0 || (nib & 1u)) && j[0] < n) {
            const unsigned long long v = ((unsigned long long)hh << 32) | hl;
            if ((nib & 1u) && !open)
                w.colsig[j[0]] = v;
            else if (v)
                atomicOr(w.colsig + j[0], v);
        }
        if (inner && j[3] < n) {
            bool more = false;
            if (!next_starts) {
                if (lane == 31) {
                    more = true;
                } else {
                    tl |= nl;
                    th |= nh;
                    more = nopen;
                }
            }
            const unsigned long long v = ((unsigned long long)th << 32) | tl;
            if (!more)
                w.colsig[j[3]] = v;
            else if (v)
                atomicOr(w.colsig + j[3], v);
        }
    }
    bits = __reduce_or_sync(FULL_MASK, bits);
    if (lane == 0 && bits)
        raise_err(w.ctl, bits);
}

// Initialisation of the matching in two passes, so that no record is
// written to a scattered address:
//   k_init_mates (per column j): mc[j] = mate_in[j], and mr[mate_in[j]] = j
//     (a 4-byte scattered store per column; mr stays in L2 while it fills);
//     checks that every mate_in[j] is a row number and a stored entry of
//     column j (the entry pass left wm[j] = NaN where (mate_in[j], j) is not
//     stored); and the matched weights' sum, one partial per block into
//     wpart (the grid is at most kWsumBlocks), summed by k_wsum_final;
//   k_init_rows (per row r): the row record of r from column mr[r] (gathers
//     of that column's range, signature and matched weight; the records are
//     written row by row, whole sectors at a time), and the check that every
//     row got a column: with n columns and n rows that holds exactly when
//     mate_in is a permutation.
__global__ void k_init_mates(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (w.ctl->err) {
        if (threadIdx.x == 0)
            w.wpart[blockIdx.x] = 0.0;
        return;
    }
    constexpr int kU = 8;
    const int64_t stride = gstride();
    const int32_t n = w.n;
    unsigned bits = 0;
    double sum = 0.0;
    for (int64_t j0 = gtid(); j0 < n; j0 += kU * stride) {
        int32_t r[kU];
        double x[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int64_t j = j0 + u * stride;
            const bool ok = j < n;
            r[u] = ok ? w.mate_in[j] : -1;
            x[u] = ok ? w.wm[j] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int64_t j = j0 + u * stride;
            if (j >= n)
                continue;
            w.mc[j] = r[u];
            if (r[u] < 0 || r[u] >= n || gbits(x[u]) == (long long)kNaNBits) {
                bits |= kErrNotPerfect;
                continue;
            }
            w.mr[r[u]] = (int32_t)j;
            sum += x[u];
        }
    }
    bits = __reduce_or_sync(FULL_MASK, bits);
    if ((threadIdx.x & 31) == 0 && bits)
        raise_err(w.ctl, bits);
    sum = block_sum_f64(sum);
    if (threadIdx.x == 0)
        w.wpart[blockIdx.x] = sum;
}

__global__ void k_init_rows(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (w.ctl->err)
        return;
    constexpr int kU = 4;
    const int64_t stride = gstride();
    const int32_t n = w.n;
    bool bad = false;
    for (int64_t r0 = gtid(); r0 < n; r0 += kU * stride) {
        int32_t j[kU], cs[kU], ce[kU];
        unsigned long long sig[kU];
        double x[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int64_t r = r0 + u * stride;
            j[u] = r < n ? w.mr[r] : 0;
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int64_t r = r0 + u * stride;
            const bool ok = r < n && j[u] >= 0;
            bad |= r < n && j[u] < 0;
            cs[u] = ok ? __ldg(w.colptr + j[u]) : 0;
            ce[u] = ok ? __ldg(w.colptr + j[u] + 1) : 0;
            sig[u] = ok ? __ldg(w.colsig + j[u]) : 0ull;
            x[u] = ok ? __ldg(w.wm + j[u]) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int64_t r = r0 + u * stride;
            if (r < n)
                put_rowrec(w, (int32_t)r, cs[u], ce[u], sig[u], x[u]);
        }
    }
    if (__any_sync(FULL_MASK, bad) && (threadIdx.x & 31) == 0)
        raise_err(w.ctl, kErrNotPerfect);
}

// Per-column hash tables (only for AWPM_LOOKUP_HASH).
__global__ void __launch_bounds__(kThreads) k_hash_build(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (w.ctl->err || w.lookup != AWPM_LOOKUP_HASH || !w.htab)
        return;
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = gstride() >> 5;
    for (int64_t t = gtid() >> 5; t < w.ntiles; t += nwarps) {
        const int32_t p = (int32_t)(t * kTile) + lane;
        if (p >= w.nnz)
            continue;
        const int32_t j = lane_column(w.tile_col[t], w.starts[t], lane);
        const int32_t r = __ldcs(w.rowidx + p);
        const int32_t base = 2 * w.colptr[j];
        const int32_t size = 2 * (w.colptr[j + 1] - w.colptr[j]);
        const unsigned long long v = ((unsigned long long)(uint32_t)p << 32) | (uint32_t)r;
        int32_t pos = slot_start(r, base, size);
        int k = 0;
        for (; k < size; ++k) {
            if (atomicCAS(w.htab + pos, kSlotEmpty, v) == kSlotEmpty)
                break;
            if (++pos == base + size)
                pos = base;
        }
        if (k == size)
            raise_err(w.ctl, kErrInternal);
    }
}

// kGreedy: the weights are in the matched columns' records (gcol).
template <bool kGreedy>
__global__ void k_wsum_partial(const Work *__restrict__ W)
{
    const Work &w = *W;
    double s = 0.0;
    if (w.ctl->err == 0u)
        for (int64_t j = gtid(); j < w.n; j += gstride())
            s += !kGreedy ? w.wm[j] : w.mc[j] >= 0 ? __longlong_as_double(w.gcol[j].key) : 0.0;
    s = block_sum_f64(s);
    if (threadIdx.x == 0)
        w.wpart[blockIdx.x] = s;
}

// The sum of the first `parts` block partials (parts <= blockDim.x); 0 after
// an error.
__global__ void k_wsum_final(const Work *__restrict__ W, int out, int parts)
{
    const Work &w = *W;
    double s = block_sum_f64((int)threadIdx.x < parts ? w.wpart[threadIdx.x] : 0.0);
    if (w.ctl->err)
        s = 0.0;
    if (threadIdx.x == 0) {
        if (out)
            w.ctl->weight_out = s;
        else
            w.ctl->weight_in = s;
    }
}

// ---------------------------------------------------------------------------
// Batched solves: many matrices as one block-diagonal union
// ---------------------------------------------------------------------------
// Cycles never cross blocks (no entry joins two blocks), so every pass of
// the union is one pass of each matrix.  A matrix whose pass flips nothing
// (or that reached the pass cap) is finished: its tiles are skipped from then
// on and its counters stop, which gives each matrix exactly the passes,
// flips and result of a solve on its own.

// Offsets non-decreasing from 0 to n; matrix of every column.
__global__ void k_batch_cols(const Work *__restrict__ W)
{
    const Work &w = *W;
    const int32_t count = w.bw.count;
    const int32_t *n_off = w.bw.n_off;
    for (int64_t x = gtid(); x <= count; x += gstride()) {
        const int32_t o = n_off[x];
        if ((x == 0 && o != 0) || (x == count && o != w.n) || (x < count && n_off[x + 1] < o))
            raise_err(w.ctl, kErrInvalid);
    }
    // a warp per matrix writes the matrix number of its columns (clamped to
    // [0, n): offsets found invalid above raise the error but write nothing
    // out of range)
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = gstride() >> 5;
    for (int64_t b = gtid() >> 5; b < count; b += nwarps) {
        const int32_t lo = max(n_off[b], 0), hi = min(n_off[b + 1], w.n);
        for (int32_t x = lo + lane; x < hi; x += 32)
            w.bw.colmat[x] = (int32_t)b;
    }
}

// Every stored row lies in its column's block; nonzeros per matrix; the
// matrix of each tile and whether the tile stays inside one matrix.
__global__ void __launch_bounds__(kThreads) k_batch_check(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (w.ctl->err)
        return;
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = gstride() >> 5;
    const BatchWork &bw = w.bw;
    unsigned bad = 0;
    // four tiles per warp round, their loads side by side (the checks are
    // chains of dependent gathers)
    constexpr int kU = 4;
    for (int64_t t0 = gtid() >> 5; t0 < w.ntiles; t0 += kU * nwarps) {
        int32_t c0[kU], b[kU], r[kU];
        uint32_t mask[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int64_t t = t0 + u * nwarps;
            const bool tv = t < w.ntiles;
            c0[u] = tv ? w.tile_col[t] : 0;
            mask[u] = tv ? w.starts[t] : 1u;
            const int64_t p = t * kTile + lane;
            r[u] = tv && p < w.nnz ? w.rowidx[p] : -1;
        }
#pragma unroll
        for (int u = 0; u < kU; ++u)
            b[u] = r[u] >= 0 ? bw.colmat[lane_column(c0[u], mask[u], lane)] : 0;
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int64_t t = t0 + u * nwarps;
            if (r[u] >= 0 && (r[u] < bw.n_off[b[u]] || r[u] >= bw.n_off[b[u] + 1]))
                bad = 1;
            if (lane == 0 && t < w.ntiles) {
                const int32_t b0 = bw.colmat[c0[u]];
                const int32_t b1 =
                    (t + 1 < w.ntiles) ? bw.colmat[w.tile_col[t + 1]] : bw.colmat[w.n - 1];
                bw.tilemat[t] = b0 | (b0 == b1 ? kTileSingle : 0);
            }
        }
    }
    if (__any_sync(FULL_MASK, bad) && lane == 0)
        raise_err(w.ctl, kErrInvalid);
    for (int64_t b = gtid(); b < bw.count; b += gstride())
        bw.mnnz[b] = w.colptr[bw.n_off[b + 1]] - w.colptr[bw.n_off[b]];
}

// The tiles the next pass of a batched solve searches: those of matrices
// still running, and every tile spanning two matrices (its lanes of a
// finished matrix are skipped in the search).  Each tile at most once; the
// list's order (warp-aggregated appends) does not change any result, since
// the search's records and counters are order-free.  The count was zeroed
// by the reset (first pass) or the end-of-pass control.
__global__ void k_batch_list(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (w.ctl->err)
        return;
    const BatchWork &bw = w.bw;
    const int lane = threadIdx.x & 31;
    for (int64_t t0 = gtid() - lane; t0 < w.ntiles; t0 += gstride()) {
        const int64_t t = t0 + lane;
        bool keep = false;
        if (t < w.ntiles) {
            const int32_t tm = __ldg(bw.tilemat + t);
            keep = !(tm & kTileSingle) || !bw.mdone[tm & ~kTileSingle];
        }
        const unsigned m = __ballot_sync(FULL_MASK, keep);
        if (!m)
            continue;
        int32_t base = 0;
        if (lane == 0)
            base = atomicAdd(bw.tlist_n, __popc(m));
        base = __shfl_sync(FULL_MASK, base, 0);
        if (keep)
            bw.tlist[base + __popc(m & ((1u << lane) - 1u))] = (int32_t)t;
    }
}

// One block per matrix (grid-stride over matrices): deterministic sum of its
// matched weights.
__global__ void k_batch_wsum(const Work *__restrict__ W, int out)
{
    const Work &w = *W;
    const BatchWork &bw = w.bw;
    for (int64_t b = blockIdx.x; b < bw.count; b += gridDim.x) {
        double s = 0.0;
        if (w.ctl->err == 0u)
            for (int64_t j = bw.n_off[b] + threadIdx.x; j < bw.n_off[b + 1]; j += blockDim.x)
                s += w.wm[j];
        s = block_sum_f64(s);
        if (threadIdx.x == 0)
            (out ? bw.mw_out : bw.mw_in)[b] = s;
    }
}

// ---------------------------------------------------------------------------
// Row marking (Section 4): marks of the rows' neighbourhoods and the
// transpose of the pattern, built once per solve for AWPM_LOOKUP_ROWMARK
// ---------------------------------------------------------------------------

// The mark of row i: the signature (see sig_mask) of the columns k with a
// stored (i, k), each column named by its first position colptr[k] (the
// search has that number at hand from the row record), OR-ed over the
// entries with 64-bit atomics (skipped when the bits are already set).  Runs
// after validation: no column is empty, so the start bitmap gives exact
// columns and distinct first positions.
__global__ void __launch_bounds__(kThreads) k_rm_marks(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (w.ctl->err || !w.rowsig)
        return;
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = gstride() >> 5;
    for (int64_t t = gtid() >> 5; t < w.ntiles; t += nwarps) {
        const int32_t p = (int32_t)(t * kTile) + lane;
        if (p >= w.nnz)
            continue;
        const int32_t j = lane_column(__ldg(w.tile_col + t), __ldg(w.starts + t), lane);
        const int32_t i = __ldcs(w.rowidx + p);
        const unsigned long long m = sig_mask(__ldg(w.colptr + j));
        // bits only ever get set: a set bit in the (possibly stale) L1 copy
        // is set; otherwise ask the L2 copy, where the atomics land
        if ((w.rowsig[i] & m) != m && (__ldcg(w.rowsig + i) & m) != m)
            atomicOr(w.rowsig + i, m);
    }
}

// Exclusive prefix of one value per thread over a block of kRsThreads
// threads; the block's total into *total.  Called by the whole block.
__device__ __forceinline__ int32_t block_excl_scan(int32_t v, int32_t *total)
{
    __shared__ int32_t s_w[kRsThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(FULL_MASK, x, o);
        if (lane >= o)
            x += y;
    }
    if (lane == 31)
        s_w[warp] = x;
    __syncthreads();
    int32_t below = 0, tot = 0;
#pragma unroll
    for (int i = 0; i < kRsThreads / 32; ++i) {
        below += i < warp ? s_w[i] : 0;
        tot += s_w[i];
    }
    __syncthreads();
    *total = tot;
    return below + x - v;
}

// The transpose is a stable LSD radix sort of the entries (in CSC order) by
// row, 8 bits per pass: afterwards the CSC positions of each row's entries
// are contiguous and ascending, i.e. in column order.  Pass `pass` reads the
// keys of the previous pass (the row indices themselves first) and writes
// buffer pass & 1; passes at or above rs_passes do nothing.

// Digit counts of each block tile of kRsTile entries, stored digit-major
// (rs_hist[digit * rs_tiles + tile]) so one scan gives every scatter offset.
// A thread loads its 16 keys first; each warp counts into its own table.
__global__ void __launch_bounds__(kRsThreads) k_rs_hist(const Work *__restrict__ W, int pass)
{
    const Work &w = *W;
    if (w.ctl->err || pass >= w.rs_passes)
        return;
    constexpr int kWarps = kRsThreads / 32;
    __shared__ int32_t s_cnt[kWarps][kRsBins];
    const int warp = threadIdx.x >> 5;
    const int shift = 8 * pass;
    const int32_t *key = pass == 0 ? w.rowidx : w.rs_key[(pass - 1) & 1];
    for (int64_t tile = blockIdx.x; tile < w.rs_tiles; tile += gridDim.x) {
#pragma unroll
        for (int x = 0; x < kWarps; ++x)
            s_cnt[x][threadIdx.x] = 0;
        uint32_t k[kRsItems];
#pragma unroll
        for (int r = 0; r < kRsItems; ++r) {
            const int64_t e = tile * kRsTile + r * kRsThreads + threadIdx.x;
            k[r] = e < w.nnz ? (uint32_t)__ldcs(key + e) : 0xffffffffu;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kRsItems; ++r)
            if (k[r] != 0xffffffffu)
                atomicAdd(&s_cnt[warp][(k[r] >> shift) & 255u], 1);
        __syncthreads();
        int32_t c = 0;
#pragma unroll
        for (int x = 0; x < kWarps; ++x)
            c += s_cnt[x][threadIdx.x];
        w.rs_hist[(int64_t)threadIdx.x * w.rs_tiles + tile] = c;
        __syncthreads();
    }
}

// Scan of the digit counts, step 1: the total of every chunk of kScanChunk.
__global__ void __launch_bounds__(kRsThreads) k_rs_scan_a(const Work *__restrict__ W, int pass)
{
    const Work &w = *W;
    if (w.ctl->err || pass >= w.rs_passes)
        return;
    const int64_t m = (int64_t)kRsBins * w.rs_tiles;
    const int64_t chunks = (m + kScanChunk - 1) / kScanChunk;
    for (int64_t c = blockIdx.x; c < chunks; c += gridDim.x) {
        int32_t s = 0;
        for (int k = 0; k < kScanChunk / kRsThreads; ++k) {
            const int64_t x = c * kScanChunk + k * kRsThreads + threadIdx.x;
            if (x < m)
                s += w.rs_hist[x];
        }
        int32_t tot = 0;
        block_excl_scan(s, &tot);
        if (threadIdx.x == 0)
            w.rs_sums[c] = tot;
    }
}

// Step 2 (one block): exclusive prefix of the chunk totals, in place.
__global__ void __launch_bounds__(kRsThreads) k_rs_scan_b(const Work *__restrict__ W, int pass)
{
    const Work &w = *W;
    if (w.ctl->err || pass >= w.rs_passes)
        return;
    const int64_t m = (int64_t)kRsBins * w.rs_tiles;
    const int64_t chunks = (m + kScanChunk - 1) / kScanChunk;
    int32_t carry = 0;
    for (int64_t b0 = 0; b0 < chunks; b0 += kRsThreads) {
        const int64_t x = b0 + threadIdx.x;
        const int32_t v = x < chunks ? w.rs_sums[x] : 0;
        int32_t tot = 0;
        const int32_t pre = block_excl_scan(v, &tot);
        if (x < chunks)
            w.rs_sums[x] = carry + pre;
        carry += tot;
    }
}

// Step 3: every chunk's exclusive prefix plus the chunk's offset, in place;
// thread t takes the chunk's counts 8t .. 8t + 7.
__global__ void __launch_bounds__(kRsThreads) k_rs_scan_c(const Work *__restrict__ W, int pass)
{
    const Work &w = *W;
    if (w.ctl->err || pass >= w.rs_passes)
        return;
    constexpr int kPer = kScanChunk / kRsThreads;
    const int64_t m = (int64_t)kRsBins * w.rs_tiles;
    const int64_t chunks = (m + kScanChunk - 1) / kScanChunk;
    for (int64_t c = blockIdx.x; c < chunks; c += gridDim.x) {
        const int64_t x0 = c * kScanChunk + (int64_t)threadIdx.x * kPer;
        int32_t v[kPer];
        int32_t s = 0;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            v[k] = x0 + k < m ? w.rs_hist[x0 + k] : 0;
            s += v[k];
        }
        int32_t tot = 0;
        int32_t run = block_excl_scan(s, &tot) + w.rs_sums[c];
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            if (x0 + k < m)
                w.rs_hist[x0 + k] = run;
            run += v[k];
        }
    }
}

// Stable scatter of one pass.  A thread loads its kRsItems entries of the
// block tile; the tile is sorted by digit in shared memory (the entries
// placed 256 at a time, in order: within a warp, entries of equal digit --
// eight ballots -- are ranked by lane, and the warps' digit counts give each
// warp's offset; counts and running offsets alternate between two tables, so
// a round needs two barriers); then each digit's run is written to its
// global offset with consecutive threads on consecutive positions.
__global__ void __launch_bounds__(kRsThreads) k_rs_scatter(const Work *__restrict__ W, int pass)
{
    const Work &w = *W;
    if (w.ctl->err || pass >= w.rs_passes)
        return;
    constexpr int kWarps = kRsThreads / 32;
    __shared__ int32_t s_key[kRsTile];
    __shared__ int32_t s_val[kRsTile];
    __shared__ int32_t s_local[kRsBins];   // start of each digit's run in the tile
    __shared__ int32_t s_global[kRsBins];  // its global offset
    __shared__ int32_t s_base[2][kRsBins];
    __shared__ int32_t s_wcnt[2][kWarps][kRsBins];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int shift = 8 * pass;
    const int32_t *kin = pass == 0 ? w.rowidx : w.rs_key[(pass - 1) & 1];
    const int32_t *vin = pass == 0 ? nullptr : w.rs_val[(pass - 1) & 1];
    int32_t *kout = w.rs_key[pass & 1];
    int32_t *vout = w.rs_val[pass & 1];
    for (int64_t tile = blockIdx.x; tile < w.rs_tiles; tile += gridDim.x) {
        const int64_t first = tile * kRsTile;
        const int32_t count =
            (int32_t)(w.nnz - first < kRsTile ? w.nnz - first : (int64_t)kRsTile);
        int32_t kv[kRsItems], vv[kRsItems];
#pragma unroll
        for (int r = 0; r < kRsItems; ++r) {
            const int32_t x = r * kRsThreads + threadIdx.x;
            const bool valid = x < count;
            kv[r] = valid ? __ldcs(kin + first + x) : -1;
            vv[r] = valid ? (vin ? __ldcs(vin + first + x) : (int32_t)(first + x)) : 0;
        }
        s_base[0][threadIdx.x] = 0;  // digit counts of the tile first
#pragma unroll
        for (int x = 0; x < kWarps; ++x) {
            s_wcnt[0][x][threadIdx.x] = 0;
            s_wcnt[1][x][threadIdx.x] = 0;
        }
        s_global[threadIdx.x] = w.rs_hist[(int64_t)threadIdx.x * w.rs_tiles + tile];
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kRsItems; ++r)
            if (kv[r] >= 0)
                atomicAdd(&s_base[0][((uint32_t)kv[r] >> shift) & 255u], 1);
        __syncthreads();
        int32_t tot = 0;
        const int32_t start = block_excl_scan(s_base[0][threadIdx.x], &tot);
        s_local[threadIdx.x] = start;
        s_base[0][threadIdx.x] = start;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kRsItems; ++r) {
            const int q = r & 1;
            const bool valid = kv[r] >= 0;
            const int d = valid ? (int)(((uint32_t)kv[r] >> shift) & 255u) : kRsBins;
            // lanes with the same digit: agree on all 8 bits and on validity
            const unsigned vm = __ballot_sync(FULL_MASK, valid);
            unsigned peers = valid ? vm : ~vm;
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                const unsigned m = __ballot_sync(FULL_MASK, (d >> b) & 1);
                peers &= ((d >> b) & 1) ? m : ~m;
            }
            const int rank = __popc(peers & ((1u << lane) - 1u));
            if (valid && rank == 0)
                s_wcnt[q][warp][d] = __popc(peers);
            __syncthreads();
            if (valid) {
                int32_t off = s_base[q][d] + rank;
                for (int x = 0; x < warp; ++x)
                    off += s_wcnt[q][x][d];
                s_key[off] = kv[r];
                s_val[off] = vv[r];
            }
            int32_t add = 0;
#pragma unroll
            for (int x = 0; x < kWarps; ++x) {
                add += s_wcnt[q][x][threadIdx.x];
                s_wcnt[q ^ 1][x][threadIdx.x] = 0;
            }
            s_base[q ^ 1][threadIdx.x] = s_base[q][threadIdx.x] + add;
            __syncthreads();
        }
        for (int32_t x = threadIdx.x; x < count; x += kRsThreads) {
            const int32_t key = s_key[x];
            const int d = (int)(((uint32_t)key >> shift) & 255u);
            const int32_t g = s_global[d] + (x - s_local[d]);
            if (g >= 0 && g < w.nnz) {
                kout[g] = key;
                vout[g] = s_val[x];
            } else {
                raise_err(w.ctl, kErrInternal);
            }
        }
        __syncthreads();
    }
}

// Row pointers of the transpose from the sorted keys: row r starts at the
// first entry whose row is >= r.
__global__ void k_rm_rowptr(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (w.ctl->err || !w.trowptr)
        return;
    const int64_t nnz = w.nnz;
    if (nnz == 0) {
        for (int64_t r = gtid(); r <= w.n; r += gstride())
            w.trowptr[r] = 0;
        return;
    }
    const int32_t *key = w.rs_key[(w.rs_passes - 1) & 1];
    for (int64_t e = gtid(); e < nnz; e += gstride()) {
        const int32_t k = key[e];
        const int32_t prev = e > 0 ? key[e - 1] : -1;
        if (k < 0 || k >= w.n || prev > k) {  // not sorted rows: no transpose
            raise_err(w.ctl, kErrInternal);
            continue;
        }
        for (int32_t r = prev + 1; r <= k; ++r)
            w.trowptr[r] = (int32_t)e;
        if (e == nnz - 1)
            for (int64_t r = (int64_t)k + 1; r <= w.n; ++r)
                w.trowptr[r] = (int32_t)nnz;
    }
}

// Warp-cooperative search, in the ascending values arr[s, s+len), of the
// last one below `key` for one lane's request (all 32 lanes take part, as in
// coop_find).  Returns its index or -1.
__device__ __forceinline__ int32_t coop_last_below(const int32_t *__restrict__ arr, int32_t s,
                                                   int32_t len, int32_t key, int lane)
{
    while (len > 32) {
        const int32_t step = (len + 31) >> 5;
        const int32_t off = lane * step;
        const int32_t v = off < len ? __ldg(arr + s + off) : 0x7fffffff;
        const unsigned lt = __ballot_sync(FULL_MASK, v < key);
        if (lt == 0)
            return -1;
        const int c = 31 - __clz(lt);
        s += c * step;
        const int32_t rest = len - c * step;
        len = rest < step ? rest : step;
    }
    const int32_t v = lane < len ? __ldg(arr + s + lane) : 0x7fffffff;
    const unsigned lt = __ballot_sync(FULL_MASK, v < key);
    return lt ? s + 31 - __clz(lt) : -1;
}

// ---------------------------------------------------------------------------
// Steps A + B + C (Algorithms 3, 4, 5): fused edge-parallel cycle search
// ---------------------------------------------------------------------------

// Closing-entry lookups of one warp, queued across tiles (a ring of 64
// entries, struct of arrays in shared memory): a lane whose candidate passed
// the signature test leaves its request here, and the warp resolves 32
// requests at a time, one per lane, instead of searching with the one or two
// lanes of a tile that need it.
constexpr int kQueue = 64;
struct LookupQueue {
    int2 im[kQueue];  // row i, and m_j (the row looked up in column m_i)
    int2 jp[kQueue];  // root column j, and the position of (i, j)
};

// Resolve the queued requests head .. head + k - 1 (k <= 32, lane x takes
// request head + x): Bloom probe for long columns, then the column search
// (per lane up to kCoopMin rows, warp-cooperative above), or the hash probe,
// or with row marking the search of row m_j's entries (CSC positions,
// ascending) for the one inside column m_i's positions [lo, lo + len) (per
// lane, warp-cooperative above kCoopMin entries);
// a closing entry found gives the gain in the fixed order
// ((w_ij + w_q) - w(i, m_i)) - w(m_j, j), and a positive gain goes into the
// root's Step-C record (maximum gain, then lowest position; Algorithm 5).
// With foundbits, the outcome is also kept per entry (for the incremental
// passes).  Called by the whole warp.
//
// Returns bit 0: closing entry found, bit 1: positive gain.
template <int kLookup>
__device__ __forceinline__ unsigned resolve_inline(const Work *__restrict__ W, const int2 *qim,
                                                 const int2 *qjp, int head, int k)
{
    const Work &w = *W;
    const int lane = threadIdx.x & 31;
    const int32_t *__restrict__ rowidx = w.rowidx;
    const int32_t nnz = w.nnz;
    [[maybe_unused]] const int32_t nrows = w.n;
    Ctl *ctl = w.ctl;
    const int x = (head + lane) & (kQueue - 1);
    const bool act = lane < k;
    const int2 im = act ? qim[x] : make_int2(0, 0);
    const int32_t mj = im.y;
    // column m_i's rows rowidx[lo, lo + len) and w(i, m_i), from the row
    // record of i
    int32_t lo = 0, len = 0;
    double wmi = 0.0;
    if (act && AWPM_IN(ctl, im.x, nrows)) {
        const RowRange rg = ld_range(w.rrange + im.x);
        lo = rg.s;
        len = rg.e - rg.s;
        wmi = rg.w;
        if (!(AWPM_IN(ctl, lo, (long long)nnz + 1) && AWPM_IN(ctl, len, (long long)nnz - lo + 1)))
            lo = len = 0;
    }
    int32_t q = -1;
    if (kLookup == AWPM_LOOKUP_HASH) {
        const int32_t hbase = 2 * lo;
        const int32_t hsize = 2 * len;
        int32_t pos = hsize > 0 ? slot_start(mj, hbase, hsize) : 0;
        for (int32_t left = hsize; left > 0; --left) {
            const unsigned long long v = __ldg(w.htab + pos);
            if ((int32_t)(uint32_t)v == mj) {
                q = (int32_t)(v >> 32);
                break;
            }
            if (v == kSlotEmpty)
                break;
            if (++pos == hbase + hsize)
                pos = hbase;
        }
    } else if (kLookup == AWPM_LOOKUP_ROWMARK) {
        // column m_i's positions are [a, b); row m_j's entries tpos[lo, lo + len)
        const int32_t a = lo, b = lo + len;
        if (act) {
            lo = __ldg(w.trowptr + mj);
            len = __ldg(w.trowptr + mj + 1) - lo;
            if (lo < 0 || len < 0 || len > nnz - lo) {
                lo = 0;
                len = 0;
                raise_err(ctl, kErrInternal);
            }
        }
        unsigned longm = __ballot_sync(FULL_MASK, len > kCoopMin);
        while (longm) {
            const int src = __ffs(longm) - 1;
            longm &= longm - 1;
            const int32_t ss = __shfl_sync(FULL_MASK, lo, src);
            const int32_t sl = __shfl_sync(FULL_MASK, len, src);
            const int32_t sb = __shfl_sync(FULL_MASK, b, src);
            const int32_t f = coop_last_below(w.tpos, ss, sl, sb, lane);
            if (lane == src) {
                const int32_t v = f >= 0 ? __ldg(w.tpos + f) : -1;
                q = v >= a ? v : -1;
                len = 0;
            }
        }
        // short rows: the last entry below column m_i's end, per lane
        const int32_t s0 = lo;
        int32_t hi = lo + len;
        while (lo < hi) {
            const int32_t mid = (lo + hi) >> 1;
            if (__ldg(w.tpos + mid) < b)
                lo = mid + 1;
            else
                hi = mid;
        }
        if (len > 0 && lo > s0) {
            const int32_t v = __ldg(w.tpos + lo - 1);
            if (v >= a)
                q = v;
        }
    } else {
        if (len > w.bloom_min) {
            // long column: its Bloom filter rules most absent rows out first
            uint32_t word, b;
            bloom_key(mj, lo, lo + len, word, b);
            if ((__ldg(w.bloom + word) & b) != b)
                len = 0;
        }
        // long columns: the warp searches them together, one request at a time
        unsigned longm = __ballot_sync(FULL_MASK, len > kCoopMin);
        while (longm) {
            const int src = __ffs(longm) - 1;
            longm &= longm - 1;
            const int32_t ss = __shfl_sync(FULL_MASK, lo, src);
            const int32_t sl = __shfl_sync(FULL_MASK, len, src);
            const int32_t sk = __shfl_sync(FULL_MASK, mj, src);
            const int32_t f = coop_find(rowidx, ss, sl, sk, lane);
            if (lane == src) {
                q = f;
                len = 0;
            }
        }
        // short columns: binary search per lane (early exit on a hit)
        while (len > 0) {
            const int32_t half = len >> 1;
            const int32_t mid = lo + half;
            const int32_t v = __ldg(rowidx + mid);
            if (v == mj) {
                q = mid;
                break;
            }
            if (v < mj) {
                lo = mid + 1;
                len -= half + 1;
            } else {
                len = half;
            }
        }
    }
    const int2 jp = act ? qjp[x] : make_int2(-1, -1);
    if (q >= 0 && !(AWPM_IN(ctl, q, nnz) && AWPM_IN(ctl, jp.y, nnz) && AWPM_IN(ctl, jp.x, nrows)))
        q = -1;
    double gg = 0.0;
    bool pos = false;
    if (q >= 0) {
        const double wij = __ldg(w.w + jp.y);
        const double wq = __ldg(w.w + q);
        gg = ((wij + wq) - wmi) - __ldg(w.wm + jp.x);
        pos = gain_positive(gg);
    }
    // The queue holds entries in the order of their positions, so entries of
    // one column (and of one tile) sit side by side: each column's best gain
    // and each tile's bits are combined in the warp first, and one lane per
    // column or tile goes to memory.
    const unsigned any_found = __ballot_sync(FULL_MASK, q >= 0);
    const unsigned any_pos = __ballot_sync(FULL_MASK, pos);
    if (w.inc && any_found) {
        const int32_t tile = act ? jp.y >> 5 : -1;
        uint32_t fb = q >= 0 ? 1u << (jp.y & 31) : 0u;
        uint32_t pb = pos ? fb : 0u;
        const bool several = (any_found & (any_found - 1u)) != 0u;
        if (several) {
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t tt = __shfl_down_sync(FULL_MASK, tile, o);
                const uint32_t f2 = __shfl_down_sync(FULL_MASK, fb, o);
                const uint32_t p2 = __shfl_down_sync(FULL_MASK, pb, o);
                if (tt == tile) {  // (past lane 31: the lane's own bits)
                    fb |= f2;
                    pb |= p2;
                }
            }
        }
        const int32_t before = __shfl_up_sync(FULL_MASK, tile, 1);
        if (fb && (!several || lane == 0 || before != tile)) {
            atomicOr(w.foundbits + tile, fb);
            if (pb)
                atomicOr(w.posbits + tile, pb);
        }
    }
    if (any_pos) {
        long long gk = pos ? gbits(gg) : 0ll;
        int best_lane = lane;
        int32_t best_p = jp.y;
        const bool several = (any_pos & (any_pos - 1u)) != 0u;
        if (several) {
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t jj = __shfl_down_sync(FULL_MASK, jp.x, o);
                const long long g2 = __shfl_down_sync(FULL_MASK, gk, o);
                const int l2 = __shfl_down_sync(FULL_MASK, best_lane, o);
                const int32_t p2 = __shfl_down_sync(FULL_MASK, best_p, o);
                // larger gain, then lower position
                if (jj == jp.x && (g2 > gk || (g2 == gk && p2 < best_p))) {
                    gk = g2;
                    best_lane = l2;
                    best_p = p2;
                }
            }
        }
        const int32_t before = __shfl_up_sync(FULL_MASK, jp.x, 1);
        Rec r;
        r.g = __longlong_as_double(gk);
        r.p = best_p;
        r.q = __shfl_sync(FULL_MASK, q, best_lane);
        if (gk > 0ll && (!several || lane == 0 || before != jp.x)) {
            const int32_t j = jp.x;
            rec_combine(w.best + j, r, ctl);
            atomicOr(w.winbits + (j >> 5), 1u << (j & 31));
        }
    }
    return (q >= 0 ? 1u : 0u) | (pos ? 2u : 0u);
}

// The same out of line, for the searches that spend most of their time
// elsewhere: with a copy at each place of use their warps wait for
// instructions (the incremental search of a 27-point stencil of 96^3: 318 us
// inlined, 267 us with one copy; the full search of the R-MAT graph of scale
// 22 is the other way round, 280 us inlined, 351 us with one copy).
template <int kLookup>
__device__ __noinline__ unsigned resolve_lookups(const Work *__restrict__ W, const int2 *qim,
                                                 const int2 *qjp, int head, int k)
{
    return resolve_inline<kLookup>(W, qim, qjp, head, k);
}

// One warp per tile of kTile consecutive nonzeros (lane = one nonzero).
// The lane's column comes from the tile's first column and its word of the
// column-start bitmap (one popcount).  Lane with nonzero p = (i, j): if
// i > m_j it is an A-request (Algorithm 3); the closing entry (m_j, m_i) is
// looked up in column m_i (Algorithm 4): the row record of i gives that
// column's range and signature, so a clear signature bit settles "absent" at
// once; otherwise the request is queued and resolved with 31 others (see
// resolve_lookups).  Step-C records (Algorithm 5) are combined by a 128-bit
// compare-and-swap; `best` must be zero on entry: only positive records are
// written.  In a batched solve, tiles of finished matrices are skipped.
// Block size of the search kernels (each warp has its own lookup queue):
// 512 threads for a single problem, 256 for a batched solve.  With the grid
// one wave of resident blocks, the single problem's search measured a little
// faster with larger blocks on an R-MAT graph of scale 22 (0.267 ms per
// launch at 512 threads, 0.270 at 256, 0.271 at 128), a batch of 4,096 small
// matrices slower (21.4 ms per batch at 512, 20.0 at 256).  The minimum blocks per SM below are given
// in warps per SM, divided by the block's warps.
#ifndef AWPM_SEARCH_THREADS
#define AWPM_SEARCH_THREADS 512
#endif
template <bool kBatch>
struct SearchBlock {
    static constexpr int kThreads = kBatch ? 256 : AWPM_SEARCH_THREADS;
    static constexpr int kWarps = kThreads / 32;
};
#ifndef AWPM_SEARCH_MINB_WIDE
#define AWPM_SEARCH_MINB_WIDE (32 / SearchBlock<kBatch>::kWarps)
#endif
template <int kLookup, bool kBatch, bool kWide>
__global__ void __launch_bounds__(SearchBlock<kBatch>::kThreads,
                                  kWide ? AWPM_SEARCH_MINB_WIDE : 48 / SearchBlock<kBatch>::kWarps)
    k_search(const Work *__restrict__ W)
{
    __shared__ int s_go;
    __shared__ LookupQueue s_queue[SearchBlock<kBatch>::kWarps];
    if (threadIdx.x == 0)
        s_go = gate(W->ctl) ? 1 : 0;
    __syncthreads();
    const int32_t nnz = W->nnz;
    const int32_t ntiles = W->ntiles;
    const int32_t *__restrict__ rowidx = W->rowidx;
    const int32_t *__restrict__ tile_col = W->tile_col;
    const uint32_t *__restrict__ starts = W->starts;
    const int32_t *__restrict__ mc = W->mc;
    const unsigned long long *__restrict__ rsig = W->rsig;
    const RowRange *__restrict__ rrange = W->rrange;
    const unsigned long long *__restrict__ rowsig = W->rowsig;
    Ctl *ctl = W->ctl;
    const int32_t *__restrict__ tilemat = W->bw.tilemat;
    const int32_t *__restrict__ colmat = W->bw.colmat;
    const int32_t *__restrict__ mdone = W->bw.mdone;
    LookupQueue &qu = s_queue[threadIdx.x >> 5];

    const int lane = threadIdx.x & 31;
    const unsigned lanes_below = (1u << lane) - 1u;
    const int64_t nwarps = gstride() >> 5;
    const unsigned long long pol = policy_evict_last();
    // per-thread counts fit 32 bits (one nonzero per tile a warp visits)
    uint32_t n_cand = 0, n_found = 0, n_pos = 0;
    int qhead = 0, qn = 0;  // the warp's queue (warp-uniform)

    auto flush = [&](int k) {
        __syncwarp();
        const unsigned got = resolve_lookups<kLookup>(W, qu.im, qu.jp, qhead, k);
        n_found += got & 1u;
        n_pos += got >> 1;
        __syncwarp();
        qhead = (qhead + k) & (kQueue - 1);
        qn -= k;
    };
    // Each round a warp takes kU tiles (t, t + nwarps, ...) and issues their
    // loads side by side, so the dependent chains (m_j, then the row record)
    // of the kU tiles overlap; the tiles of the next round have their first
    // column, start bits and row indices loaded (prefetched) meanwhile.
    constexpr int kU = kWide ? 4 : 1;
    // a batched solve walks the list of the running matrices' tiles (built
    // after every pass); a single solve walks every tile
    const int64_t steps = kBatch ? (int64_t)*W->bw.tlist_n : (int64_t)ntiles;
    const int32_t *__restrict__ tlist = W->bw.tlist;
    int64_t t = s_go ? (gtid() >> 5) : steps;
    int32_t pf_c0[kU], pf_i[kU], pf_t[kU];
    uint32_t pf_mask[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
        const int64_t xu = t + u * nwarps;
        pf_c0[u] = 0;
        pf_i[u] = 0;
        pf_mask[u] = 1u;
        pf_t[u] = 0;
        if (xu < steps) {
            const int64_t tu = kBatch ? (int64_t)__ldg(tlist + xu) : xu;
            if (kBatch)
                pf_t[u] = (int32_t)tu;
            pf_c0[u] = __ldg(tile_col + tu);
            pf_mask[u] = __ldg(starts + tu);
            const int32_t pp = (int32_t)(tu * kTile) + lane;
            pf_i[u] = pp < nnz ? __ldcs(rowidx + pp) : 0;
        }
    }
    for (;;) {
        const bool more = t < steps;
        if (more) {
            int32_t c0[kU], iv[kU], jv[kU], mjv[kU], pv[kU];
            uint32_t mask[kU];
            bool valid[kU], mixed[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int64_t xu = t + u * nwarps;
                const int64_t tu = kBatch ? (int64_t)pf_t[u] : xu;
                pv[u] = (int32_t)(tu * kTile) + lane;
                valid[u] = xu < steps && pv[u] < nnz;
                mixed[u] = false;
                c0[u] = pf_c0[u];
                mask[u] = pf_mask[u];
                iv[u] = pf_i[u];
                if (kBatch && xu < steps) {
                    const int32_t tm = __ldg(tilemat + tu);
                    if (tm & kTileSingle) {
                        if (__ldg(mdone + (tm & ~kTileSingle)))
                            valid[u] = false;
                    } else {
                        mixed[u] = true;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int64_t xn = t + (kU + u) * nwarps;
                if (xn < steps) {
                    const int64_t tn = kBatch ? (int64_t)__ldg(tlist + xn) : xn;
                    if (kBatch)
                        pf_t[u] = (int32_t)tn;
                    pf_c0[u] = __ldg(tile_col + tn);
                    pf_mask[u] = __ldg(starts + tn);
                    const int32_t pn = (int32_t)(tn * kTile) + lane;
                    pf_i[u] = pn < nnz ? __ldcs(rowidx + pn) : 0;
                }
            }
            if (kBatch) {
                // every tile of the round belongs to finished matrices: on
                // to the next round (its loads are already in flight)
                bool any = false;
#pragma unroll
                for (int u = 0; u < kU; ++u)
                    any |= valid[u];
                if (!__any_sync(FULL_MASK, any)) {
                    t += kU * nwarps;
                    continue;
                }
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                iv[u] = valid[u] ? iv[u] : 0;
                jv[u] = valid[u] ? lane_column(c0[u], mask[u], lane) : -1 - lane;
                if (valid[u] && !(AWPM_IN(ctl, jv[u], W->n) && AWPM_IN(ctl, iv[u], W->n))) {
                    valid[u] = false;
                    jv[u] = -1 - lane;
                }
                mjv[u] = valid[u] ? ld_i32_last(mc + jv[u], pol) : 0x7fffffff;
            }
            unsigned long long sig[kU], mark[kU];
            int32_t cs[kU];  // row marking: first position of column m_i
            bool cand[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                if (kBatch && mixed[u] && valid[u] && __ldg(mdone + __ldg(colmat + jv[u])))
                    mjv[u] = 0x7fffffff;  // finished matrix: no candidate
                cand[u] = valid[u] && iv[u] > mjv[u];
                sig[u] = 0ull;
                mark[u] = 0ull;
                cs[u] = 0;
                if (cand[u]) {
                    ++n_cand;
                    sig[u] = ld_u64_last(rsig + iv[u], pol);
                    if (kLookup == AWPM_LOOKUP_ROWMARK) {
                        cs[u] = __ldg(&rrange[iv[u]].s);
                        mark[u] = __ldg(rowsig + mjv[u]);  // the mark of row m_j
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                // row m_j in column m_i's signature; with row marking also
                // column m_i (first position rg.x) marked by row m_j
                const bool pass = cand[u] && sig_has(sig[u], mjv[u]) &&
                                  (kLookup != AWPM_LOOKUP_ROWMARK || sig_has(mark[u], cs[u]));
                const unsigned need = __ballot_sync(FULL_MASK, pass);
                if (pass) {
                    const int x = (qhead + qn + __popc(need & lanes_below)) & (kQueue - 1);
                    qu.im[x] = make_int2(iv[u], mjv[u]);
                    qu.jp[x] = make_int2(jv[u], pv[u]);
                }
                qn += __popc(need);
                if (qn >= 32)
                    flush(32);
            }
            t += kU * nwarps;
        }
        if (!more && qn > 0)
            flush(qn);
        if (!more)
            break;
    }
    block_add_u64((unsigned long long)n_cand, &ctl->candidates);
    block_add_u64((unsigned long long)n_found, &ctl->found);
    block_add_u64((unsigned long long)n_pos, &ctl->positive);
}

// Pipelined form of the single-problem search (the same work and results as
// k_search<kLookup, false, ...>).  A warp's tiles are taken kU at a time
// (tiles t, t + nwarps, ...), and each round advances four stages at once,
// each on loads issued one round earlier: the signature test of one round,
// the candidate test (i > m_j) and signature loads of the next, the lanes'
// columns and the loads of m_j of the one after, the tile loads (first
// column, start bits, row indices) of the one after that.  So the two
// dependent gathers of a nonzero (m_j, then the signature of its row's
// column) are each hidden behind a round of other work.  Three slot sets
// carry a round's tiles through the stages; the loop body is written out
// three times with the slots' roles rotated, so no value is copied from one
// stage's registers to the next.  Tile loads take the tile index clamped to
// ntiles (always in bounds) and a lane is valid exactly when its position, of
// the clamped tile (see tile_pos), is below nnz; a lane's request goes to its queue slot, or to a discard slot
// of its own when it does not pass, so the stores need no branch.  All tile
// arithmetic is 32-bit (ntiles < 2^26).
#ifndef AWPM_PIPE_U_WIDE
#define AWPM_PIPE_U_WIDE 2
#endif
#ifndef AWPM_PIPE_U_NARROW
#define AWPM_PIPE_U_NARROW 1
#endif
#ifndef AWPM_PIPE_WARPS_WIDE
#define AWPM_PIPE_WARPS_WIDE 32
#endif
#ifndef AWPM_PIPE_WARPS_NARROW
#define AWPM_PIPE_WARPS_NARROW 40
#endif
template <bool kWide>
struct PipeCfg {
    static constexpr int kU = kWide ? AWPM_PIPE_U_WIDE : AWPM_PIPE_U_NARROW;
    // resident warps per SM aimed at (the launch bound divides by the block's warps)
    static constexpr int kWarpsPerSM = kWide ? AWPM_PIPE_WARPS_WIDE : AWPM_PIPE_WARPS_NARROW;
};

// The lookup queue with a discard slot per lane after the 64 ring slots.
constexpr int kQueueDiscard = kQueue + 32;
struct LookupQueueD {
    int2 im[kQueueDiscard];
    int2 jp[kQueueDiscard];
};

template <int kLookup, bool kWide, bool kBatch>
__global__ void __launch_bounds__(SearchBlock<kBatch>::kThreads,
                                  PipeCfg<kWide>::kWarpsPerSM / SearchBlock<kBatch>::kWarps)
    k_search_pipe(const Work *__restrict__ W)
{
    constexpr int kU = PipeCfg<kWide>::kU;
    __shared__ int s_go;
    __shared__ LookupQueueD s_queue[SearchBlock<kBatch>::kWarps];
    if (threadIdx.x == 0)
        s_go = gate(W->ctl) ? 1 : 0;
    __syncthreads();
    const int32_t nnz = W->nnz;
    const int32_t ntiles = W->ntiles;
    const int32_t *__restrict__ rowidx = W->rowidx;
    const int32_t *__restrict__ tile_col = W->tile_col;
    const uint32_t *__restrict__ starts = W->starts;
    const int32_t *__restrict__ mc = W->mc;
    const unsigned long long *__restrict__ rsig = W->rsig;
    const RowRange *__restrict__ rrange = W->rrange;
    const unsigned long long *__restrict__ rowsig = W->rowsig;
    Ctl *ctl = W->ctl;
    LookupQueueD &qd = s_queue[threadIdx.x >> 5];
    // a batched solve walks the list of the running matrices' tiles
    const int32_t steps = kBatch ? *W->bw.tlist_n : ntiles;
    const int32_t *__restrict__ tlist = W->bw.tlist;
    const int32_t *__restrict__ tilemat = W->bw.tilemat;
    const int32_t *__restrict__ colmat = W->bw.colmat;
    const int32_t *__restrict__ mdone = W->bw.mdone;

    const int lane = threadIdx.x & 31;
    const unsigned lanes_below = (1u << lane) - 1u;
    const int32_t nwarps = (int32_t)(gstride() >> 5);
    const int32_t stride = kU * nwarps;
    const unsigned long long pol = policy_evict_last();
    uint32_t n_cand = 0, n_found = 0, n_pos = 0;
    int qhead = 0, qn = 0;  // the warp's queue (warp-uniform)

    auto flush = [&](int k) {
        __syncwarp();
        const unsigned got = resolve_inline<kLookup>(W, qd.im, qd.jp, qhead, k);
        n_found += got & 1u;
        n_pos += got >> 1;
        __syncwarp();
        qhead = (qhead + k) & (kQueue - 1);
        qn -= k;
    };

    // slot set s, tile u: row i, column (the tile's first column before the
    // column step), start bits then m_j, the signature, the candidate flag
    int32_t si[3][kU], sj[3][kU], sx[3][kU];
    int32_t stile[3][kU];  // batched solve: the tile of the walk's entry
    unsigned long long ssig[3][kU], smark[3][kU];
    int32_t scs[3][kU];
    bool scand[3][kU];

    // stage 1: tile loads of the round starting at tile tr into slot s
    auto st_load = [&](int s, int32_t tr) {
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int32_t xu = tr + u * nwarps;
            const int32_t tu = kBatch ? (xu < steps ? __ldg(tlist + xu) : ntiles) : xu;
            if (kBatch)
                stile[s][u] = tu;
            const int32_t tl = tu < ntiles ? tu : ntiles;  // in bounds
            sj[s][u] = __ldg(tile_col + tl);
            sx[s][u] = (int32_t)__ldg(starts + tl);
            const int32_t p = tl * kTile + lane;
            si[s][u] = p < nnz ? __ldcs(rowidx + p) : 0;
        }
    };
    // stage 2: columns, and the loads of m_j
    auto st_cols = [&](int s, int32_t tr) {
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int32_t tu = kBatch ? stile[s][u] : tr + u * nwarps;
            bool valid = tile_pos(tu, ntiles, lane) < nnz;
            const int32_t j = lane_column(sj[s][u], (uint32_t)sx[s][u], lane);
            if (kBatch && valid) {
                // lanes of finished matrices take no part
                const int32_t tm = __ldg(tilemat + tu);
                valid = (tm & kTileSingle) ? !__ldg(mdone + (tm & ~kTileSingle))
                                           : !__ldg(mdone + __ldg(colmat + j));
            }
            const bool ok = valid && AWPM_IN(ctl, j, W->n) && AWPM_IN(ctl, si[s][u], W->n);
            sj[s][u] = ok ? j : -1;
            sx[s][u] = ok ? ld_i32_last(mc + j, pol) : 0x7fffffff;
        }
    };
    // stage 3: candidate test, and the signature loads
    auto st_cand = [&](int s) {
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            bool c = sj[s][u] >= 0 && si[s][u] > sx[s][u];
            if (c && !AWPM_IN(ctl, sx[s][u], W->n))
                c = false;
            scand[s][u] = c;
            ssig[s][u] = 0ull;
            if (c) {
                ++n_cand;
                ssig[s][u] = ld_u64_last(rsig + si[s][u], pol);
                if (kLookup == AWPM_LOOKUP_ROWMARK) {
                    scs[s][u] = __ldg(&rrange[si[s][u]].s);
                    smark[s][u] = __ldg(rowsig + sx[s][u]);
                }
            }
        }
    };
    // stage 4: signature test, passing requests queued
    auto st_test = [&](int s, int32_t tr) {
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const bool pass = scand[s][u] && sig_has(ssig[s][u], sx[s][u]) &&
                              (kLookup != AWPM_LOOKUP_ROWMARK ||
                               sig_has(smark[s][u], scs[s][u]));
            const unsigned need = __ballot_sync(FULL_MASK, pass);
            const int x = pass ? ((qhead + qn + __popc(need & lanes_below)) & (kQueue - 1))
                               : kQueue + lane;
            qd.im[x] = make_int2(si[s][u], sx[s][u]);
            // (past the last tile no lane passes: that position is discarded)
            const uint32_t tu = (uint32_t)(kBatch ? stile[s][u] : tr + u * nwarps);
            qd.jp[x] = make_int2(sj[s][u], (int32_t)(tu * kTile + (uint32_t)lane));
            qn += __popc(need);
            if (qn >= 32)
                flush(32);
        }
    };

    const int32_t t0 = s_go ? (int32_t)(gtid() >> 5) : steps;
#pragma unroll
    for (int s = 0; s < 3; ++s)
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            scand[s][u] = false;
            ssig[s][u] = smark[s][u] = 0ull;
            scs[s][u] = 0;
        }
    // prologue: round t0 through stage 3, round t0 + stride through stage 2,
    // round t0 + 2 stride through stage 1
    st_load(0, t0);
    st_cols(0, t0);
    st_load(1, t0 + stride);
    st_cand(0);
    st_cols(1, t0 + stride);
    st_load(2, t0 + 2 * stride);
    // steady state: each step tests round tr, requests round tr + stride's
    // signatures, makes round tr + 2 stride's columns, loads round tr + 3 stride
#define AWPM_ROT_STEP(A, B, C)                                                      \
    {                                                                               \
        if (tr >= steps)                                                            \
            break;                                                                  \
        st_test(A, tr);                                                             \
        st_cand(B);                                                                 \
        st_cols(C, tr + 2 * stride);                                                \
        st_load(A, tr + 3 * stride);                                                \
        tr += stride;                                                               \
    }
    for (int32_t tr = t0;;) {
        AWPM_ROT_STEP(0, 1, 2)
        AWPM_ROT_STEP(1, 2, 0)
        AWPM_ROT_STEP(2, 0, 1)
    }
#undef AWPM_ROT_STEP
    if (qn > 0)
        flush(qn);
    block_add_u64((unsigned long long)n_cand, &ctl->candidates);
    block_add_u64((unsigned long long)n_found, &ctl->found);
    block_add_u64((unsigned long long)n_pos, &ctl->positive);
}

// The search of a pass after the first.  An entry (i, j) evaluates to the same
// outcome as in the pass before unless the last flips changed the mate of row
// i or of column j, so this search streams the row indices and evaluates
//   - the entries whose row is in the bitmap of changed rows (folded, in
//     shared memory: a false positive only evaluates an entry again),
//   - every entry of a column whose mate changed, and
//   - of a column whose Step-C record had to go because its row's mate
//     changed, the entries that had a positive gain (no other unchanged entry
//     can give the column's maximum).
// Everything else stands: a column's record is emptied by the flip in just
// those two cases, and otherwise the maximum over the entries evaluated again
// joins it.  The pass's counts are the last pass's plus the differences: two
// bits per entry keep what it counted for.
//
// A warp takes chunks of up to eight consecutive tiles (fewer when there are
// not enough tiles to go round).  The tiles of marked columns are in a bitmap
// of their own, so a chunk without a changed row or a marked tile costs its
// row loads, one shared-memory word per entry and a vote.  Entries to evaluate
// are queued per warp and taken 32 at a time, all lanes busy: the candidate
// and signature tests, then the lookups as in the full search.  Bound by the
// row stream and the shared-memory reads of the scan when little is affected,
// by the lookups' latency and their random DRAM sectors when much is.
// Measured against whole searches: R-MAT graph of scale 22, 264 us per pass,
// now 286 for the first and 83 on average for the four after it; the 27-point
// stencil of 96^3, 33 passes, 14.05 ms per solve, now 6.37 (6.57 when every
// tile of an affected chunk was looked at).
struct IncQueue {
    int2 ij[kQueue];     // row i; column j, with the sign bit set when j is searched whole
    int32_t p[kQueue];   // position of (i, j)
    LookupQueue look;
};

template <bool kLarge>
struct IncBlock {
    static constexpr int kThreads = kLarge ? 1024 : 512;
    static constexpr int kWarps = kThreads / 32;
    static constexpr unsigned kSmem =
        kWarps * sizeof(IncQueue) + (kLarge ? kMapLargeBits : kMapSmallBits) / 8;
};

template <int kLookup, bool kLarge>
__global__ void __launch_bounds__(IncBlock<kLarge>::kThreads, kLarge ? 1 : 2)
    k_search_inc(const Work *__restrict__ W)
{
    extern __shared__ __align__(16) unsigned char s_raw[];
    __shared__ int s_go;
    constexpr int kT = 8;
    uint32_t *s_map = reinterpret_cast<uint32_t *>(s_raw);
    const Work &w = *W;
    Ctl *ctl = w.ctl;
    if (threadIdx.x == 0)
        s_go = gate(ctl) ? 1 : 0;
    __syncthreads();
    if (!s_go)
        return;
    const int set = (ctl->iterations - 1) & 1;
    // the bitmap of changed rows
    const bool use_large = kLarge && ctl->last_flips > kSmallFlips;
    const int32_t bits = use_large ? w.map_bits : kMapSmallBits;
    {
        const uint4 *src = reinterpret_cast<const uint4 *>(use_large ? w.map_large[set]
                                                                     : w.map_small[set]);
        for (int x = threadIdx.x; x < bits / 128; x += IncBlock<kLarge>::kThreads)
            reinterpret_cast<uint4 *>(s_map)[x] = __ldcg(src + x);
    }
    const uint32_t fold = (uint32_t)bits - 1u;
    IncQueue &q1 = *reinterpret_cast<IncQueue *>(
        s_raw + (kLarge ? kMapLargeBits : kMapSmallBits) / 8 + (threadIdx.x >> 5) * sizeof(IncQueue));
    LookupQueue &q2 = q1.look;
    __syncthreads();

    [[maybe_unused]] const int32_t n = w.n;
    const int32_t nnz = w.nnz, ntiles = w.ntiles;
    const int32_t *__restrict__ rowidx = w.rowidx;
    const int32_t *__restrict__ mc = w.mc;
    const int32_t *__restrict__ mc_old = w.mc_old;
    const unsigned long long *__restrict__ rsig = w.rsig;
    const uint32_t *__restrict__ colfull = w.colfull[set];
    const uint32_t *__restrict__ colpos = w.colpos[set];
    const int lane = threadIdx.x & 31;
    const unsigned lanes_below = (1u << lane) - 1u;
    const int32_t nwarps = (int32_t)(gstride() >> 5);
    const unsigned long long pol = policy_evict_last();
    int32_t n_cand = 0;
    uint32_t n_found = 0, n_pos = 0;  // differences, modulo 2^32
    int h1 = 0, c1 = 0, h2 = 0, c2 = 0;  // the warp's queues (warp-uniform)

    auto lookups = [&](int k) {
        __syncwarp();
        const unsigned got = resolve_lookups<kLookup>(W, q2.im, q2.jp, h2, k);
        n_found += got & 1u;
        n_pos += got >> 1;
        __syncwarp();
        h2 = (h2 + k) & (kQueue - 1);
        c2 -= k;
    };
    // entries h1 .. h1 + k - 1: candidate test, signature test, lookup queue
    auto evaluate = [&](int k) {
        __syncwarp();
        const int x = (h1 + lane) & (kQueue - 1);
        bool pass = false;
        int32_t i = 0, j = 0, mj = 0, p = 0;
        if (lane < k) {
            const int2 ij = q1.ij[x];
            i = ij.x;
            j = ij.y & 0x7fffffff;
            p = q1.p[x];
            if (AWPM_IN(ctl, i, n) && AWPM_IN(ctl, j, n)) {
                mj = ld_i32_last(mc + j, pol);
                const unsigned long long sig = ld_u64_last(rsig + i, pol);
                const bool cand = i > mj;
                if (ij.y < 0)  // a column searched whole may have another mate now
                    n_cand += (int)cand - (int)(i > __ldg(mc_old + j));
                pass = cand && AWPM_IN(ctl, mj, n) && sig_has(sig, mj);
                if (kLookup == AWPM_LOOKUP_ROWMARK && pass)
                    pass = sig_has(__ldg(w.rowsig + mj), __ldg(&w.rrange[i].s));
            }
        }
        const unsigned need = __ballot_sync(FULL_MASK, pass);
        if (pass) {
            const int y = (h2 + c2 + __popc(need & lanes_below)) & (kQueue - 1);
            q2.im[y] = make_int2(i, mj);
            q2.jp[y] = make_int2(j, p);
        }
        __syncwarp();
        h1 = (h1 + k) & (kQueue - 1);
        c1 -= k;
        c2 += __popc(need);
        if (c2 >= 32)
            lookups(32);
    };

    int T = 1;
    while (T < kT && ntiles >= 2 * T * nwarps)
        T *= 2;
    const int32_t step = T * nwarps;
    const uint32_t *__restrict__ tmark = w.tilemark[set];
    const uint32_t tbits = (1u << T) - 1u;
    // the row indices of the chunk's tiles (-1 past the end), and which of
    // its tiles hold marked columns
    int32_t pr[kT];
    uint32_t pmark = 0u;
    auto fetch = [&](int32_t t0) {
        pmark = (__ldg(tmark + (t0 >> 5)) >> (t0 & 31)) & tbits;
        const int32_t *src = rowidx + ((int64_t)t0 * kTile + lane);
        if (T == kT && t0 + kT < ntiles) {
#pragma unroll
            for (int u = 0; u < kT; ++u)
                pr[u] = __ldg(src + u * kTile);
        } else {
#pragma unroll
            for (int u = 0; u < kT; ++u) {
                const int32_t p = (t0 + u) * kTile + lane;
                pr[u] = u < T && t0 + u < ntiles && p < nnz ? __ldg(src + u * kTile) : -1;
            }
        }
    };
    const unsigned char *map8 = reinterpret_cast<const unsigned char *>(s_map);
    const uint32_t fold8 = fold >> 3 & ~3u;  // byte address of a row's word
    int32_t t0 = T * (int32_t)(gtid() >> 5);
    if (t0 < ntiles)
        fetch(t0);
    for (; t0 < ntiles; t0 += step) {
        const uint32_t marked = pmark;
        uint32_t hits = 0u;  // bit u: the lane's entry of tile u is in a changed row
#pragma unroll
        for (int u = 0; u < kT; ++u) {
            const uint32_t r = (uint32_t)pr[u];
            const uint32_t word = *reinterpret_cast<const uint32_t *>(map8 + ((r >> 3) & fold8));
            hits |= (__funnelshift_r(word, word, r) & 1u) << u;
        }
        // (past the end r = -1 may match: masked below)
        if (t0 + step < ntiles)
            fetch(t0 + step);
        unsigned todo = __reduce_or_sync(FULL_MASK, hits) | marked;  // tiles to look at
        if (!todo)
            continue;
        // words of the chunk's tiles, one tile per lane
        int32_t c0 = 0;
        uint32_t mask = 1u, fw = 0u, pw = 0u, cwin = 0u, pwin = 0u;
        if (lane < T && t0 + lane < ntiles) {
            c0 = __ldg(w.tile_col + t0 + lane);
            mask = __ldg(w.starts + t0 + lane);
            fw = w.foundbits[t0 + lane];
            pw = w.posbits[t0 + lane];
            if ((marked >> lane) & 1u) {
                // the 32 columns from c0 on: to be searched whole, or by
                // their entries of positive gain
                const int32_t x = c0 >> 5;
                cwin = __funnelshift_r(__ldg(colfull + x), __ldg(colfull + x + 1), c0 & 31);
                pwin = __funnelshift_r(__ldg(colpos + x), __ldg(colpos + x + 1), c0 & 31);
            }
        }
        // (rolled: the row indices are read again, from L1)
#pragma unroll 1
        while (todo) {
            const int u = __ffs(todo) - 1;
            todo &= todo - 1;
            const uint32_t mk = __shfl_sync(FULL_MASK, mask, u);
            const int32_t rank = lane_column(0, mk, lane);
            const uint32_t g = __shfl_sync(FULL_MASK, pw, u);
            bool hit = (hits >> u) & 1u, full = false;
            if ((marked >> u) & 1u) {
                full = (__shfl_sync(FULL_MASK, cwin, u) >> rank) & 1u;
                hit |= full |
                       (((__shfl_sync(FULL_MASK, pwin, u) >> rank) & (g >> lane) & 1u) != 0u);
            }
            const int32_t t = t0 + u, p = t * kTile + lane;
            hit &= t < ntiles && p < nnz;
            const unsigned m = __ballot_sync(FULL_MASK, hit);
            if (!m)
                continue;
            const int32_t j = __shfl_sync(FULL_MASK, c0, u) + rank;
            // what these entries counted for at their last evaluation
            const uint32_t f = __shfl_sync(FULL_MASK, fw, u);
            if (lane == 0 && (f & m)) {
                n_found -= __popc(f & m);
                n_pos -= __popc(g & m);
                w.foundbits[t] = f & ~m;
                w.posbits[t] = g & ~m;
            }
            if (hit) {
                const int x = (h1 + c1 + __popc(m & lanes_below)) & (kQueue - 1);
                q1.ij[x] = make_int2(__ldg(rowidx + p),
                                     full ? (int)((uint32_t)j | 0x80000000u) : j);
                q1.p[x] = p;
            }
            c1 += __popc(m);
            if (c1 >= 32)
                evaluate(32);
        }
    }
    if (c1 > 0)
        evaluate(c1);
    if (c2 > 0)
        lookups(c2);
    // (counts taken off and added: signed 32-bit per thread)
    block_add_u64((unsigned long long)(long long)n_cand, &ctl->d_candidates);
    block_add_u64((unsigned long long)(long long)(int32_t)n_found, &ctl->d_found);
    block_add_u64((unsigned long long)(long long)(int32_t)n_pos, &ctl->d_positive);
}

// ---------------------------------------------------------------------------
// Step D (Algorithm 6): conflicts, per-key selection, flip
// ---------------------------------------------------------------------------

// The epoch of the running pass's Step-D records.
__device__ __forceinline__ int32_t pass_epoch(const Work &w)
{
    return w.epoch0 + w.ctl->iterations + 1;
}

// For every Step-C winner rooted at j (a set bit of the winner bitmap) with
// second matched edge at column k = m_i: drop it if column k is itself the
// root of a Step-C winner, otherwise compete for key k (maximum gain, then
// lowest root j).  The winner's key (or its complement) is kept for the flip.
// A warp takes up to 32 bitmap words at a time and their winners 32 at a
// time, a lane per winner.
// A pass of a single problem that follows one with few flips has few winners:
// its warps take 32 bitmap words each, so that most of them find nothing to do
// (R-MAT, 40,000 columns, 640,000 entries: 209 us per solve spread always, 205
// so; with 32 words always 188, but a 27-point stencil of 30^3 takes 1,580 us
// instead of 940, for its winners).
__device__ __forceinline__ bool few_winners(const Work &w, int64_t nwarps)
{
    return w.bw.count == 0 && w.ctl->iterations > 0 &&
           w.ctl->last_flips * 4 < (unsigned long long)nwarps;
}

__global__ void k_select(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (!gate(w.ctl))
        return;
    const int lane = threadIdx.x & 31;
    const int64_t words = (int64_t)w.n / 32 + 1;
    const int64_t nwarps = gstride() >> 5;
    const int per = few_winners(w, nwarps) ? 32 : words_per_warp(words, nwarps);
    const int32_t epoch = pass_epoch(w);
    for (int64_t x0 = (gtid() >> 5) * per; x0 < words; x0 += nwarps * per) {
        for_winners(w.winbits, x0, per, words, lane, false, [&](int32_t j) {
            if (j < 0 || !AWPM_IN(w.ctl, j, w.n))
                return;
            const Rec r = w.best[j];
            if (!AWPM_IN(w.ctl, r.p, w.nnz))
                return;
            const int32_t i = __ldg(w.rowidx + r.p);
            if (!AWPM_IN(w.ctl, i, w.n))
                return;
            const int32_t k = w.mr[i];
            if (!AWPM_IN(w.ctl, k, w.n))
                return;
            if ((w.winbits[k >> 5] >> (k & 31)) & 1u) {
                w.wkey[j] = ~k;
                return;
            }
            w.wkey[j] = k;
            Sel sl;
            sl.g = r.g;
            sl.j = j;
            sl.epoch = epoch;
            sel_combine(w.dsel + k, sl, w.ctl);
        });
    }
}

// Row r has another mate now: into this pass's bitmaps of changed rows.
__device__ __forceinline__ void mark_row(const Work &w, int set, int32_t r)
{
    const uint32_t s = (uint32_t)r & (kMapSmallBits - 1);
    atomicOr(w.map_small[set] + (s >> 5), 1u << (s & 31));
    if (w.map_bits) {
        const uint32_t b = (uint32_t)r & (uint32_t)(w.map_bits - 1);
        atomicOr(w.map_large[set] + (b >> 5), 1u << (b & 31));
    }
}

// The next pass looks at the tiles of the column at positions [s, e).
__device__ __forceinline__ void mark_tiles(const Work &w, int set, int32_t s, int32_t e)
{
    const int32_t t1 = (e - 1) >> 5;
    for (int32_t t = s >> 5; t <= t1;) {
        const int32_t last = min(t1, t | 31);  // last tile of the bitmap word
        const uint32_t bits = (0xffffffffu >> (31 - (last - t))) << (t & 31);
        atomicOr(w.tilemark[set] + (t >> 5), bits);
        t = last + 1;
    }
}

// The next pass searches column j whole; `was` is the row its entries were
// last evaluated with.
__device__ __forceinline__ void mark_column(const Work &w, int set, int32_t j, int32_t was,
                                            int32_t s, int32_t e)
{
    atomicOr(w.colfull[set] + (j >> 5), 1u << (j & 31));
    w.mc_old[j] = was;
    mark_tiles(w, set, s, e);
}

// Flip every selected cycle: column j takes row i, key column k takes m_j;
// the row records of rows i and m_j follow their new mates.  The selected
// cycles are vertex-disjoint, so each lane owns its four vertices.  Winners
// are taken as in k_select; in a batched solve the flips of a round are
// counted per matrix with one atomic per matrix.
//
// The Step-C records and winner bits visited are cleared, which leaves them
// empty for the next pass -- except, with incremental passes, those of
// winners whose row i keeps its mate: their entry's outcome stands, and so
// does their column's maximum.  Row i's mate is column k; it changes exactly
// when k is flipped: as the key of the winner selected there (j lost to it),
// or as the root of the winner that dropped j, if that one was selected.
// (The greedy selection drops a winner only for sharing a column with a kept
// cycle, so all its winners' records go.)  In the graph form of a single
// problem's pass kInc says which passes these are, and a flip without
// incremental passes holds none of their code: with few winners it is short, and
// fetching its code is part of it (R-MAT, 20,000 columns, 8 passes: 276 us per
// solve with one kernel for both, 271 so).  -1 asks the descriptor: a batch's
// union, with many winners, takes 6.4 ms so and 7.0 without that code (1,024
// matrices of 200 to 20,000 columns).
template <int kInc>
__device__ __forceinline__ unsigned long long flip_body(const Work &w)
{
    unsigned long long flips = 0;
    if (gate(w.ctl)) {
        const int lane = threadIdx.x & 31;
        const int64_t words = (int64_t)w.n / 32 + 1;
        const int64_t nwarps = gstride() >> 5;
        const int per = few_winners(w, nwarps) ? 32 : words_per_warp(words, nwarps);
        const int32_t epoch = pass_epoch(w);
        const bool inc = kInc < 0 ? w.inc != 0 : kInc != 0;
        const int set = inc ? w.ctl->iterations & 1 : 0;
        auto selected = [&](int32_t key, int32_t j) {
            const Sel sl = w.dsel[key];
            return sl.epoch == epoch && sl.j == j;
        };
        for (int64_t x0 = (gtid() >> 5) * per; x0 < words; x0 += nwarps * per) {
            for_winners(w.winbits, x0, per, words, lane, true, [&](int32_t j) {
                int32_t mat = -1;  // matrix of a flipped cycle (batched solve)
                if (j >= 0 && AWPM_IN(w.ctl, j, w.n)) {
                    const Rec r = w.best[j];
                    const int32_t key = w.wkey[j];
                    const int32_t k = key >= 0 ? key : -1;
                    bool sel = false, stands = false;
                    if (k >= 0 && AWPM_IN(w.ctl, k, w.n) && AWPM_IN(w.ctl, r.p, w.nnz) &&
                        AWPM_IN(w.ctl, r.q, w.nnz)) {
                        sel = selected(k, j);
                    } else if (inc && !w.psel && key < 0 && AWPM_IN(w.ctl, ~key, w.n)) {
                        const int32_t k2 = w.wkey[~key];
                        stands = k2 < 0 || !AWPM_IN(w.ctl, k2, w.n) || !selected(k2, ~key);
                    }
                    if (stands) {
                        atomicOr(w.winbits + (j >> 5), 1u << (j & 31));
                    } else {
                        w.best[j] = Rec{0.0, 0, 0};
                        if (inc && !sel) {
                            atomicOr(w.colpos[set] + (j >> 5), 1u << (j & 31));
                            mark_tiles(w, set, w.colptr[j], w.colptr[j + 1]);
                        }
                    }
                    if (sel) {
                        const int32_t i = w.rowidx[r.p];
                        const int32_t mj = w.mc[j];
                        if (AWPM_IN(w.ctl, i, w.n) && AWPM_IN(w.ctl, mj, w.n)) {
                            const double wij = w.w[r.p];
                            const double wq = w.w[r.q];
                            w.mc[j] = i;
                            w.mr[i] = j;
                            w.mc[k] = mj;
                            w.mr[mj] = k;
                            w.wm[j] = wij;
                            w.wm[k] = wq;
                            const int32_t js = w.colptr[j], je = w.colptr[j + 1];
                            const int32_t ks = w.colptr[k], ke = w.colptr[k + 1];
                            put_rowrec(w, i, js, je, w.colsig[j], wij);
                            put_rowrec(w, mj, ks, ke, w.colsig[k], wq);
                            ++flips;
                            if (w.bw.count > 0)
                                mat = w.bw.colmat[k];
                            if (inc) {
                                mark_row(w, set, i);
                                mark_row(w, set, mj);
                                mark_column(w, set, j, mj, js, je);
                                mark_column(w, set, k, i, ks, ke);
                            }
                        }
                    }
                }
                // every lane reaches the warp-wide match: no early exit above
                if (w.bw.count > 0) {
                    const unsigned peers = __match_any_sync(FULL_MASK, mat);
                    if (mat >= 0 && (peers & ((1u << lane) - 1u)) == 0u)
                        atomicAdd(w.bw.mflips + mat, (unsigned long long)__popc(peers));
                }
            });
        }
        // the set of bitmaps that this pass's search read, for the next flips
        if (inc && w.ctl->iterations > 0)
            inc_clear(w, set ^ 1);
    }
    return flips;
}

__global__ void k_flip(const Work *__restrict__ W)
{
    const Work &w = *W;
    block_add_u64(flip_body<-1>(w), &w.ctl->pass_flips);
}

__global__ void k_control(const Work *__restrict__ W)
{
    control_step(W->ctl, W->inc != 0);
}

__global__ void k_control_graph(const Work *__restrict__ W, cudaGraphConditionalHandle h)
{
    cudaGraphSetConditional(h, control_step(W->ctl, W->inc != 0) ? 1u : 0u);
}

// The flip in the graph form of a single problem's pass: the block that
// finishes last (its count of finished blocks orders it after every other
// block's flip count) ends the pass and sets the WHILE condition.
template <int kInc>
__global__ void k_flip_graph(const Work *__restrict__ W, cudaGraphConditionalHandle h)
{
    const Work &w = *W;
    block_add_u64(flip_body<kInc>(w), &w.ctl->pass_flips);
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned prev = atomicAdd(&w.ctl->flip_done, 1u);
        if (prev == gridDim.x - 1) {
            __threadfence();
            w.ctl->flip_done = 0u;
            cudaGraphSetConditional(h, control_step(w.ctl, kInc != 0) ? 1u : 0u);
        }
    }
}

// End of a pass for every matrix still running: count the pass, stop the
// matrix when it flipped nothing or reached the cap; count the running ones.
__global__ void k_batch_control(const Work *__restrict__ W)
{
    const Work &w = *W;
    const BatchWork &bw = w.bw;
    const bool go = !w.ctl->err && w.ctl->active;
    for (int64_t b0 = (int64_t)blockIdx.x * blockDim.x; b0 < bw.count;
         b0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = b0 + threadIdx.x;
        int still = 0;
        if (go && b < bw.count && !bw.mdone[b]) {
            const unsigned long long f = bw.mflips[b];
            bw.mflips[b] = 0;
            bw.miter[b] += 1;
            bw.mcycles[b] += f;
            if (f == 0) {
                bw.mconv[b] = 1;
                bw.mdone[b] = 1;
            } else if (bw.miter[b] >= w.ctl->max_passes) {
                bw.mdone[b] = 1;
            } else {
                still = 1;
            }
        }
        still = __syncthreads_count(still);
        if (threadIdx.x == 0 && still)
            atomicAdd(bw.active, still);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0)
        *bw.tlist_n = 0;  // the list of the next pass is built after this
}

// Pass counter of the whole batch; another pass runs while any matrix runs.
__device__ __forceinline__ int batch_step(Ctl *ctl, int32_t *active)
{
    if (ctl->err || !ctl->active) {
        ctl->active = 0;
        return 0;
    }
    ctl->iterations += 1;
    const int32_t a = *active;
    *active = 0;
    ctl->cycles += ctl->pass_flips;
    ctl->pass_flips = 0;
    if (a == 0) {
        ctl->converged = 1;
        ctl->active = 0;
    }
    return ctl->active;
}

__global__ void k_batch_step(const Work *__restrict__ W)
{
    batch_step(W->ctl, W->bw.active);
}

__global__ void k_batch_step_graph(const Work *__restrict__ W, cudaGraphConditionalHandle h)
{
    cudaGraphSetConditional(h, batch_step(W->ctl, W->bw.active) ? 1u : 0u);
}

__global__ void k_export_stepc(const Work *__restrict__ W, double *gain, int32_t *row)
{
    const Work &w = *W;
    if (w.ctl->err)
        return;
    for (int64_t j = gtid(); j < w.n; j += gstride()) {
        const Rec r = w.best[j];
        const bool has = gbits(r.g) > 0ll;
        gain[j] = has ? r.g : 0.0;
        row[j] = has ? w.rowidx[r.p] : -1;
    }
}

// ---------------------------------------------------------------------------
// Greedy (Pettie-Sanders) selection of the Step-C winners (Section 4)
// ---------------------------------------------------------------------------
// Instead of Step D: the winners in order of gain, descending (equal gains:
// lower root column), each kept when its columns j and k = m_i -- hence also
// its rows m_j and i -- belong to no cycle kept before.  Computed in rounds:
// every column names the first undecided winner touching it (maximum gain,
// then lowest root, through the 128-bit compare-and-swap of the Step-D
// records); a winner named by both its columns is kept; undecided winners
// touching a kept cycle are dropped.  The first undecided winner is always
// named by both its columns, so every round decides at least one.  At the
// end the kept winners are handed to k_flip exactly as Step D hands them:
// the key column's record names the root, dropped winners get key -1.

// The kernels below take the winners of a bitmap a lane each (for_winners);
// with a thread per bitmap word, its winners one after another, a solve of a
// 27-point stencil of 64^3 spent 1.63 ms in them, with a lane each 1.23 ms (by
// the launch list; most of that launches that find few winners).
template <typename F>
__device__ __forceinline__ void for_all_winners(const Work &w, uint32_t *bits, F f)
{
    const int64_t words = (int64_t)w.n / 32 + 1;
    const int64_t nwarps = gstride() >> 5;
    const int per = words_per_warp(words, nwarps);
    for (int64_t x0 = (gtid() >> 5) * per; x0 < words; x0 += nwarps * per)
        for_winners(bits, x0, per, words, threadIdx.x & 31, false, f);
}

// Keys of all winners; every winner undecided; their number into Ctl::live.
__device__ __forceinline__ int ps_begin(const Work &w)
{
    int live = 0;
    if (gate(w.ctl)) {
        const int64_t words = (int64_t)w.n / 32 + 1;
        for (int64_t x = gtid(); x < words; x += gstride())
            w.pslive[x] = w.winbits[x];
        for_all_winners(w, w.winbits, [&](int32_t j) {
            if (j < 0)
                return;
            w.wkey[j] = w.mr[w.rowidx[w.best[j].p]];
            ++live;
        });
    }
    return live;
}

__global__ void k_ps_begin(const Work *__restrict__ W)
{
    // (a selection done by k_ps_small leaves nothing to decide)
    const int live = W->ctl->ps_done ? 0 : ps_begin(*W);
    warp_add_i32(live, &W->ctl->live);
}

// Loop condition of the rounds: undecided winners remain (counter reset).
__global__ void k_ps_cond(const Work *__restrict__ W, cudaGraphConditionalHandle h)
{
    Ctl *c = W->ctl;
    const int32_t live = c->live;
    c->live = 0;
    cudaGraphSetConditional(h, (live > 0 && c->err == 0u && c->active) ? 1u : 0u);
}

// Round, step 1: every undecided winner names itself at both its columns.
__device__ __forceinline__ void ps_name(const Work &w)
{
    if (!gate(w.ctl))
        return;
    for_all_winners(w, w.pslive, [&](int32_t j) {
        if (j < 0)
            return;
        const Sel s{w.best[j].g, j, 0};
        sel_combine(w.psel + j, s, w.ctl);
        sel_combine(w.psel + w.wkey[j], s, w.ctl);
    });
}

// Round, step 2: a winner named by both its columns is kept; its columns
// are marked used.
__device__ __forceinline__ void ps_take(const Work &w)
{
    if (!gate(w.ctl))
        return;
    for_all_winners(w, w.pslive, [&](int32_t j) {
        if (j < 0)
            return;
        const int32_t k = w.wkey[j];
        const Sel a = w.psel[j], c = w.psel[k];
        if (gbits(a.g) > 0ll && a.j == j && gbits(c.g) > 0ll && c.j == j) {
            atomicOr(w.pstaken + (j >> 5), 1u << (j & 31));
            atomicOr(w.psused + (j >> 5), 1u << (j & 31));
            atomicOr(w.psused + (k >> 5), 1u << (k & 31));
        }
    });
}

// Round, step 3: clear the records this round touched; drop the undecided
// winners that touch a used column; count the undecided ones left.
__device__ __forceinline__ int ps_prune(const Work &w)
{
    int live = 0;
    if (gate(w.ctl)) {
        for_all_winners(w, w.pslive, [&](int32_t j) {
            if (j < 0)
                return;
            const int32_t k = w.wkey[j];
            w.psel[j] = Sel{0.0, 0, 0};
            w.psel[k] = Sel{0.0, 0, 0};
            // (a kept winner's columns are used too)
            const bool used = ((w.psused[j >> 5] >> (j & 31)) & 1u) ||
                              ((w.psused[k >> 5] >> (k & 31)) & 1u);
            if (used)
                atomicAnd(w.pslive + (j >> 5), ~(1u << (j & 31)));
            else
                ++live;
        });
    }
    return live;
}

__global__ void k_ps_name(const Work *__restrict__ W)
{
    ps_name(*W);
}

__global__ void k_ps_take(const Work *__restrict__ W)
{
    ps_take(*W);
}

__global__ void k_ps_prune(const Work *__restrict__ W)
{
    const int live = ps_prune(*W);
    warp_add_i32(live, &W->ctl->live);
}

// After the rounds: kept winners get their key column's record (the form
// k_flip reads), dropped ones key -1; the kept-set and used-column bitmaps
// are cleared for the next pass.
__device__ __forceinline__ void ps_end(const Work &w)
{
    if (!gate(w.ctl))
        return;
    const int32_t epoch = pass_epoch(w);
    for_all_winners(w, w.winbits, [&](int32_t j) {
        if (j < 0)
            return;
        const int32_t k = w.wkey[j];
        if ((w.pstaken[j >> 5] >> (j & 31)) & 1u) {
            w.dsel[k] = Sel{w.best[j].g, j, epoch};
            atomicAnd(w.pstaken + (j >> 5), ~(1u << (j & 31)));
            atomicAnd(w.psused + (j >> 5), ~(1u << (j & 31)));
            atomicAnd(w.psused + (k >> 5), ~(1u << (k & 31)));
        } else {
            w.wkey[j] = -1;
        }
    });
}

__global__ void k_ps_end(const Work *__restrict__ W)
{
    if (!W->ctl->ps_done)
        ps_end(*W);
}

// The whole selection of a pass with few winners in one cluster of blocks, with
// cluster barriers between the steps (otherwise five launches or more, each
// longer than its work).  With more winners it leaves the pass to the kernels
// above.  Most passes have few: of the 17 of a 27-point stencil of 64^3, ten
// have less than kPsSmall.
constexpr int kPsSmall = 8192;
__global__ void __cluster_dims__(8, 1, 1) __launch_bounds__(1024)
    k_ps_small(const Work *__restrict__ W)
{
    const Work &w = *W;
    Ctl *c = w.ctl;
    // (counted by the blocks' own sums, so that every block decides alike)
    int mine = 0;
    if (gate(c))
        for (int64_t x = gtid(); x < (int64_t)w.n / 32 + 1; x += gstride())
            mine += __popc(w.winbits[x]);
    if (gtid() == 0) {
        c->ps_done = 0;
        c->ps_count = 0;
    }
    cluster_sync();
    warp_add_i32(mine, &c->ps_count);
    cluster_sync();
    const int32_t count = *(volatile int32_t *)&c->ps_count;
    if (count == 0 || count > kPsSmall)
        return;
    ps_begin(w);
    cluster_sync();
    for (int round = 0;; ++round) {
        ps_name(w);
        cluster_sync();
        ps_take(w);
        cluster_sync();
        const int live = ps_prune(w);
        if (gtid() == 0)
            c->ps_count = 0;
        cluster_sync();
        warp_add_i32(live, &c->ps_count);
        cluster_sync();
        if (*(volatile int32_t *)&c->ps_count == 0)
            break;
        if (round > kPsSmall) {  // (every round decides a winner)
            if (gtid() == 0)
                raise_err(c, kErrTimeout);
            break;
        }
        cluster_sync();  // (read by all before it is emptied again)
    }
    ps_end(w);
    if (gtid() == 0)
        c->ps_done = 1;
}

// ---------------------------------------------------------------------------
// Entry checks of the greedy and the maximum matching: row range, sortedness,
// finite weights
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads) k_gm_check(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (w.ctl->err & kErrInvalid)
        return;
    // four tiles per round, their loads side by side
    constexpr int kU = 4;
    const int lane = threadIdx.x & 31;
    const int32_t nwarps = (int32_t)(gstride() >> 5);
    unsigned bits = 0;
    for (int32_t t0 = (int32_t)(gtid() >> 5); t0 < w.ntiles; t0 += kU * nwarps) {
        int32_t r[kU], prev[kU];
        uint32_t mask[kU];
        int x[kU];  // upper words of the weights
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int32_t t = t0 + u * nwarps;
            const int32_t p = t < w.ntiles ? t * kTile + lane : w.nnz;
            const bool valid = p < w.nnz;
            mask[u] = t < w.ntiles ? __ldg(w.starts + t) : 1u;
            r[u] = valid ? __ldcs(w.rowidx + p) : 0;
            x[u] = valid ? __double2hiint(__ldcs(w.w + p)) : 0;
            prev[u] = valid && lane == 0 && p > 0 ? __ldg(w.rowidx + p - 1) : 0;
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int32_t t = t0 + u * nwarps;
            const int32_t p = t < w.ntiles ? t * kTile + lane : w.nnz;
            const int32_t up = __shfl_up_sync(FULL_MASK, r[u], 1);
            const int32_t before = lane == 0 ? prev[u] : up;
            if (p < w.nnz) {
                if (r[u] < 0 || r[u] >= w.n)
                    bits |= kErrInvalid;
                if ((x[u] & 0x7ff00000) == 0x7ff00000)
                    bits |= kErrNonfinite;
                if (p > 0 && !((mask[u] >> lane) & 1u) && before >= r[u])
                    bits |= kErrUnsorted;
            }
        }
    }
    bits = __reduce_or_sync(FULL_MASK, bits);
    if (lane == 0 && bits)
        raise_err(w.ctl, bits);
}

// ---------------------------------------------------------------------------
// launchers: fixed grids (a multiple of the SM count)
// ---------------------------------------------------------------------------

static inline unsigned util_grid(const Shape &sh)
{
    return (unsigned)(sh.num_sms * 4);
}

static inline unsigned tile_grid(const Shape &sh)
{
    return (unsigned)(sh.num_sms * 8);
}

// The one-off initialisation kernels are chains of dependent loads per
// column (or per tile); wider grids keep more of them in flight.
static inline unsigned init_grid(const Shape &sh)
{
    return (unsigned)(sh.num_sms * 16);
}

static inline unsigned init_tile_grid(const Shape &sh)
{
    return (unsigned)(sh.num_sms * 32);
}

// The mate initialisation, which leaves one partial sum per block in wpart:
// its resident blocks (80 registers: three blocks of 256 per SM), at most
// kWsumBlocks.
#ifndef AWPM_SUM_BPS
#define AWPM_SUM_BPS 3
#endif
static inline unsigned sum_grid(const Shape &sh)
{
    const int g = sh.num_sms * AWPM_SUM_BPS;
    return (unsigned)(g < kWsumBlocks ? g : kWsumBlocks);
}

void Sink::launch(const void *func, unsigned grid, unsigned block, void **args, unsigned smem)
{
    if (err != cudaSuccess)
        return;
    if (graph) {
        cudaKernelNodeParams p;
        p.func = const_cast<void *>(func);
        p.gridDim = dim3(grid);
        p.blockDim = dim3(block);
        p.sharedMemBytes = smem;
        p.kernelParams = args;
        p.extra = nullptr;
        cudaGraphNode_t node;
        err = cudaGraphAddKernelNode(&node, graph, last ? &last : nullptr, last ? 1 : 0, &p);
        if (err == cudaSuccess)
            last = node;
    } else {
        err = cudaLaunchKernel(func, dim3(grid), dim3(block), args, smem, stream);
    }
}

void launch_init(const Work *d, const Shape &sh, Sink &k)
{
    void *a[] = {(void *)&d};
    k.launch((const void *)k_reset, util_grid(sh), kThreads, a);
    k.launch((const void *)k_check_mark, init_grid(sh), kThreads, a);
    k.launch((const void *)k_entries, init_tile_grid(sh), kThreads, a);
    if (sh.batch)
        k.launch((const void *)k_batch_cols, init_grid(sh), kThreads, a);
    k.launch((const void *)k_init_mates, sum_grid(sh), kThreads, a);
    k.launch((const void *)k_init_rows, init_grid(sh), kThreads, a);
    if (sh.batch) {
        k.launch((const void *)k_batch_check, init_tile_grid(sh), kThreads, a);
        k.launch((const void *)k_batch_list, init_grid(sh), kThreads, a);
    }
    if (sh.lookup == AWPM_LOOKUP_HASH)
        k.launch((const void *)k_hash_build, init_tile_grid(sh), kThreads, a);
    if (sh.lookup == AWPM_LOOKUP_ROWMARK) {
        k.launch((const void *)k_rm_marks, init_tile_grid(sh), kThreads, a);
        // four passes cover every row index; the unneeded ones return at once.
        // Grids: the resident blocks (scatter: 48 registers, 36 KB shared)
        const unsigned rs_grid = (unsigned)sh.num_sms * 8;
        const unsigned sc_grid = (unsigned)sh.num_sms * 5;
        for (int pass = 0; pass < 4; ++pass) {
            void *ap[] = {(void *)&d, (void *)&pass};
            k.launch((const void *)k_rs_hist, rs_grid, kRsThreads, ap);
            k.launch((const void *)k_rs_scan_a, rs_grid, kRsThreads, ap);
            k.launch((const void *)k_rs_scan_b, 1, kRsThreads, ap);
            k.launch((const void *)k_rs_scan_c, rs_grid, kRsThreads, ap);
            k.launch((const void *)k_rs_scatter, sc_grid, kRsThreads, ap);
        }
        k.launch((const void *)k_rm_rowptr, init_grid(sh), kThreads, a);
    }
}

// The matched weights' sum (the input matching's when !out).  The mate
// initialisation of a single solve already left its partials in wpart;
// otherwise k_wsum_partial writes them.
void launch_weight_sum(const Work *d, const Shape &sh, bool out, Sink &k)
{
    int o = out ? 1 : 0;
    const bool from_init = !out && !sh.batch;
    int parts = from_init ? (int)sum_grid(sh) : kWsumBlocks;
    void *a[] = {(void *)&d};
    void *ao[] = {(void *)&d, (void *)&o};
    void *af[] = {(void *)&d, (void *)&o, (void *)&parts};
    if (!from_init)
        k.launch(sh.greedy ? (const void *)k_wsum_partial<true>
                           : (const void *)k_wsum_partial<false>,
                 kWsumBlocks, kWsumThreads, a);
    k.launch((const void *)k_wsum_final, 1, kWsumBlocks, af);
    if (sh.batch)
        k.launch((const void *)k_batch_wsum, util_grid(sh), kThreads, ao);
}

bool search_pipe()
{
    const char *v = getenv("AWPM_SEARCH_PIPE");
    if (v && (v[0] == '0' || v[0] == '1') && v[1] == 0)
        return v[0] == '1';
    return true;
}

template <bool kWide>
static const void *search_fn(int lookup, bool batch)
{
    if (search_pipe()) {
        if (batch) {
            if (lookup == AWPM_LOOKUP_ROWMARK)
                return (const void *)k_search_pipe<AWPM_LOOKUP_ROWMARK, kWide, true>;
            if (lookup == AWPM_LOOKUP_HASH)
                return (const void *)k_search_pipe<AWPM_LOOKUP_HASH, kWide, true>;
            return (const void *)k_search_pipe<AWPM_LOOKUP_BSEARCH, kWide, true>;
        }
        if (lookup == AWPM_LOOKUP_ROWMARK)
            return (const void *)k_search_pipe<AWPM_LOOKUP_ROWMARK, kWide, false>;
        if (lookup == AWPM_LOOKUP_HASH)
            return (const void *)k_search_pipe<AWPM_LOOKUP_HASH, kWide, false>;
        return (const void *)k_search_pipe<AWPM_LOOKUP_BSEARCH, kWide, false>;
    }
    if (lookup == AWPM_LOOKUP_ROWMARK)
        return batch ? (const void *)k_search<AWPM_LOOKUP_ROWMARK, true, kWide>
                     : (const void *)k_search<AWPM_LOOKUP_ROWMARK, false, kWide>;
    if (lookup == AWPM_LOOKUP_HASH)
        return batch ? (const void *)k_search<AWPM_LOOKUP_HASH, true, kWide>
                     : (const void *)k_search<AWPM_LOOKUP_HASH, false, kWide>;
    return batch ? (const void *)k_search<AWPM_LOOKUP_BSEARCH, true, kWide>
                 : (const void *)k_search<AWPM_LOOKUP_BSEARCH, false, kWide>;
}

int search_blocks_per_sm(int lookup, bool batch, bool wide)
{
    const void *f = wide ? search_fn<true>(lookup, batch) : search_fn<false>(lookup, batch);
    const int threads = batch ? SearchBlock<true>::kThreads : SearchBlock<false>::kThreads;
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, f, threads, 0) != cudaSuccess) {
        cudaGetLastError();
        b = 1;
    }
    return b < 1 ? 1 : b;
}

bool default_search_wide()
{
    const char *v = getenv("AWPM_SEARCH_WIDE");
    if (v && (v[0] == '0' || v[0] == '1') && v[1] == 0)
        return v[0] == '1';
    return true;
}

// The search grid is one wave of resident blocks: each warp walks its tiles
// to the end (two, three, four and eight waves were measured slower on an
// R-MAT graph of scale 22: the later waves' blocks start only as whole
// blocks finish).
void launch_search(const Work *d, const Shape &sh, Sink &k)
{
    const unsigned grid = (unsigned)(sh.num_sms * (sh.search_bps > 0 ? sh.search_bps : 1));
    void *a[] = {(void *)&d};
    const void *f = sh.wide ? search_fn<true>(sh.lookup, sh.batch)
                            : search_fn<false>(sh.lookup, sh.batch);
    k.launch(f, grid, sh.batch ? SearchBlock<true>::kThreads : SearchBlock<false>::kThreads, a);
}

template <bool kLarge>
static const void *search_inc_fn(int lookup)
{
    if (lookup == AWPM_LOOKUP_ROWMARK)
        return (const void *)k_search_inc<AWPM_LOOKUP_ROWMARK, kLarge>;
    if (lookup == AWPM_LOOKUP_HASH)
        return (const void *)k_search_inc<AWPM_LOOKUP_HASH, kLarge>;
    return (const void *)k_search_inc<AWPM_LOOKUP_BSEARCH, kLarge>;
}

cudaError_t search_inc_setup()
{
    for (int lookup : {AWPM_LOOKUP_BSEARCH, AWPM_LOOKUP_HASH, AWPM_LOOKUP_ROWMARK}) {
        cudaError_t e = cudaFuncSetAttribute(search_inc_fn<true>(lookup),
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)IncBlock<true>::kSmem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(search_inc_fn<false>(lookup),
                                     cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)IncBlock<false>::kSmem);
        if (e != cudaSuccess)
            return e;
    }
    return cudaSuccess;
}

// One wave: a block of 1,024 threads per SM with the large bitmap, two of 512
// with the small one.
void launch_search_inc(const Work *d, const Shape &sh, Sink &k)
{
    void *a[] = {(void *)&d};
    if (sh.large)
        k.launch(search_inc_fn<true>(sh.lookup), (unsigned)sh.num_sms, IncBlock<true>::kThreads, a,
                 IncBlock<true>::kSmem);
    else
        k.launch(search_inc_fn<false>(sh.lookup), (unsigned)sh.num_sms * 2,
                 IncBlock<false>::kThreads, a, IncBlock<false>::kSmem);
}

int search_waves(int num_sms, int search_bps, int32_t ntiles)
{
    const int64_t warps =
        (int64_t)num_sms * (search_bps > 0 ? search_bps : 1) * SearchBlock<false>::kWarps;
    return (int64_t)ntiles >= 64 * warps ? 2 : 1;
}

void launch_greedy_select_begin(const Work *d, const Shape &sh, bool graph,
                                cudaGraphConditionalHandle h, Sink &k)
{
    void *a[] = {(void *)&d};
    void *ah[] = {(void *)&d, (void *)&h};
    k.launch((const void *)k_ps_small, 8, 1024, a);
    k.launch((const void *)k_ps_begin, tile_grid(sh), kThreads, a);
    if (graph)
        k.launch((const void *)k_ps_cond, 1, 1, ah);
}

void launch_greedy_select_round(const Work *d, const Shape &sh, bool graph,
                                cudaGraphConditionalHandle h, Sink &k)
{
    void *a[] = {(void *)&d};
    void *ah[] = {(void *)&d, (void *)&h};
    k.launch((const void *)k_ps_name, tile_grid(sh), kThreads, a);
    k.launch((const void *)k_ps_take, tile_grid(sh), kThreads, a);
    k.launch((const void *)k_ps_prune, tile_grid(sh), kThreads, a);
    if (graph)
        k.launch((const void *)k_ps_cond, 1, 1, ah);
}

void launch_greedy_select_end_and_flip(const Work *d, const Shape &sh, Sink &k)
{
    void *a[] = {(void *)&d};
    k.launch((const void *)k_ps_end, tile_grid(sh), kThreads, a);
    k.launch((const void *)k_flip, tile_grid(sh), kThreads, a);
}

// Step D's kernels take 32 words of the winner bitmap per warp; a single
// problem of the large size class (at least 64 tiles per resident search
// warp) gets four blocks per SM (one round of words covers n up to about
// 5 M), a smaller one one block per SM.  Late
// passes have few winners, so the kernels cost about their launch and a
// read of the bitmap; blocks past the bitmap's end would only add to that.
static inline unsigned winner_grid(const Shape &sh)
{
    return sh.batch ? tile_grid(sh) : (unsigned)(sh.num_sms * (sh.search_waves > 1 ? 4 : 1));
}

void launch_select_flip_control_graph(const Work *d, const Shape &sh,
                                      cudaGraphConditionalHandle h, Sink &k)
{
    void *a[] = {(void *)&d};
    void *ah[] = {(void *)&d, (void *)&h};
    k.launch((const void *)k_select, winner_grid(sh), kThreads, a);
    k.launch(sh.inc ? (const void *)k_flip_graph<1> : (const void *)k_flip_graph<0>,
             winner_grid(sh), kThreads, ah);
}

void launch_select_and_flip(const Work *d, const Shape &sh, Sink &k)
{
    void *a[] = {(void *)&d};
    k.launch((const void *)k_select, winner_grid(sh), kThreads, a);
    k.launch((const void *)k_flip, winner_grid(sh), kThreads, a);
}

void launch_control(const Work *d, const Shape &sh, bool graph, cudaGraphConditionalHandle h,
                    Sink &k)
{
    void *a[] = {(void *)&d};
    void *ah[] = {(void *)&d, (void *)&h};
    if (sh.batch) {
        k.launch((const void *)k_batch_control, util_grid(sh), kThreads, a);
        k.launch((const void *)k_batch_list, init_grid(sh), kThreads, a);
        if (graph)
            k.launch((const void *)k_batch_step_graph, 1, 1, ah);
        else
            k.launch((const void *)k_batch_step, 1, 1, a);
        return;
    }
    if (graph)
        k.launch((const void *)k_control_graph, 1, 1, ah);
    else
        k.launch((const void *)k_control, 1, 1, a);
}

void launch_check_colptr(const Work *d, const Shape &sh, Sink &k)
{
    void *a[] = {(void *)&d};
    k.launch((const void *)k_check_colptr, init_grid(sh), kThreads, a);
}

void launch_mark_starts(const Work *d, const Shape &sh, Sink &k)
{
    void *a[] = {(void *)&d};
    k.launch((const void *)k_mark_starts, init_grid(sh), kThreads, a);
}

void launch_check_entries(const Work *d, const Shape &sh, Sink &k)
{
    void *a[] = {(void *)&d};
    k.launch((const void *)k_gm_check, init_tile_grid(sh), kThreads, a);
}

void launch_check_mark(const Work *d, const Shape &sh, Sink &k)
{
    void *a[] = {(void *)&d};
    k.launch((const void *)k_check_mark, init_grid(sh), kThreads, a);
}

void launch_export_stepc(const Work *d, const Shape &sh, double *gain, int32_t *row, Sink &k)
{
    void *a[] = {(void *)&d, (void *)&gain, (void *)&row};
    k.launch((const void *)k_export_stepc, util_grid(sh), kThreads, a);
}

}  // namespace awpm

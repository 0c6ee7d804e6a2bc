// Whole solves of small matrices (sm_103a): one block per matrix, the
// matching and the columns' pointers in shared memory.
//
// Algorithm 2 of one matrix needs, per candidate entry, the mates of its row
// and column and the place of the closing entry's column: for n up to 20,096
// these fit a block's shared memory as 16- and 32-bit words.  So a block runs
// the checks, the initialisation and all passes of its matrix with block
// barriers between the steps, streams the row indices from L2, and goes to
// global memory only for what survives the filters.  Passes after the first
// evaluate only the entries that the last flips affect, as the incremental
// searches of large matrices do.  Against the passes over the union of all
// matrices this replaces, nothing is launched per pass, finished matrices cost
// nothing, and no per-column state crosses the memory system.
//
// A single small matrix gets a cluster of blocks instead of one.
//
// Bound by instruction issue (about 1,300 instructions per 32-entry tile and
// solve at 44 % issue utilisation) and the lookups' latency.  Measured: 4,096
// matrices of 200 to 20,000 columns, 21.2 ms over the union, now 12.0 ms; a
// single random matrix of 2,000 columns and 16,000 entries 128 us, now 67 us.
// With few matrices most SMs are idle and the call lasts as long as its largest
// one: BatchLoad (awpm_rules.h) says which batches come here.
//
// The kernel only reports that something is wrong with an input (kErrRetry);
// the caller then solves the batch by the general path, which names the error.
#include <cooperative_groups.h>

#include "awpm.h"
#include "awpm_dev.h"
#include "awpm_internal.h"

namespace awpm {

namespace {

// Classes of matrix sizes, each with its block size and blocks per SM (the
// shared memory of the largest n decides): small blocks keep several matrices
// on an SM, since most of a small one's time is latency.
template <int kClass>
struct Cls;
template <>
struct Cls<0> {
    static constexpr int kThreads = 1024, kBlocks = 1;
};
template <>
struct Cls<1> {
    static constexpr int kThreads = 512, kBlocks = 2;
};
template <>
struct Cls<2> {
    static constexpr int kThreads = 256, kBlocks = 4;
};

// A single matrix: a cluster of blocks shares its tiles; each block keeps the
// matching and the bitmaps of its own, and a flip goes to all of them through
// distributed shared memory.
constexpr int kOneBlocks = 8;
template <>
struct Cls<kSmallOne> {
    static constexpr int kThreads = 512, kBlocks = 1;
};

constexpr int kRing = 64;

// The address of p, in this block's shared memory, in block `rank` of the
// cluster (kC blocks; 1: no cluster).
template <int kC, typename T>
__device__ __forceinline__ T *in_block(T *p, int rank)
{
    if (kC == 1)
        return p;
    return cooperative_groups::this_cluster().map_shared_rank(p, rank);
}

template <int kC>
__device__ __forceinline__ int block_rank()
{
    return kC == 1 ? 0 : (int)cooperative_groups::this_cluster().block_rank();
}

// Barrier of the threads that solve a matrix together.
template <int kC>
__device__ __forceinline__ void solve_sync()
{
    if (kC == 1)
        __syncthreads();
    else
        cooperative_groups::this_cluster().sync();
}

// One matrix's arrays in shared memory.
struct Lay {
    uint16_t *mc, *mr, *mold;  // row of a column, column of a row, row before the last flip
    int32_t *cp;               // column pointers, from the matrix's first entry
    uint32_t *sig;             // 32-bit signatures of the columns' rows, or null
    uint32_t *win, *rdirty, *cfull, *cpos;
    uint32_t *tmark;           // tiles of columns in cfull or cpos, or null (no room)
    int words, twords;         // of a bitmap of columns, of tiles
};

__device__ __forceinline__ uint32_t sig32(int32_t r)
{
    const uint32_t h = (uint32_t)r * 0x9E3779B1u;
    return (1u << (h >> 28)) | (0x10000u << ((h >> 24) & 15u));
}

__device__ __forceinline__ bool bit_of(const uint32_t *map, int32_t x)
{
    return (map[x >> 5] >> (x & 31)) & 1u;
}

// Exact record reads after other threads' exchanges: from L2.
__device__ __forceinline__ Rec ld_best(const Rec *p)
{
    const int4 v = __ldcg(reinterpret_cast<const int4 *>(p));
    Rec r;
    r.g = __hiloint2double(v.y, v.x);
    r.p = v.z;
    r.q = v.w;
    return r;
}

// Column of the lane's entry of the tile at `base`, whose first entry is in
// column c0 (no column is empty).
__device__ __forceinline__ int32_t tile_column(const int32_t *cp, int32_t n, int32_t c0,
                                               int32_t base, int lane)
{
    const int32_t x = c0 + 1 + lane;
    const int32_t d = x < n ? cp[x] - base : 32;
    const uint32_t starts = __reduce_or_sync(FULL_MASK, d < 32 ? 1u << d : 0u);
    return c0 + __popc(starts & ((2u << lane) - 1u));
}

// Requests (entry, row and column) of one warp, resolved 32 at a time: the
// closing entry (m_j, m_i) by binary search in column m_i, the gain, the
// columns' Step-C records.
struct Ring {
    int2 e[kRing];  // local position; row | column << 16
};

template <int kClass, int kC>
struct Solver {
    const Work &w;
    Lay L;
    int32_t o, n, p0, nz;
    uint32_t *fb, *pb;  // found and positive bits of the matrix's tiles
    int32_t *c0;        // column of the tiles' first entries
    Ring *ring;
    int head, have;     // warp-uniform
    uint32_t n_found, n_pos;

    __device__ __forceinline__ void resolve(int k)
    {
        __syncwarp();
        const int lane = threadIdx.x & 31;
        const bool act = lane < k;
        const int2 e = act ? ring->e[(head + lane) & (kRing - 1)] : make_int2(-1, 0);
        const int32_t i = e.y & 0xffff, j = act ? (int32_t)((uint32_t)e.y >> 16) : -1;
        int32_t q = -1, mi = 0;
        if (act) {
            const int32_t key = L.mc[j] + o;
            mi = L.mr[i];
            int32_t lo = L.cp[mi], len = L.cp[mi + 1] - lo;
            while (len > 0) {
                const int32_t half = len >> 1;
                const int32_t v = __ldg(w.rowidx + p0 + lo + half);
                if (v == key) {
                    q = lo + half;
                    break;
                }
                if (v < key) {
                    lo += half + 1;
                    len -= half + 1;
                } else {
                    len = half;
                }
            }
        }
        double g = 0.0;
        bool pos = false;
        if (q >= 0) {
            g = ((__ldg(w.w + p0 + e.x) + __ldg(w.w + p0 + q)) - w.wm[o + mi]) - w.wm[o + j];
            pos = gain_positive(g);
            ++n_found;
            n_pos += pos;
        }
        if (q >= 0) {
            atomicOr(fb + (e.x >> 5), 1u << (e.x & 31));
            if (pos)
                atomicOr(pb + (e.x >> 5), 1u << (e.x & 31));
        }
        const unsigned any_pos = __ballot_sync(FULL_MASK, pos);
        if (any_pos) {
            // one record per column (a column's requests are side by side)
            long long gk = pos ? gbits(g) : 0ll;
            int from = lane;
            const bool several = (any_pos & (any_pos - 1u)) != 0u;
            if (several) {
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int32_t j2 = __shfl_down_sync(FULL_MASK, j, d);
                    const long long g2 = __shfl_down_sync(FULL_MASK, gk, d);
                    const int f2 = __shfl_down_sync(FULL_MASK, from, d);
                    if (j2 == j && g2 > gk) {  // equal gains: the lower position, this lane's
                        gk = g2;
                        from = f2;
                    }
                }
            }
            const int32_t before = __shfl_up_sync(FULL_MASK, j, 1);
            Rec r;
            r.g = __longlong_as_double(gk);
            r.p = __shfl_sync(FULL_MASK, e.x, from);
            r.q = __shfl_sync(FULL_MASK, q, from);
            if (gk > 0ll && (!several || lane == 0 || before != j)) {
                rec_combine(w.best + o + j, r, w.ctl);
                atomicOr(L.win + (j >> 5), 1u << (j & 31));
            }
        }
        __syncwarp();
        head = (head + k) & (kRing - 1);
        have -= k;
    }

    // Steps A-C of a pass over the warp's tiles; returns the lane's candidates
    // (differences after the first pass).  Blocks of 32 tiles have their words
    // read a tile per lane; the row indices come four tiles ahead.  After the
    // first pass a tile without a changed row or a marked column costs its
    // rows' bits and a vote.  The tiles that are looked at take a rolled loop
    // (their rows read again, from L1), so that the code stays small.
    __device__ __forceinline__ int32_t search(bool first, int32_t t_lo, int32_t t_hi)
    {
        constexpr int kU = 4;
        const int lane = threadIdx.x & 31;
        const unsigned lanes_below = (1u << lane) - 1u;
        const int32_t *__restrict__ rows = w.rowidx + p0;
        int32_t cand_n = 0;
        int32_t nr[kU];
        auto fetch = [&](int32_t t) {
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int32_t p = (t + u) * 32 + lane;
                nr[u] = t + u < t_hi && p < nz ? __ldg(rows + p) - o : 0;
            }
        };
        if (t_lo < t_hi)
            fetch(t_lo);
        for (int32_t tb = t_lo; tb < t_hi; tb += 32) {
            int32_t c0l = 0;
            uint32_t fl = 0u, sl = 0u;
            bool marked = false;
            if (tb + lane < t_hi) {
                c0l = c0[tb + lane];
                if (!first) {
                    fl = __ldcg(fb + tb + lane);
                    sl = __ldcg(pb + tb + lane);
                }
                marked = first || !L.tmark || bit_of(L.tmark, tb + lane);
            }
            const unsigned marks = __ballot_sync(FULL_MASK, marked);
            for (int u0 = 0; u0 < 32 && tb + u0 < t_hi; u0 += kU) {
                uint32_t hits = 0u;
#pragma unroll
                for (int u = 0; u < kU; ++u)
                    hits |= ((L.rdirty[nr[u] >> 5] >> (nr[u] & 31)) & 1u) << u;
                fetch(tb + u0 + kU);
                unsigned todo = (marks >> u0) & ((1u << kU) - 1u);
                todo |= __reduce_or_sync(FULL_MASK, hits);
#pragma unroll 1
                while (todo) {
                    const int u = __ffs(todo) - 1;
                    todo &= todo - 1;
                    const int32_t t = tb + u0 + u, base = t * 32, p = base + lane;
                    if (t >= t_hi)
                        break;
                    const int32_t c = __shfl_sync(FULL_MASK, c0l, u0 + u);
                    const uint32_t f = __shfl_sync(FULL_MASK, fl, u0 + u);
                    const uint32_t s = __shfl_sync(FULL_MASK, sl, u0 + u);
                    const bool valid = p < nz;
                    const int32_t r = valid ? __ldg(rows + p) - o : 0;
                    const int32_t j = tile_column(L.cp, n, c, base, lane);
                    bool ev = valid, whole = false;
                    if (!first) {
                        if (valid) {
                            whole = bit_of(L.cfull, j);
                            ev = whole || ((hits >> u) & 1u) ||
                                 (bit_of(L.cpos, j) && ((s >> lane) & 1u));
                        }
                        const unsigned m = __ballot_sync(FULL_MASK, ev);
                        if (lane == 0 && (f & m)) {
                            n_found -= __popc(f & m);
                            n_pos -= __popc(s & m);
                            fb[t] = f & ~m;
                            pb[t] = s & ~m;
                        }
                    }
                    bool pass = false;
                    if (ev) {
                        const int32_t mj = L.mc[j];
                        pass = r > mj;
                        if (first)
                            cand_n += pass;
                        else if (whole)
                            cand_n += (int)pass - (int)(r > (int32_t)L.mold[j]);
                        if (pass && L.sig) {
                            const uint32_t b = sig32(mj);
                            pass = (L.sig[L.mr[r]] & b) == b;
                        }
                    }
                    const unsigned m = __ballot_sync(FULL_MASK, pass);
                    if (pass)
                        ring->e[(head + have + __popc(m & lanes_below)) & (kRing - 1)] =
                            make_int2(p, r | (j << 16));
                    have += __popc(m);
                    if (have >= 32)
                        resolve(32);
                }
            }
        }
        if (have > 0)
            resolve(have);
        return cand_n;
    }
};

template <int kThr>
__device__ double block_sum(double v)
{
    __shared__ double s[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1)
        v += __shfl_down_sync(FULL_MASK, v, d);
    __syncthreads();
    if (lane == 0)
        s[wid] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int x = 0; x < kThr / 32; ++x)
            t += s[x];
    return t;  // thread 0
}

template <int kClass, int kC>
__device__ void solve_matrix(const Work &w, int32_t b, unsigned char *smem)
{
    constexpr int kThr = Cls<kClass>::kThreads, kW = kThr / 32;
    // (block 0's of a cluster are the matrix's)
    __shared__ int s_bad, s_matched, s_go;
    __shared__ int s_flips;
    __shared__ int s_cnt[3];
    __shared__ double s_part[kC];
    const BatchWork &bw = w.bw;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int rank = block_rank<kC>();
    // thread and warp among all that solve the matrix
    const int gt = rank * kThr + tid, gw = rank * kW + wid;
    constexpr int kGT = kThr * kC, kGW = kW * kC;
    const int32_t o = bw.n_off[b], n = bw.n_off[b + 1] - o;
    Ctl *ctl = w.ctl;
    if (n == 0) {
        if (gt == 0) {
            bw.miter[b] = 1;
            bw.mconv[b] = 1;
            bw.mnnz[b] = 0;
            bw.mcycles[b] = 0ull;
            bw.mw_in[b] = bw.mw_out[b] = 0.0;
            atomicMax(&ctl->iterations, 1);
        }
        return;
    }
    const int32_t nnz = w.small_nnz ? *w.small_nnz : w.nnz;
    const int32_t p0 = w.colptr[o], p1 = w.colptr[o + n], nz = p1 - p0;

    // shared memory of this matrix
    Lay L;
    unsigned char *at = smem + kW * sizeof(Ring);
    L.words = n / 32 + 1;
    L.cp = reinterpret_cast<int32_t *>(at);
    at += 4 * (size_t)(n + 1);
    L.win = kC == 1 ? reinterpret_cast<uint32_t *>(at) : w.winbits;
    L.rdirty = reinterpret_cast<uint32_t *>(at) + L.words;
    L.cfull = L.rdirty + L.words;
    L.cpos = L.cfull + L.words;
    at += 16 * (size_t)L.words;
    const bool sigs = small_smem(n, kW, true) <= (size_t)w.small_smem[kClass];
    uint32_t *sig = nullptr;  // where the signatures are put together
    L.sig = sigs ? reinterpret_cast<uint32_t *>(at) : nullptr;
    if (sigs) {
        at += 4 * (size_t)n;
        sig = kC == 1 ? L.sig : w.small_sig;
    }
    L.mc = reinterpret_cast<uint16_t *>(at);
    L.mr = L.mc + n;
    L.mold = L.mr + n;
    at += 6 * (size_t)n;
    const int32_t nt = (nz + 31) / 32;
    L.twords = nt / 32 + 1;
    at = smem + ((at - smem + 3) & ~(size_t)3);
    L.tmark = nz >= 0 && (size_t)(at - smem) + 4 * (size_t)L.twords <= (size_t)w.small_smem[kClass]
                  ? reinterpret_cast<uint32_t *>(at)
                  : nullptr;

    if (tid == 0) {
        s_bad = 0;
        s_matched = 0;
    }
    solve_sync<kC>();
    // (the same in every thread)
    // (the pointers run from 0 to exactly nnz, which a served request states)
    const bool fits = p0 >= 0 && p1 <= nnz && nz >= n && nnz <= w.small_cap &&
                      (o != 0 || p0 == 0) && (o + n != w.n || p1 == nnz);
    if (fits) {
        bool bad = false;
        for (int32_t j = tid; j <= n; j += kThr) {
            const int32_t c = w.colptr[o + j];
            L.cp[j] = c - p0;
            bad |= j < n && w.colptr[o + j + 1] <= c;
        }
        for (int32_t x = tid; x < 3 * L.words; x += kThr)
            L.rdirty[x] = 0u;  // (and cfull, cpos)
        for (int32_t x = gt % (kC == 1 ? kThr : kGT); x < L.words; x += kC == 1 ? kThr : kGT)
            L.win[x] = 0u;
        if (L.tmark)
            for (int32_t x = tid; x < L.twords; x += kThr)
                L.tmark[x] = 0u;
        for (int32_t j = tid; j < n; j += kThr) {
            const int32_t r = w.mate_in[o + j] - o;
            bad |= r < 0 || r >= n;
            L.mc[j] = (uint16_t)r;
            L.mr[j] = 0xffff;
            if (sigs)
                sig[j] = 0u;
            if (!w.rec_clean && (kC == 1 || j % kC == rank)) {
                w.best[o + j] = Rec{0.0, 0, 0};
                w.dsel[o + j] = Sel{0.0, 0, 0};
            }
        }
        if (bad)
            *in_block<kC>(&s_bad, 0) = 1;
    }
    solve_sync<kC>();
    const bool ok = fits && !*in_block<kC>(&s_bad, 0);
    solve_sync<kC>();  // (read by all before it is written again)
    if (ok) {
        for (int32_t j = tid; j < n; j += kThr)
            L.mr[L.mc[j]] = (uint16_t)j;
    }
    __syncthreads();
    const int32_t t_lo = (int32_t)((int64_t)nt * gw / kGW);
    const int32_t t_hi = (int32_t)((int64_t)nt * (gw + 1) / kGW);
    uint32_t *fb = w.small_fb + (p0 >> 5) + b, *pb = w.small_pb + (p0 >> 5) + b;
    int32_t *tc = w.small_c0 + (p0 >> 5) + b;
    if (ok) {
        // the entries: rows in the block, ascending, weights finite; the
        // columns' signatures and matched weights
        bool bad = false;
        for (int32_t j = tid; j < n; j += kThr)
            bad |= L.mr[L.mc[j]] != j;  // two columns with one row
        int matched = 0;
        if (t_lo < t_hi) {
            constexpr int kU = 4;
            int32_t c0 = 0;  // last column starting at or before the first tile
            for (int32_t hi = n - 1; c0 < hi;) {
                const int32_t mid = (c0 + hi + 1) >> 1;
                if (L.cp[mid] <= t_lo * 32)
                    c0 = mid;
                else
                    hi = mid - 1;
            }
            int32_t last = t_lo > 0 ? __ldg(w.rowidx + p0 + t_lo * 32 - 1) - o : -1;
            for (int32_t t = t_lo; t < t_hi; t += kU) {
                int32_t r[kU];
                double x[kU];
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const int32_t p = (t + u) * 32 + lane;
                    const bool v = t + u < t_hi && p < nz;
                    r[u] = v ? __ldg(w.rowidx + p0 + p) - o : 0;
                    x[u] = v ? __ldcs(w.w + p0 + p) : 0.0;
                }
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    if (t + u >= t_hi)
                        break;
                    const int32_t base = (t + u) * 32, p = base + lane;
                    const int32_t j = tile_column(L.cp, n, c0, base, lane);
                    int32_t before = __shfl_up_sync(FULL_MASK, r[u], 1);
                    if (lane == 0)
                        before = last;
                    last = __shfl_sync(FULL_MASK, r[u], 31);
                    if (lane == 0) {
                        fb[t + u] = 0u;
                        pb[t + u] = 0u;
                        tc[t + u] = c0;
                    }
                    // the next tile's first column: the last lane's, or the one after
                    c0 = __shfl_sync(FULL_MASK, j, 31);
                    if (c0 + 1 < n && L.cp[c0 + 1] == base + 32)
                        ++c0;
                    if (p < nz) {
                        const bool first = L.cp[j] == p;
                        const bool in = r[u] >= 0 && r[u] < n;
                        bad |= !in || (!first && before >= r[u]) ||
                               (__double2hiint(x[u]) & 0x7ff00000) == 0x7ff00000;
                        if (in) {
                            if (sigs)
                                atomicOr(sig + j, sig32(r[u]));
                            if (r[u] == (int32_t)L.mc[j]) {
                                w.wm[o + j] = x[u];
                                ++matched;
                            }
                        }
                    }
                }
            }
        }
        matched = __reduce_add_sync(FULL_MASK, matched);
        if (lane == 0)
            atomicAdd(in_block<kC>(&s_matched, 0), matched);
        if (bad)
            *in_block<kC>(&s_bad, 0) = 1;
    }
    solve_sync<kC>();
    // (the same in every thread: nothing changes them any more)
    const bool good = ok && !*in_block<kC>(&s_bad, 0) && *in_block<kC>(&s_matched, 0) == n;
    if (!good) {
        if (gt == 0)
            raise_err(ctl, kErrRetry);
        if (kC > 1)
            solve_sync<kC>();  // (block 0's words are read until here)
        return;
    }
    if (kC > 1 && sigs) {
        // the signatures were put together in global memory
        for (int32_t j = tid; j < n; j += kThr)
            L.sig[j] = __ldcg(sig + j);
        __syncthreads();
    }
    auto weight = [&]() {
        double v = 0.0;
        for (int32_t j = gt; j < n; j += kGT)
            v += w.wm[o + j];
        v = block_sum<kThr>(v);
        if (kC > 1) {
            if (tid == 0)
                in_block<kC>(s_part, 0)[rank] = v;
            solve_sync<kC>();
            if (gt == 0)
                for (int x = 1; x < kC; ++x)
                    v += s_part[x];
        }
        return v;  // in thread 0 (of block 0)
    };
    const double w_in = weight();

    Solver<kClass, kC> S{w, L, o, n, p0, nz, fb, pb, tc,
                     reinterpret_cast<Ring *>(smem) + wid, 0, 0, 0u, 0u};
    long long cand = 0, found = 0, posi = 0;           // thread 0: totals
    long long cur_cand = 0, cur_found = 0, cur_pos = 0;  // and the last pass's counts
    long long cycles = 0;
    int32_t it = 0;
    bool conv = false;
    const int per = words_per_warp(L.words, kGW);
    if (tid == 0)
        s_cnt[0] = s_cnt[1] = s_cnt[2] = s_flips = 0;
    solve_sync<kC>();
    for (;;) {
        S.n_found = S.n_pos = 0u;
        int c = S.search(it == 0, t_lo, t_hi);
        c = __reduce_add_sync(FULL_MASK, c);
        const int f = __reduce_add_sync(FULL_MASK, (int)S.n_found);
        const int g = __reduce_add_sync(FULL_MASK, (int)S.n_pos);
        if (lane == 0) {
            int *cnt = in_block<kC>(s_cnt, 0);
            atomicAdd(cnt, c);
            atomicAdd(cnt + 1, f);
            atomicAdd(cnt + 2, g);
        }
        solve_sync<kC>();
        // Step D: keys and selection; the bitmaps this search read are emptied
        const int32_t epoch = w.epoch0 + it + 1;
        for (int32_t x = tid; x < 3 * L.words; x += kThr)
            L.rdirty[x] = 0u;  // (and cfull, cpos)
        if (L.tmark)
            for (int32_t x = tid; x < L.twords; x += kThr)
                L.tmark[x] = 0u;
        for (int32_t x0 = gw * per; x0 < L.words; x0 += kGW * per)
            for_winners(L.win, x0, per, L.words, lane, false, [&](int32_t j) {
                if (j < 0)
                    return;
                const Rec r = ld_best(w.best + o + j);
                const int32_t k = L.mr[__ldg(w.rowidx + p0 + r.p) - o];
                if (bit_of(L.win, k)) {
                    w.wkey[o + j] = ~k;
                    return;
                }
                w.wkey[o + j] = k;
                sel_combine(w.dsel + o + k, Sel{r.g, j, epoch}, ctl);
            });
        solve_sync<kC>();
        // the flip (see flip_body for the records that stand)
        auto selected = [&](int32_t key, int32_t j) {
            const Sel s = ld_record(w.dsel + o + key);
            return s.epoch == epoch && s.j == j;
        };
        // in every block's copy
        auto set_bit = [&](uint32_t *map, int32_t x) {
#pragma unroll
            for (int y = 0; y < kC; ++y)
                atomicOr(in_block<kC>(map + (x >> 5), y), 1u << (x & 31));
        };
        auto put16 = [&](uint16_t *a, int32_t x, int32_t v) {
#pragma unroll
            for (int y = 0; y < kC; ++y)
                *in_block<kC>(a + x, y) = (uint16_t)v;
        };
        auto mark_tiles = [&](int32_t j) {
            if (L.tmark)
                for (int32_t x = L.cp[j] >> 5; x <= (L.cp[j + 1] - 1) >> 5; ++x)
                    set_bit(L.tmark, x);
        };
        int flips = 0;
        for (int32_t x0 = gw * per; x0 < L.words; x0 += kGW * per)
            for_winners(L.win, x0, per, L.words, lane, true, [&](int32_t j) {
                if (j < 0)
                    return;
                const Rec r = ld_best(w.best + o + j);
                const int32_t k = w.wkey[o + j];
                if (k < 0) {
                    const int32_t k2 = w.wkey[o + ~k];
                    if (k2 < 0 || !selected(k2, ~k)) {  // stands
                        atomicOr(L.win + (j >> 5), 1u << (j & 31));
                        return;
                    }
                }
                w.best[o + j] = Rec{0.0, 0, 0};
                if (k < 0 || !selected(k, j)) {
                    set_bit(L.cpos, j);
                    mark_tiles(j);
                    return;
                }
                const int32_t i = __ldg(w.rowidx + p0 + r.p) - o;
                const int32_t mj = L.mc[j];
                put16(L.mold, j, mj);
                put16(L.mold, k, i);
                put16(L.mc, j, i);
                put16(L.mr, i, j);
                put16(L.mc, k, mj);
                put16(L.mr, mj, k);
                w.wm[o + j] = __ldg(w.w + p0 + r.p);
                w.wm[o + k] = __ldg(w.w + p0 + r.q);
                set_bit(L.rdirty, i);
                set_bit(L.rdirty, mj);
                set_bit(L.cfull, j);
                set_bit(L.cfull, k);
                mark_tiles(j);
                mark_tiles(k);
                ++flips;
            });
        flips = __reduce_add_sync(FULL_MASK, flips);
        if (lane == 0 && flips)
            atomicAdd(in_block<kC>(&s_flips, 0), flips);
        solve_sync<kC>();
        ++it;
        if (gt == 0) {
            cand += cur_cand += s_cnt[0];
            found += cur_found += s_cnt[1];
            posi += cur_pos += s_cnt[2];
            cycles += s_flips;
            conv = s_flips == 0;
            const int go = s_flips != 0 && it < w.max_passes &&
                           *(volatile unsigned *)&ctl->err == 0u;
            for (int y = 0; y < kC; ++y)
                *in_block<kC>(&s_go, y) = go;
            s_cnt[0] = s_cnt[1] = s_cnt[2] = s_flips = 0;
        }
        solve_sync<kC>();
        if (!s_go)
            break;
    }
    const double w_out = weight();
    for (int32_t j = gt; j < n; j += kGT)
        w.small_out[o + j] = L.mc[j] + o;
    if (gt == 0) {
        bw.miter[b] = it;
        bw.mconv[b] = conv ? 1 : 0;
        bw.mnnz[b] = nz;
        bw.mcycles[b] = (unsigned long long)cycles;
        bw.mw_in[b] = w_in;
        bw.mw_out[b] = w_out;
        atomicAdd(&ctl->candidates, (unsigned long long)cand);
        atomicAdd(&ctl->found, (unsigned long long)found);
        atomicAdd(&ctl->positive, (unsigned long long)posi);
        atomicAdd(&ctl->cycles, (unsigned long long)cycles);
        atomicMax(&ctl->iterations, it);
        if (!conv)
            ctl->converged = 0;
    }
}

__device__ __forceinline__ void small_reset(const Work &w)
{
    Ctl *c = w.ctl;
    c->err = 0u;
    c->active = 1;
    c->iterations = 0;
    c->converged = 1;
    c->cycles = 0ull;
    c->candidates = 0ull;
    c->found = 0ull;
    c->positive = 0ull;
    c->weight_in = 0.0;
    c->weight_out = 0.0;
    for (int x = 0; x < kSmallClasses; ++x)
        w.small_next[x] = 0;
}

__global__ void k_small_reset(const Work *__restrict__ W)
{
    small_reset(*W);
}

// Nothing: what a stream does before a class's kernel to let the kernels of the
// larger classes, submitted before, take their places first.
__global__ void k_small_later() {}

// The matrices of one class, largest first, from a queue.
template <int kClass>
__global__ void __launch_bounds__(Cls<kClass>::kThreads, Cls<kClass>::kBlocks)
    k_small(const Work *__restrict__ W)
{
    extern __shared__ __align__(16) unsigned char s_raw[];
    __shared__ int32_t s_b;
    const Work &w = *W;
    for (;;) {
        if (threadIdx.x == 0) {
            const int32_t x = atomicAdd(w.small_next + kClass, 1);
            s_b = x < w.small_count[kClass] ? w.small_order[w.small_first[kClass] + x] : -1;
        }
        __syncthreads();
        const int32_t b = s_b;
        if (b < 0)
            return;
        solve_matrix<kClass, 1>(w, b, s_raw);
        __syncthreads();
    }
}

// A single matrix: one cluster, which also prepares and ends the solve.
__global__ void __cluster_dims__(kOneBlocks, 1, 1)
    __launch_bounds__(Cls<kSmallOne>::kThreads, Cls<kSmallOne>::kBlocks)
        k_small_one(const Work *__restrict__ W)
{
    extern __shared__ __align__(16) unsigned char s_raw[];
    const Work &w = *W;
    if (gtid() == 0) {
        small_reset(w);
        w.ctl->small_nnz = w.small_nnz ? *w.small_nnz : w.nnz;
    }
    // (the reset is ordered before every use by the solve's first barrier)
    solve_matrix<kSmallOne, kOneBlocks>(w, 0, s_raw);
    if (gtid() == 0 && !w.ctl->err) {
        w.ctl->weight_in = w.bw.mw_in[0];
        w.ctl->weight_out = w.bw.mw_out[0];
    }
}

// The whole batch's weights, in a fixed order.
__global__ void k_small_total(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (w.ctl->err)
        return;
    double a = 0.0, b = 0.0;
    for (int32_t x = threadIdx.x; x < w.bw.count; x += 1024) {
        a += w.bw.mw_in[x];
        b += w.bw.mw_out[x];
    }
    a = block_sum<1024>(a);
    b = block_sum<1024>(b);
    if (threadIdx.x == 0) {
        w.ctl->weight_in = a;
        w.ctl->weight_out = b;
    }
}

__global__ void k_small_entries(const int32_t *__restrict__ off, const int32_t *__restrict__ colptr,
                                int32_t n, int32_t count, int32_t *__restrict__ at)
{
    // (the host has checked its copy of the offsets)
    for (int64_t b = gtid(); b <= count; b += gstride())
        at[b] = __ldg(colptr + min(max(__ldg(off + b), 0), n));
}

cudaError_t allow(const void *f, int c)
{
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)small_class_smem(c));
}

}  // namespace

cudaError_t small_setup()
{
    cudaError_t e = allow((const void *)k_small<0>, 0);
    if (e == cudaSuccess)
        e = allow((const void *)k_small<1>, 1);
    if (e == cudaSuccess)
        e = allow((const void *)k_small<2>, 2);
    if (e == cudaSuccess)
        e = allow((const void *)k_small_one, kSmallOne);
    return e;
}

void launch_small_batch(const Work *d, const Shape &sh, const int32_t *counts,
                        const SmallStreams &ss, Sink &k)
{
    void *a[] = {(void *)&d};
    const unsigned sms = (unsigned)sh.num_sms;
    k.launch((const void *)k_small_reset, 1, 1, a);
    const void *f[kSmallClasses] = {(const void *)k_small<0>, (const void *)k_small<1>,
                                    (const void *)k_small<2>};
    const unsigned threads[kSmallClasses] = {Cls<0>::kThreads, Cls<1>::kThreads, Cls<2>::kThreads};
    const unsigned blocks[kSmallClasses] = {Cls<0>::kBlocks, Cls<1>::kBlocks, Cls<2>::kBlocks};
    // The classes side by side, the largest first: as the blocks of one run out of
    // matrices, the next one's take their SMs.  A class that starts before a
    // larger one keeps the SMs until its queue is empty, which made some calls
    // longer (4,096 matrices of 200 to 20,000 columns 13.3 ms instead of 12.2), so
    // each class lets those before it go first.
    auto note = [&k](cudaError_t e) {
        if (k.err == cudaSuccess)
            k.err = e;
    };
    note(cudaEventRecord(ss.fork, k.stream));
    int before = 0;  // classes launched
    for (int c = 0; c < kSmallClasses; ++c) {
        const unsigned most = sms * blocks[c];
        if (counts[c] <= 0)
            continue;
        Sink s;
        s.stream = before == 0 ? k.stream : ss.side[before - 1];
        if (before > 0)
            note(cudaStreamWaitEvent(s.stream, ss.fork, 0));
        for (int x = 0; x < before; ++x)
            s.launch((const void *)k_small_later, 1, 32, nullptr);
        s.launch(f[c], (unsigned)counts[c] < most ? (unsigned)counts[c] : most, threads[c], a,
                 (unsigned)small_class_smem(c));
        note(s.err);
        if (before > 0)
            note(cudaEventRecord(ss.join[before - 1], s.stream));
        ++before;
    }
    for (int x = 0; x + 1 < before; ++x)
        note(cudaStreamWaitEvent(k.stream, ss.join[x], 0));
    k.launch((const void *)k_small_total, 1, 1024, a);
}

void launch_small_entries(const int32_t *off, const int32_t *colptr, int32_t n, int32_t count,
                          int32_t *at, Sink &k)
{
    void *a[] = {(void *)&off, (void *)&colptr, (void *)&n, (void *)&count, (void *)&at};
    const int64_t blocks = ((int64_t)count + kThreads) / kThreads;
    k.launch((const void *)k_small_entries, (unsigned)(blocks < 1024 ? blocks : 1024), kThreads, a);
}

void launch_small_one(const Work *d, int32_t smem, Sink &k)
{
    void *a[] = {(void *)&d};
    k.launch((const void *)k_small_one, kOneBlocks, Cls<kSmallOne>::kThreads, a,
             (unsigned)smem);
}

}  // namespace awpm

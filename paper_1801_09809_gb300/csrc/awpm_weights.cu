// Matching weights from matrix values (Section 6.1): kernels (sm_103a).
//
// One sweep of max-equilibration, columns first: v_ij = |a_ij| / max_k |a_kj|,
// w_ij = v_ij / max_l v_il, so every row's largest weight is exactly 1; the
// weight is w (Option A, sum objective) or log(w) (Option B, product
// objective).  Maxima compare bit patterns of positive doubles as integers,
// and divisions and logarithms run on the integer units (awpm_fixed.h: the
// quotients correctly rounded, so Option A is bit-for-bit reproducible),
// because a GB300 SM issues about two FP64 operations per clock: with FP64
// comparisons, two FP64 divisions per entry and the device's log the three
// kernels took 3.5, 7.1 and 22.4 ms on an R-MAT matrix of scale 22 (n = 4.2 M,
// 69 M entries), against 0.2 ms for the bytes; now 0.40, 0.64 and 0.75 ms (a
// call 29.0 -> 1.83 ms).  What bounds them: instruction issue in the last
// (2.7 instructions per clock and SM), the gathers of the columns' scales and
// the rows' maxima in the second.
//
// The work is spread by entries (a warp per 32-entry tile, four tiles per
// round with their loads side by side), not by columns: a warp per column
// left most lanes idle on short columns and one warp alone on a hub's.  Small
// matrices, whose time is launches, take a form with fewer of them.
#include <math.h>

#include "awpm.h"
#include "awpm_dev.h"
#include "awpm_internal.h"

namespace awpm {

namespace {

constexpr unsigned long long kAbs = 0x7fffffffffffffffull;

__device__ const LogTable g_log_table = fx_make_log_table();

__device__ __forceinline__ bool wt_gate(const Ctl *ctl)
{
    return (*(volatile const unsigned *)&ctl->err & (kErrInvalid | kErrNonfinite)) == 0u;
}

// Column of the lane's entry p of tile t.  The start bits give it when no
// column between the first columns of this tile and the next is empty;
// otherwise the last column starting at or before p is searched for.
__device__ __forceinline__ int32_t entry_column(const Work &w, int32_t t, int32_t p, int lane)
{
    const int32_t c0 = __ldg(w.tile_col + t);
    const uint32_t mask = __ldg(w.starts + t);
    const bool last = t + 1 >= w.ntiles;
    const int32_t c1 = last ? w.n - 1 : __ldg(w.tile_col + t + 1);
    const int32_t inside = __popc(mask & ~1u) + (int32_t)(last ? 0u : __ldg(w.starts + t + 1) & 1u);
    if (c1 - c0 == inside)
        return lane_column(c0, mask, lane);
    int32_t lo = c0, hi = c1;
    while (lo < hi) {
        const int32_t mid = (int32_t)(((int64_t)lo + hi + 1) >> 1);
        if (__ldg(w.colptr + mid) <= p)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// |a| / s.v as bits; the FP64 division where an operand or the quotient is
// not a normal number.
__device__ __forceinline__ unsigned long long divide(unsigned long long a, const Scale &s)
{
    bool ok;
    unsigned long long q = quotient(a, s, ok);
    if (!ok)
        q = fx_bits(fx_double(a) / fx_double(s.v));
    return q;
}

__device__ __forceinline__ Scale ld_scale(const Scale *p)
{
    const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2 *>(p));
    Scale s;
    s.v = v.x;
    s.inv = v.y;
    return s;
}

// The state the weights' kernels start from.
__device__ __forceinline__ void wt_reset(const Work &w)
{
    if (gtid() == 0) {
        w.ctl->err = 0u;
        w.ctl->active = 1;
    }
    for (int64_t x = gtid(); x < w.n; x += gstride()) {
        w.wt_max[x] = 0ull;
    }
    const int64_t words = w.starts ? ((int64_t)w.nnz + 31) / 32 + 1 : 0;
    for (int64_t x = gtid(); x < words; x += gstride())
        w.starts[x] = 0u;
}

__global__ void k_wt_reset(const Work *__restrict__ W)
{
    wt_reset(*W);
}

// Checks (rows in range; values finite and nonzero) and the column maxima: a
// segmented maximum in the warp, stored by the first lane of a column that
// lies in the tile whole, merged by a 64-bit atomic for a column cut by a
// tile's end.
__global__ void __launch_bounds__(kThreads) k_wt_colmax(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (w.ctl->err & kErrInvalid)
        return;
    constexpr int kU = 4;
    const int lane = threadIdx.x & 31;
    const int32_t nwarps = (int32_t)(gstride() >> 5);
    const int32_t n = w.n, nnz = w.nnz, ntiles = w.ntiles;
    const unsigned long long *__restrict__ av =
        reinterpret_cast<const unsigned long long *>(w.wt_a);
    unsigned bits = 0;
    for (int32_t t0 = (int32_t)(gtid() >> 5); t0 < ntiles; t0 += kU * nwarps) {
        int32_t r[kU];
        uint32_t mask[kU];
        unsigned long long v[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int32_t t = t0 + u * nwarps;
            const int32_t p = t < ntiles ? t * kTile + lane : nnz;
            const bool valid = p < nnz;
            mask[u] = t < ntiles ? __ldg(w.starts + t) : 1u;
            r[u] = valid ? __ldcs(w.rowidx + p) : 0;
            v[u] = valid ? __ldcs(av + p) & kAbs : 1ull;
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int32_t t = t0 + u * nwarps;
            if (t >= ntiles)
                continue;
            const int32_t base = t * kTile, p = base + lane;
            const bool valid = p < nnz;
            if (r[u] < 0 || r[u] >= n)
                bits |= kErrInvalid;
            if (v[u] == 0ull || v[u] >= 0x7ff0000000000000ull)
                bits |= kErrNonfinite;
            if (mask[u] <= 1u) {
                const unsigned hi = (unsigned)(v[u] >> 32);
                const unsigned mh = __reduce_max_sync(FULL_MASK, hi);
                const unsigned ml =
                    __reduce_max_sync(FULL_MASK, hi == mh ? (unsigned)v[u] : 0u);
                v[u] = ((unsigned long long)mh << 32) | ml;
            } else {
                const uint32_t after = __funnelshift_rc(mask[u], 0u, lane + 1);
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    // (past lane 31 the shuffle returns the lane's own value)
                    const unsigned long long o = __shfl_down_sync(FULL_MASK, v[u], off);
                    if ((after & ((1u << off) - 1u)) == 0u && o > v[u])
                        v[u] = o;
                }
            }
            if (valid && (lane == 0 || ((mask[u] >> lane) & 1u))) {
                const int32_t j = entry_column(w, t, p, lane);
                if (segment_complete(mask[u], lane, base, nnz, w.starts, t))
                    w.wt_max[j] = v[u];
                else
                    atomicMax(w.wt_max + j, v[u]);
            }
        }
    }
    bits = __reduce_or_sync(FULL_MASK, bits);
    if (lane == 0 && bits)
        raise_err(w.ctl, bits);
}

// The reciprocals of the columns' (then of the rows') maxima; the maxima are
// cleared, for the rows'.
__global__ void k_wt_scale(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (!wt_gate(w.ctl))
        return;
    for (int64_t x = gtid(); x < w.n; x += gstride()) {
        const Scale s = make_scale(w.wt_max[x]);
        w.wt_max[x] = 0ull;
        *reinterpret_cast<ulonglong2 *>(w.wt_scale + x) = make_ulonglong2(s.v, s.inv);
    }
}

// The column-scaled magnitudes (into the output array, read back by
// k_wt_out) and their row maxima (a 64-bit atomic where the value exceeds
// the maximum last seen in L2).  Bound by the gathers of the maxima: two tiles
// a round with six blocks per SM measured a little faster (1.85 ms per call on
// the R-MAT matrix) than four tiles with four (1.89 ms).
__global__ void __launch_bounds__(kThreads, 6) k_wt_rowmax(const Work *__restrict__ W)
{
    const Work &w = *W;
    if (!wt_gate(w.ctl))
        return;
    constexpr int kU = 2;
    const int lane = threadIdx.x & 31;
    const int32_t nwarps = (int32_t)(gstride() >> 5);
    const int32_t nnz = w.nnz, ntiles = w.ntiles;
    const unsigned long long *av = reinterpret_cast<const unsigned long long *>(w.wt_a);
    unsigned long long *out = reinterpret_cast<unsigned long long *>(w.wt_out);
    for (int32_t t0 = (int32_t)(gtid() >> 5); t0 < ntiles; t0 += kU * nwarps) {
        int32_t r[kU];
        unsigned long long v[kU], cur[kU];
        Scale s[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int32_t t = t0 + u * nwarps;
            const int32_t p = t < ntiles ? t * kTile + lane : nnz;
            r[u] = p < nnz ? __ldcs(w.rowidx + p) : -1;
            v[u] = p < nnz ? __ldcs(av + p) & kAbs : kFxOne;
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int32_t t = t0 + u * nwarps;
            s[u].v = kFxOne;
            s[u].inv = 0;
            cur[u] = 0ull;
            if (r[u] >= 0) {
                s[u] = ld_scale(w.wt_scale + entry_column(w, t, t * kTile + lane, lane));
                cur[u] = __ldcg(w.wt_max + r[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            if (r[u] < 0)
                continue;
            const int32_t p = (t0 + u * nwarps) * kTile + lane;
            const unsigned long long q = divide(v[u], s[u]);
            out[p] = q;
            if (q > cur[u])
                atomicMax(w.wt_max + r[u], q);
        }
    }
}

// The thin form of the column maxima and the row maxima, without the columns'
// scales and the tiles' columns: a warp per column, its entries read once for
// the checks (and the column pointers') and, when all are good, twice for the
// maximum and the quotients.
__device__ __forceinline__ void wt_thin_check(const Work &w)
{
    unsigned bits = 0;
    for (int64_t j = gtid(); j <= w.n; j += gstride()) {
        const int32_t c = w.colptr[j];
        if ((j == 0 && c != 0) || (j < w.n && w.colptr[j + 1] < c) || (j == w.n && c != w.nnz))
            bits |= kErrInvalid;
    }
    for (int64_t p = gtid(); p < w.nnz; p += gstride()) {
        const int32_t r = w.rowidx[p];
        const unsigned long long v = fx_bits(w.wt_a[p]) & kAbs;
        if (r < 0 || r >= w.n)
            bits |= kErrInvalid;
        if (v == 0ull || v >= 0x7ff0000000000000ull)
            bits |= kErrNonfinite;
    }
    bits = __reduce_or_sync(FULL_MASK, bits);
    if ((threadIdx.x & 31) == 0 && bits)
        raise_err(w.ctl, bits);
}

__global__ void __launch_bounds__(kThreads) k_wt_thin_check(const Work *__restrict__ W)
{
    wt_thin_check(*W);
}

__device__ __forceinline__ void wt_thin_rowmax(const Work &w)
{
    if (!wt_gate(w.ctl))
        return;
    const int lane = threadIdx.x & 31;
    for (int64_t j = gtid() >> 5; j < w.n; j += gstride() >> 5) {
        const int32_t p0 = w.colptr[j], p1 = w.colptr[j + 1];
        unsigned long long m = 0ull;
        for (int64_t p = (int64_t)p0 + lane; p < p1; p += 32)
            m = max(m, fx_bits(w.wt_a[p]) & kAbs);
#pragma unroll
        for (int off = 16; off; off >>= 1)
            m = max(m, __shfl_xor_sync(FULL_MASK, m, off));
        const Scale s = make_scale(m);
        for (int64_t p = (int64_t)p0 + lane; p < p1; p += 32) {
            const unsigned long long q = divide(fx_bits(w.wt_a[p]) & kAbs, s);
            w.wt_out[p] = fx_double(q);
            atomicMax(w.wt_max + w.rowidx[p], q);
        }
    }
}

__global__ void __launch_bounds__(kThreads) k_wt_thin_rowmax(const Work *__restrict__ W)
{
    wt_thin_rowmax(*W);
}

// The weights, from the column-scaled magnitudes and the row maxima.
template <bool kThin>
__device__ __forceinline__ void wt_out(const Work &w, LogEntry *s_log)
{
    if (!wt_gate(w.ctl))
        return;
    const bool logs = w.wt_mode != 0;
    if (logs) {
        for (int x = threadIdx.x; x < 512; x += (int)blockDim.x)
            s_log[x] = g_log_table.e[x];
        __syncthreads();
    }
    constexpr int kU = 4;
    const int64_t nnz = w.nnz, stride = gstride();
    unsigned long long *out = reinterpret_cast<unsigned long long *>(w.wt_out);
    for (int64_t p0 = gtid(); p0 < nnz; p0 += kU * stride) {
        int32_t r[kU];
        unsigned long long v[kU];
        Scale s[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int64_t p = p0 + u * stride;
            r[u] = p < nnz ? __ldcs(w.rowidx + p) : -1;
            v[u] = p < nnz ? __ldcs(out + p) : kFxOne;
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            s[u].v = kFxOne;
            s[u].inv = 0;
            if (r[u] >= 0)
                s[u] = kThin ? make_scale(w.wt_max[r[u]]) : ld_scale(w.wt_scale + r[u]);
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            if (r[u] < 0)
                continue;
            unsigned long long x = divide(v[u], s[u]);
            if (logs) {
                if (x == kFxOne)
                    x = 0ull;  // log(1) = +0
                else if (x < kFxOne && (x >> 52) != 0ull)
                    x = log_below_one(x, s_log);
                else
                    x = fx_bits(log(fx_double(x)));
            }
            __stcs(out + (p0 + u * stride), x);
        }
    }
}

template <bool kThin>
__global__ void __launch_bounds__(kThreads) k_wt_out(const Work *__restrict__ W)
{
    __shared__ LogEntry s_log[512];
    wt_out<kThin>(*W, s_log);
}

// A small matrix: the thin form in one cluster, with cluster barriers between
// the steps.
__global__ void __cluster_dims__(8, 1, 1) __launch_bounds__(1024)
    k_wt_cluster(const Work *__restrict__ W)
{
    __shared__ LogEntry s_log[512];
    const Work &w = *W;
    wt_reset(w);
    cluster_sync();
    wt_thin_check(w);
    cluster_sync();
    wt_thin_rowmax(w);
    cluster_sync();
    wt_out<true>(w, s_log);
}

}  // namespace

void launch_weights(const Work *d, const Shape &sh, bool thin, Sink &k)
{
    void *a[] = {(void *)&d};
    const unsigned grid = (unsigned)(sh.num_sms * 8);
    if (sh.cluster) {
        k.launch((const void *)k_wt_cluster, 8, 1024, a);
        return;
    }
    k.launch((const void *)k_wt_reset, grid, kThreads, a);
    if (thin) {
        k.launch((const void *)k_wt_thin_check, 2 * grid, kThreads, a);
        k.launch((const void *)k_wt_thin_rowmax, 2 * grid, kThreads, a);
        k.launch((const void *)k_wt_out<true>, 2 * grid, kThreads, a);
        return;
    }
    launch_check_mark(d, sh, k);
    k.launch((const void *)k_wt_colmax, 2 * grid, kThreads, a);
    k.launch((const void *)k_wt_scale, grid, kThreads, a);
    k.launch((const void *)k_wt_rowmax, 2 * grid, kThreads, a);
    k.launch((const void *)k_wt_scale, grid, kThreads, a);
    k.launch((const void *)k_wt_out<false>, 2 * grid, kThreads, a);
}

}  // namespace awpm

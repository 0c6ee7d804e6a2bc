// Host side of libawpm: contexts and the synchronous C ABI of include/awpm.h.
//
// A context owns a device workspace sized for the largest problem seen, the
// staging buffers for host-resident inputs, a device-resident problem
// descriptor (Work) and one instantiated CUDA graph per launch shape.  One
// solve is: write the descriptor, launch the graph (validation and
// initialisation; a conditional WHILE node whose body is one pass of Steps
// A-D, the control kernel at the end of the body deciding on the device
// whether another pass runs, Algorithm 2; the final weight reduction), copy
// the results back.  The host waits once, at the end.  Because every kernel
// reads the problem from the descriptor and runs a GPU-sized grid, the same
// graph serves every problem of the context.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <vector>

#include "awpm.h"
#include "awpm_ctx.h"
#include "awpm_internal.h"

using namespace awpm;

namespace awpm {

thread_local char g_last_error[512] = "";

void note_cuda_error(cudaError_t e, const char *what, int line)
{
    snprintf(g_last_error, sizeof(g_last_error), "%s (%s) at line %d: %s", cudaGetErrorName(e),
             what, line, cudaGetErrorString(e));
}

}  // namespace awpm

namespace {

#define CUDA_TRY(x)                                                        \
    do {                                                                   \
        cudaError_t e_ = (x);                                              \
        if (e_ != cudaSuccess) {                                           \
            note_cuda_error(e_, #x, __LINE__);                             \
            return e_ == cudaErrorMemoryAllocation ? AWPM_ERR_OOM          \
                                                   : AWPM_ERR_CUDA;        \
        }                                                                  \
    } while (0)

#define AWPM_TRY(x)            \
    do {                       \
        int rc_ = (x);         \
        if (rc_ != AWPM_OK)    \
            return rc_;        \
    } while (0)

// Largest nnz served by the hash lookup (slot 2 * position in int32).
constexpr int32_t kMaxHashNnz = (1 << 30) - 1;
constexpr int kLookahead = 2;
constexpr int kRing = 4;

void release(awpm_ctx *c, DevBuf &b)
{
    if (b.p) {
        cudaFree(b.p);
        c->held -= b.bytes;
        b.p = nullptr;
        b.bytes = 0;
    }
}

// Give back the buffers of the faster paths if the call does not use them.
// True if that made room.
bool release_spares(awpm_ctx *c)
{
    if (c->spares_used || !(c->incbuf.p || c->smallbuf.p || c->b_order.p))
        return false;
    release(c, c->incbuf);
    release(c, c->smallbuf);
    release(c, c->b_order);
    return true;
}

int ensure(awpm_ctx *c, DevBuf &b, size_t bytes)
{
    if (bytes == 0)
        bytes = 16;
    if (b.bytes >= bytes)
        return AWPM_OK;
    release(c, b);
    c->injected = false;
    size_t want = bytes + bytes / 8;  // headroom against small growth steps
    if (c->opt.mem_budget_bytes && c->held + want > c->opt.mem_budget_bytes) {
        want = bytes;
        if (c->held + want > c->opt.mem_budget_bytes &&
            (!release_spares(c) || c->held + want > c->opt.mem_budget_bytes))
            return AWPM_ERR_BUDGET;
    }
    if (c->fail_after >= 0) {  // injected failure (awpm_inject_alloc_failure)
        if (c->fail_after == 0) {
            c->fail_after = -1;
            c->injected = true;
            return AWPM_ERR_OOM;
        }
        --c->fail_after;
    }
    void *p = nullptr;
    cudaError_t e = cudaMalloc(&p, want);
    if (e == cudaErrorMemoryAllocation && release_spares(c)) {
        cudaGetLastError();
        e = cudaMalloc(&p, want);
    }
    if (e != cudaSuccess) {
        note_cuda_error(e, "cudaMalloc", __LINE__);
        cudaGetLastError();
        return AWPM_ERR_OOM;
    }
    b.p = p;
    b.bytes = want;
    c->held += want;
    if (c->held > c->peak)
        c->peak = c->held;
    return AWPM_OK;
}

// 1 = device memory of the context's GPU, 0 = host memory, -1 = another GPU.
int where(const awpm_ctx *c, const void *p)
{
    if (!p)
        return 0;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    if (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) {
        if (a.type == cudaMemoryTypeDevice && a.device != c->device)
            return -1;
        return 1;
    }
    return 0;
}

// Bloom filters of the long columns with the binary-search lookup (default
// on; the environment variable AWPM_BLOOM=0 switches them off, a tuning knob:
// results are the same either way).
bool bloom_enabled()
{
    static const bool on = [] {
        const char *v = getenv("AWPM_BLOOM");
        return !(v && v[0] == '0' && v[1] == 0);
    }();
    return on;
}

// Tiles from which a solve's later passes are incremental (the environment
// variable AWPM_INC overrides it, a tuning knob: 0 never, 1 always; results
// are the same either way).
constexpr int32_t kIncTiles = 98304;
int32_t inc_min_tiles()
{
    static const int32_t least = [] {
        const char *v = getenv("AWPM_INC");
        if (v && (v[0] == '0' || v[0] == '1') && v[1] == 0)
            return v[0] == '0' ? 0x7fffffff : 0;
        return kIncTiles;
    }();
    return least;
}

// Largest n tried without reading the number of entries first (a round trip
// of about 10 us): above, an average column of 20 entries is too many.
constexpr int32_t kSmallOneN = 2048;

// Whether small matrices are solved by a block (or a cluster) each: where the
// rules say so (1), never (0), or every batch whose matrices fit (2).  The
// environment variable AWPM_SMALL=0 or 1, read when a context is made, selects
// the latter two (a tuning knob: results are the same either way).
int small_mode()
{
    const char *v = getenv("AWPM_SMALL");
    return v && v[0] == '0' && v[1] == 0 ? 0 : v && v[0] == '1' && v[1] == 0 ? 2 : 1;
}

// Whether greedy and maximum matching and the weights of small problems run in
// one cluster (default on; the environment variable AWPM_CLUSTER=0, read when a
// context is made, switches it off, a tuning knob: results are the same either
// way).
bool cluster_enabled()
{
    const char *v = getenv("AWPM_CLUSTER");
    return !(v && v[0] == '0' && v[1] == 0);
}

int code_of(unsigned err)
{
    return awpm_code_of_bits(err);
}

int check_sink(const Sink &k)
{
    if (k.err != cudaSuccess) {
        note_cuda_error(k.err, "kernel launch", __LINE__);
        cudaGetLastError();
        return AWPM_ERR_CUDA;
    }
    return AWPM_OK;
}

// Index of a lookup in the per-lookup tables: binary search, hash, row marking.
int lookup_slot(int lookup)
{
    return lookup == AWPM_LOOKUP_HASH ? 1 : lookup == AWPM_LOOKUP_ROWMARK ? 2 : 0;
}

Shape shape_of(const awpm_ctx *c, bool batch, int lookup, bool wide, int32_t ntiles)
{
    Shape sh;
    sh.num_sms = c->num_sms;
    sh.batch = batch;
    sh.lookup = lookup;
    sh.wide = wide;
    sh.search_bps = c->search_bps[batch ? 1 : 0][lookup_slot(lookup)][wide ? 1 : 0];
    sh.search_waves = search_waves(sh.num_sms, sh.search_bps, ntiles);
    sh.select = c->opt.select == AWPM_SELECT_GREEDY ? AWPM_SELECT_GREEDY : AWPM_SELECT_STEP_D;
    return sh;
}

// Append one pass to `sb` (the search, the selection and the flip, which
// decides whether another pass runs: handle h).  The greedy selection's rounds
// are a WHILE node nested in it.
int add_pass(const Work *d, const Shape &sh, bool first, cudaGraphConditionalHandle h, Sink &sb)
{
    cudaError_t e;
    if (first || !sh.inc)
        launch_search(d, sh, sb);
    else
        launch_search_inc(d, sh, sb);
    if (sh.select == AWPM_SELECT_GREEDY) {
        cudaGraphConditionalHandle h2;
        cudaGraphNodeParams cp2 = {cudaGraphNodeTypeConditional};
        cudaGraphNode_t n_inner;
        if ((e = cudaGraphConditionalHandleCreate(&h2, sb.graph, 0, 0)) != cudaSuccess) {
            note_cuda_error(e, "inner conditional handle", __LINE__);
            return AWPM_ERR_CUDA;
        }
        launch_greedy_select_begin(d, sh, true, h2, sb);
        cp2.conditional.handle = h2;
        cp2.conditional.type = cudaGraphCondTypeWhile;
        cp2.conditional.size = 1;
        if (sb.err != cudaSuccess ||
            (e = cudaGraphAddNode(&n_inner, sb.graph, &sb.last, nullptr, 1, &cp2)) !=
                cudaSuccess) {
            note_cuda_error(sb.err != cudaSuccess ? sb.err : e, "inner conditional node",
                            __LINE__);
            return AWPM_ERR_CUDA;
        }
        Sink sr;
        sr.graph = cp2.conditional.phGraph_out[0];
        launch_greedy_select_round(d, sh, true, h2, sr);
        if (sr.err != cudaSuccess) {
            note_cuda_error(sr.err, "selection round nodes", __LINE__);
            return AWPM_ERR_CUDA;
        }
        sb.last = n_inner;
        launch_greedy_select_end_and_flip(d, sh, sb);
    } else if (!sh.batch) {
        // the flip's last block ends the pass (no control kernel)
        launch_select_flip_control_graph(d, sh, h, sb);
    } else {
        launch_select_and_flip(d, sh, sb);
    }
    if (sh.batch || sh.select == AWPM_SELECT_GREEDY)
        launch_control(d, sh, true, h, sb);
    if (sb.err != cudaSuccess) {
        note_cuda_error(sb.err, "pass nodes", __LINE__);
        return AWPM_ERR_CUDA;
    }
    return AWPM_OK;
}

int ilog2(int64_t x)
{
    int l = 0;
    while (x > 1) {
        x >>= 1;
        ++l;
    }
    return l;
}

// The solve graph of one launch shape: initialisation, WHILE{pass}, final
// sum, assembled node by node (no stream capture).  With incremental passes
// the first pass, whose search is another kernel, stands before the WHILE.
int build_graph(awpm_ctx *c, const Shape &sh, cudaGraphExec_t *out)
{
    const Work *d = (const Work *)c->d_work.p;
    cudaGraph_t top = nullptr, g_init = nullptr, g_final = nullptr;
    cudaGraphNode_t n_init, n_cond, n_final;
    cudaGraphConditionalHandle h;
    cudaGraphNodeParams cp = {cudaGraphNodeTypeConditional};
    int rc = AWPM_OK;
    cudaError_t e;
    Sink si, sf, sb;
    if ((e = cudaGraphCreate(&g_init, 0)) != cudaSuccess ||
        (e = cudaGraphCreate(&g_final, 0)) != cudaSuccess ||
        (e = cudaGraphCreate(&top, 0)) != cudaSuccess) {
        note_cuda_error(e, "cudaGraphCreate", __LINE__);
        rc = AWPM_ERR_CUDA;
        goto done;
    }
    si.graph = g_init;
    launch_init(d, sh, si);
    launch_weight_sum(d, sh, false, si);
    sf.graph = g_final;
    launch_weight_sum(d, sh, true, sf);
    if (si.err != cudaSuccess || sf.err != cudaSuccess) {
        note_cuda_error(si.err != cudaSuccess ? si.err : sf.err, "kernel nodes", __LINE__);
        rc = AWPM_ERR_CUDA;
        goto done;
    }
    if ((e = cudaGraphAddChildGraphNode(&n_init, top, nullptr, 0, g_init)) != cudaSuccess ||
        (e = cudaGraphConditionalHandleCreate(&h, top, 1, cudaGraphCondAssignDefault)) !=
            cudaSuccess) {
        note_cuda_error(e, "graph assembly", __LINE__);
        rc = AWPM_ERR_CUDA;
        goto done;
    }
    cp.conditional.handle = h;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    if (sh.inc) {
        Sink s1;
        s1.graph = top;
        s1.last = n_init;
        if ((rc = add_pass(d, sh, true, h, s1)) != AWPM_OK)
            goto done;
        n_init = s1.last;
    }
    if ((e = cudaGraphAddNode(&n_cond, top, &n_init, nullptr, 1, &cp)) != cudaSuccess) {
        note_cuda_error(e, "conditional node", __LINE__);
        rc = AWPM_ERR_CUDA;
        goto done;
    }
    sb.graph = cp.conditional.phGraph_out[0];
    if ((rc = add_pass(d, sh, false, h, sb)) != AWPM_OK)
        goto done;
    if ((e = cudaGraphAddChildGraphNode(&n_final, top, &n_cond, 1, g_final)) != cudaSuccess ||
        (e = cudaGraphInstantiate(out, top, 0)) != cudaSuccess) {
        note_cuda_error(e, "graph instantiation", __LINE__);
        *out = nullptr;
        rc = AWPM_ERR_CUDA;
        goto done;
    }
done:
    if (top)
        cudaGraphDestroy(top);
    if (g_init)
        cudaGraphDestroy(g_init);
    if (g_final)
        cudaGraphDestroy(g_final);
    cudaGetLastError();
    return rc;
}

// Graph of the greedy maximal matching: state reset and input checks, a
// conditional WHILE node over the rounds, the matched-weight sum.
int build_greedy_graph(awpm_ctx *c, const Shape &sh, cudaGraphExec_t *out)
{
    const Work *d = (const Work *)c->d_work.p;
    cudaGraph_t top = nullptr, g_init = nullptr, g_final = nullptr;
    cudaGraphNode_t n_init, n_cond, n_final;
    cudaGraphConditionalHandle h;
    cudaGraphNodeParams cp = {cudaGraphNodeTypeConditional};
    int rc = AWPM_OK;
    cudaError_t e;
    Sink si, sf, sb;
    if ((e = cudaGraphCreate(&g_init, 0)) != cudaSuccess ||
        (e = cudaGraphCreate(&g_final, 0)) != cudaSuccess ||
        (e = cudaGraphCreate(&top, 0)) != cudaSuccess) {
        note_cuda_error(e, "cudaGraphCreate", __LINE__);
        rc = AWPM_ERR_CUDA;
        goto done;
    }
    si.graph = g_init;
    launch_greedy_init(d, sh, si);
    sf.graph = g_final;
    launch_weight_sum(d, sh, true, sf);
    if (si.err != cudaSuccess || sf.err != cudaSuccess) {
        note_cuda_error(si.err != cudaSuccess ? si.err : sf.err, "kernel nodes", __LINE__);
        rc = AWPM_ERR_CUDA;
        goto done;
    }
    if (sh.cluster) {
        // a straight line: the rounds are one kernel
        launch_greedy_cluster(d, sh, si);
        launch_weight_sum(d, sh, true, si);
        if ((e = si.err) != cudaSuccess || (e = cudaGraphInstantiate(out, g_init, 0)) != cudaSuccess) {
            note_cuda_error(e, "greedy graph", __LINE__);
            *out = nullptr;
            rc = AWPM_ERR_CUDA;
        }
        goto done;
    }
    if ((e = cudaGraphAddChildGraphNode(&n_init, top, nullptr, 0, g_init)) != cudaSuccess ||
        (e = cudaGraphConditionalHandleCreate(&h, top, 1, cudaGraphCondAssignDefault)) !=
            cudaSuccess) {
        note_cuda_error(e, "graph assembly", __LINE__);
        rc = AWPM_ERR_CUDA;
        goto done;
    }
    cp.conditional.handle = h;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    if ((e = cudaGraphAddNode(&n_cond, top, &n_init, nullptr, 1, &cp)) != cudaSuccess) {
        note_cuda_error(e, "conditional node", __LINE__);
        rc = AWPM_ERR_CUDA;
        goto done;
    }
    sb.graph = cp.conditional.phGraph_out[0];
    launch_greedy_round(d, sh, true, h, sb);
    if (sb.err != cudaSuccess) {
        note_cuda_error(sb.err, "round body nodes", __LINE__);
        rc = AWPM_ERR_CUDA;
        goto done;
    }
    if ((e = cudaGraphAddChildGraphNode(&n_final, top, &n_cond, 1, g_final)) != cudaSuccess ||
        (e = cudaGraphInstantiate(out, top, 0)) != cudaSuccess) {
        note_cuda_error(e, "graph instantiation", __LINE__);
        *out = nullptr;
        rc = AWPM_ERR_CUDA;
        goto done;
    }
done:
    if (top)
        cudaGraphDestroy(top);
    if (g_init)
        cudaGraphDestroy(g_init);
    if (g_final)
        cudaGraphDestroy(g_final);
    cudaGetLastError();
    return rc;
}

// Graph of the maximum cardinality matching: load and checks; a WHILE node
// over the phases whose body starts a phase, runs a WHILE node over the
// levels, augments and decides whether to continue; the result stored.
int build_mcm_graph(awpm_ctx *c, const Shape &sh, cudaGraphExec_t *out)
{
    const Work *d = (const Work *)c->d_work.p;
    cudaGraph_t top = nullptr, g_init = nullptr, g_final = nullptr;
    cudaGraphNode_t n_init, n_cond, n_final, n_inner;
    cudaGraphConditionalHandle h1, h2;
    cudaGraphNodeParams cp = {cudaGraphNodeTypeConditional};
    cudaGraphNodeParams cp2 = {cudaGraphNodeTypeConditional};
    int rc = AWPM_OK;
    cudaError_t e;
    Sink si, sf, sb, sl;
    if ((e = cudaGraphCreate(&g_init, 0)) != cudaSuccess ||
        (e = cudaGraphCreate(&g_final, 0)) != cudaSuccess ||
        (e = cudaGraphCreate(&top, 0)) != cudaSuccess) {
        note_cuda_error(e, "cudaGraphCreate", __LINE__);
        rc = AWPM_ERR_CUDA;
        goto done;
    }
    si.graph = g_init;
    launch_mcm_load(d, sh, si);
    sf.graph = g_final;
    launch_mcm_store(d, sh, sf);
    if (si.err != cudaSuccess || sf.err != cudaSuccess) {
        note_cuda_error(si.err != cudaSuccess ? si.err : sf.err, "kernel nodes", __LINE__);
        rc = AWPM_ERR_CUDA;
        goto done;
    }
    if (sh.cluster) {
        // a straight line: the phases and levels are one kernel
        launch_mcm_cluster(d, sh, si);
        launch_mcm_store(d, sh, si);
        if ((e = si.err) != cudaSuccess || (e = cudaGraphInstantiate(out, g_init, 0)) != cudaSuccess) {
            note_cuda_error(e, "maximum matching graph", __LINE__);
            *out = nullptr;
            rc = AWPM_ERR_CUDA;
        }
        goto done;
    }
    if ((e = cudaGraphAddChildGraphNode(&n_init, top, nullptr, 0, g_init)) != cudaSuccess ||
        (e = cudaGraphConditionalHandleCreate(&h1, top, 1, cudaGraphCondAssignDefault)) !=
            cudaSuccess) {
        note_cuda_error(e, "graph assembly", __LINE__);
        rc = AWPM_ERR_CUDA;
        goto done;
    }
    cp.conditional.handle = h1;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    if ((e = cudaGraphAddNode(&n_cond, top, &n_init, nullptr, 1, &cp)) != cudaSuccess) {
        note_cuda_error(e, "phase node", __LINE__);
        rc = AWPM_ERR_CUDA;
        goto done;
    }
    sb.graph = cp.conditional.phGraph_out[0];
    if ((e = cudaGraphConditionalHandleCreate(&h2, sb.graph, 0, 0)) != cudaSuccess) {
        note_cuda_error(e, "level handle", __LINE__);
        rc = AWPM_ERR_CUDA;
        goto done;
    }
    launch_mcm_phase(d, sh, sb);
    launch_mcm_cond_level(d, sh, h2, sb);
    cp2.conditional.handle = h2;
    cp2.conditional.type = cudaGraphCondTypeWhile;
    cp2.conditional.size = 1;
    if (sb.err != cudaSuccess ||
        (e = cudaGraphAddNode(&n_inner, sb.graph, &sb.last, nullptr, 1, &cp2)) != cudaSuccess) {
        note_cuda_error(sb.err != cudaSuccess ? sb.err : e, "level node", __LINE__);
        rc = AWPM_ERR_CUDA;
        goto done;
    }
    sl.graph = cp2.conditional.phGraph_out[0];
    launch_mcm_level_graph(d, sh, h2, sl);
    sb.last = n_inner;
    launch_mcm_augment(d, sh, sb);
    launch_mcm_cond_phase(d, sh, h1, sb);
    if (sb.err != cudaSuccess || sl.err != cudaSuccess) {
        note_cuda_error(sb.err != cudaSuccess ? sb.err : sl.err, "phase body nodes", __LINE__);
        rc = AWPM_ERR_CUDA;
        goto done;
    }
    if ((e = cudaGraphAddChildGraphNode(&n_final, top, &n_cond, 1, g_final)) != cudaSuccess ||
        (e = cudaGraphInstantiate(out, top, 0)) != cudaSuccess) {
        note_cuda_error(e, "graph instantiation", __LINE__);
        *out = nullptr;
        rc = AWPM_ERR_CUDA;
        goto done;
    }
done:
    if (top)
        cudaGraphDestroy(top);
    if (g_init)
        cudaGraphDestroy(g_init);
    if (g_final)
        cudaGraphDestroy(g_final);
    cudaGetLastError();
    return rc;
}

int ensure_timing_events(awpm_ctx *c, size_t pairs)
{
    while (c->tev.size() < 2 * pairs) {
        cudaEvent_t ev;
        CUDA_TRY(cudaEventCreate(&ev));
        c->tev.push_back(ev);
    }
    return AWPM_OK;
}

// Host-driven pass loop (AWPM_FLAG_TIME_SEARCH): CUDA events around every
// search launch; the host stays kLookahead passes ahead of the device and
// stops enqueueing once a finished pass reports that the loop ended.  Passes
// enqueued after the end are no-ops (every kernel checks ctl->active).
int run_timed(awpm_ctx *c, const Shape &sh, int max_passes, int *passes_enqueued)
{
    cudaStream_t s = c->stream;
    const Work *d = (const Work *)c->d_work.p;
    Ctl *ctl = (Ctl *)c->ctl.p;
    Sink k;
    k.stream = s;
    launch_init(d, sh, k);
    launch_weight_sum(d, sh, false, k);
    AWPM_TRY(check_sink(k));
    int t = 0;
    for (; t < max_passes; ++t) {
        if (t >= kLookahead) {
            const int slot = (t - kLookahead) % kRing;
            CUDA_TRY(cudaEventSynchronize(c->flagev[slot]));
            if (!c->h_active[slot])
                break;
        }
        NvtxRange pass_range("pass");
        AWPM_TRY(ensure_timing_events(c, (size_t)t + 1));
        CUDA_TRY(cudaEventRecord(c->tev[2 * t], s));
        if (t > 0 && sh.inc)
            launch_search_inc(d, sh, k);
        else
            launch_search(d, sh, k);
        CUDA_TRY(cudaEventRecord(c->tev[2 * t + 1], s));
        if (sh.select == AWPM_SELECT_GREEDY) {
            // the selection's rounds, driven from the host by the count of
            // undecided winners
            launch_greedy_select_begin(d, sh, false, cudaGraphConditionalHandle(), k);
            for (;;) {
                AWPM_TRY(check_sink(k));
                CUDA_TRY(cudaMemcpyAsync(&c->h_ctl->live, &ctl->live, sizeof(int32_t),
                                         cudaMemcpyDeviceToHost, s));
                CUDA_TRY(cudaStreamSynchronize(s));
                const int32_t live = c->h_ctl->live;
                CUDA_TRY(cudaMemsetAsync(&ctl->live, 0, sizeof(int32_t), s));
                if (live <= 0)
                    break;
                launch_greedy_select_round(d, sh, false, cudaGraphConditionalHandle(), k);
            }
            launch_greedy_select_end_and_flip(d, sh, k);
        } else {
            launch_select_and_flip(d, sh, k);
        }
        launch_control(d, sh, false, cudaGraphConditionalHandle(), k);
        AWPM_TRY(check_sink(k));
        CUDA_TRY(cudaMemcpyAsync(&c->h_active[t % kRing], &ctl->active, sizeof(int32_t),
                                 cudaMemcpyDeviceToHost, s));
        CUDA_TRY(cudaEventRecord(c->flagev[t % kRing], s));
    }
    launch_weight_sum(d, sh, true, k);
    AWPM_TRY(check_sink(k));
    *passes_enqueued = t;
    return AWPM_OK;
}

template <typename T>
int stage_in(awpm_ctx *c, DevBuf &buf, const T *src, size_t count, int loc, const T **out)
{
    if (loc == 1) {
        *out = src;
        return AWPM_OK;
    }
    AWPM_TRY(ensure(c, buf, sizeof(T) * count));
    if (count)
        CUDA_TRY(cudaMemcpyAsync(buf.p, src, sizeof(T) * count, cudaMemcpyHostToDevice, c->stream));
    *out = (const T *)buf.p;
    return AWPM_OK;
}

std::mutex g_default_mu;
std::map<int, awpm_ctx *> g_default;

}  // namespace

namespace awpm {

// Layout of the incremental passes' buffer (byte offsets, each 256-byte
// aligned): entry bits twice, old rows, and two sets of bitmaps.
struct IncLayout {
    size_t found, pos, mc_old, small[2], large[2], full[2], posi[2], mark[2], bytes;
    int32_t map_bits;  // of the large folded bitmap (0: none)
    IncLayout(int32_t n, int32_t ntiles)
    {
        size_t at = 0;
        auto take = [&at](size_t b) {
            const size_t o = at;
            at += (b + 255) / 256 * 256;
            return o;
        };
        map_bits = 0;
        if (n > kMapSmallBits)
            for (map_bits = kMapSmallBits; map_bits < n && map_bits < kMapLargeBits;)
                map_bits *= 2;
        found = take(4 * ((size_t)ntiles + 1));
        pos = take(4 * ((size_t)ntiles + 1));
        mc_old = take(4 * (size_t)n);
        for (int x = 0; x < 2; ++x) {
            small[x] = take(kMapSmallBits / 8);
            large[x] = take((size_t)map_bits / 8);
            full[x] = take(4 * ((size_t)n / 32 + 2));
            posi[x] = take(4 * ((size_t)n / 32 + 2));
            mark[x] = take(4 * ((size_t)ntiles / 32 + 1));
        }
        bytes = at;
    }
};

size_t ctx_bytes_needed(int32_t n, int32_t nnz, bool host_inputs, int lookup, int select,
                        bool least)
{
    const size_t N = (size_t)n, Z = (size_t)nnz, T = Z / kTile + 1;
    size_t b = N * (4 + 4 + 8 + sizeof(RowRange) + 8 + 8 + sizeof(Rec) + sizeof(Sel) + 4) + N / 8 +
               4 * T +
               4 * (Z / 32 + 1) + sizeof(Ctl) + 8 * kWsumBlocks;
    if (lookup != AWPM_LOOKUP_BSEARCH)  // hash tables (AUTO may pick them)
        b += 16 * Z;
    if (lookup != AWPM_LOOKUP_HASH && lookup != AWPM_LOOKUP_ROWMARK)  // Bloom filters
        b += Z + 4;
    if (lookup == AWPM_LOOKUP_ROWMARK)  // marks, transpose, radix-sort buffers
        b += 12 * N + 4 + 16 * Z + 4 * (size_t)kRsBins * (Z / kRsTile + 1) + 4 * kRsBins;
    if (host_inputs)
        b += 4 * (N + 1) + 12 * Z + 8 * N;
    if (select == AWPM_SELECT_GREEDY)  // selection records and three bitmaps
        b += sizeof(Sel) * N + 3 * 4 * (N / 32 + 1);
    if (!least)
        b += IncLayout(n, (int32_t)T).bytes;
    return b + b / 8;
}

size_t ctx_bytes_held(const awpm_ctx *c)
{
    return c->held;
}

void ctx_trim(awpm_ctx *c)
{
    DevBuf *bufs[] = {&c->mc,      &c->mr,       &c->wm,       &c->rr,       &c->rsig,
                      &c->colsig,  &c->best,     &c->dsel,     &c->tile_col, &c->starts,
                      &c->wpart,   &c->htab,     &c->b_noff,   &c->b_colmat, &c->b_tilemat,
                      &c->b_tlist, &c->b_i32,    &c->b_u64,    &c->b_f64,    &c->s_colptr,
                      &c->s_rowidx, &c->s_w,     &c->s_mate,   &c->s_out,    &c->s_gain,
                      &c->s_row,   &c->winbits,  &c->wkey,     &c->bloom, &c->incbuf,
                      &c->smallbuf, &c->b_order,
                      &c->gmate,   &c->gdead,
                      &c->psel,    &c->pslive,   &c->pstaken,  &c->psused,   &c->wt_max,
                      &c->wt_scale, &c->wt_stage, &c->mroot,   &c->mrpar,    &c->mfront,
                      &c->mreach,  &c->mtmark,   &c->mfl,      &c->mroff,    &c->mtend,
                      &c->mtouch,
                      &c->mstage,  &c->mcolof,   &c->mtiles,   &c->rowsig,   &c->trowptr,
                      &c->rs_k0,   &c->rs_k1,    &c->rs_v0,    &c->rs_v1,    &c->rs_hist,
                      &c->rs_sums};
    if (c->stream)
        cudaStreamSynchronize(c->stream);
    for (DevBuf *b : bufs)
        release(c, *b);
    c->rec_clean = 0;
    cudaGetLastError();
}

int setup_ctx(awpm_ctx *c, const awpm_options *opt)
{
    if (opt)
        c->opt = *opt;
    else
        awpm_default_options(&c->opt);
    if (c->opt.max_iters < 0 || c->opt.lookup < 0 || c->opt.lookup > 3 || c->opt.slots < 0 ||
        c->opt.select < 0 || c->opt.select > 1)
        return AWPM_ERR_INVALID_ARG;
    int dev = c->opt.device;
    if (dev < 0)
        CUDA_TRY(cudaGetDevice(&dev));
    c->device = dev;
    CUDA_TRY(cudaSetDevice(dev));
    CUDA_TRY(cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, dev));
    CUDA_TRY(search_inc_setup());
    CUDA_TRY(small_setup());
    c->search_wide = default_search_wide();
    c->small_mode = small_mode();
    c->clusters = cluster_enabled();
    for (int b = 0; b < 2; ++b)
        for (int p = 0; p < 2; ++p) {
            c->search_bps[b][0][p] = search_blocks_per_sm(AWPM_LOOKUP_BSEARCH, b == 1, p == 1);
            c->search_bps[b][1][p] = search_blocks_per_sm(AWPM_LOOKUP_HASH, b == 1, p == 1);
            c->search_bps[b][2][p] = search_blocks_per_sm(AWPM_LOOKUP_ROWMARK, b == 1, p == 1);
        }
    if (c->opt.stream) {
        c->stream = (cudaStream_t)c->opt.stream;
        c->own_stream = false;
    } else {
        CUDA_TRY(cudaStreamCreate(&c->stream));
        c->own_stream = true;
    }
    AWPM_TRY(ensure(c, c->d_work, sizeof(Work)));
    CUDA_TRY(cudaMallocHost((void **)&c->h_work, sizeof(Work)));
    CUDA_TRY(cudaMallocHost((void **)&c->h_ctl, sizeof(Ctl)));
    CUDA_TRY(cudaMallocHost((void **)&c->h_active, sizeof(int32_t) * kRing));
    CUDA_TRY(cudaEventCreate(&c->ev_a));
    CUDA_TRY(cudaEventCreate(&c->ev_b));
    for (int i = 0; i < kRing; ++i) {
        cudaEvent_t ev;
        CUDA_TRY(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
        c->flagev.push_back(ev);
    }
    return AWPM_OK;
}

void teardown_ctx(awpm_ctx *c)
{
    if (c->stream)
        cudaStreamSynchronize(c->stream);
    for (int b = 0; b < 2; ++b)
        for (int h = 0; h < 3; ++h)
            for (int p = 0; p < 2; ++p)
                for (int v = 0; v < 2; ++v)
                    for (int q = 0; q < 2; ++q)
                        for (cudaGraphExec_t &g : c->g_exec[b][h][p][v][q])
                            if (g) {
                                cudaGraphExecDestroy(g);
                                g = nullptr;
                            }
    for (int v = 0; v < 3; ++v) {
        if (c->g_greedy[v]) {
            cudaGraphExecDestroy(c->g_greedy[v]);
            c->g_greedy[v] = nullptr;
        }
        if (c->g_mcm[v]) {
            cudaGraphExecDestroy(c->g_mcm[v]);
            c->g_mcm[v] = nullptr;
        }
    }
    DevBuf *bufs[] = {&c->mc,      &c->mr,       &c->wm,       &c->rr,       &c->rsig,
                      &c->colsig,  &c->best,     &c->dsel,     &c->tile_col, &c->starts,
                      &c->ctl,     &c->wpart,    &c->htab,     &c->b_noff,   &c->b_colmat,
                      &c->b_tilemat, &c->b_tlist, &c->b_i32,  &c->b_u64,    &c->b_f64,    &c->s_colptr,
                      &c->s_rowidx, &c->s_w,     &c->s_mate,   &c->s_out,    &c->s_gain,
                      &c->s_row,   &c->d_work,   &c->winbits,  &c->wkey,     &c->bloom, &c->incbuf,
                      &c->smallbuf, &c->b_order,
                      &c->gmate,
                      &c->gdead,  &c->psel,     &c->pslive,   &c->pstaken,  &c->psused,
                      &c->wt_max,  &c->wt_scale, &c->wt_stage,
                      &c->mroot,   &c->mrpar,    &c->mfront,   &c->mreach,   &c->mtmark,
                      &c->mfl,     &c->mroff,
                      &c->mtend,   &c->mtouch,   &c->mstage,   &c->mcolof,
                      &c->mtiles,  &c->rowsig,   &c->trowptr,  &c->rs_k0,    &c->rs_k1,
                      &c->rs_v0,   &c->rs_v1,    &c->rs_hist,  &c->rs_sums};
    for (DevBuf *b : bufs)
        release(c, *b);
    if (c->h_work)
        cudaFreeHost(c->h_work);
    if (c->h_ctl)
        cudaFreeHost(c->h_ctl);
    if (c->h_active)
        cudaFreeHost(c->h_active);
    if (c->h_batch)
        cudaFreeHost(c->h_batch);
    for (cudaEvent_t ev : c->tev)
        cudaEventDestroy(ev);
    for (cudaEvent_t ev : c->flagev)
        cudaEventDestroy(ev);
    if (c->ev_a)
        cudaEventDestroy(c->ev_a);
    if (c->ev_b)
        cudaEventDestroy(c->ev_b);
    if (c->small_streams.fork) {
        for (cudaStream_t s : c->small_streams.side)
            cudaStreamDestroy(s);
        for (cudaEvent_t e : c->small_streams.join)
            cudaEventDestroy(e);
        cudaEventDestroy(c->small_streams.fork);
    }
    if (c->own_stream && c->stream)
        cudaStreamDestroy(c->stream);
    cudaGetLastError();
}

// Room in pinned memory for a batch's per-matrix results (miter, mconv, mnnz
// (i32), mcycles (u64), mw_in, mw_out (f64)).
int ensure_pinned(awpm_ctx *c, int32_t count)
{
    const size_t bytes = (size_t)count * (3 * sizeof(int32_t) + 3 * 8);
    if (c->h_batch_bytes >= bytes)
        return AWPM_OK;
    if (c->h_batch)
        cudaFreeHost(c->h_batch);
    c->h_batch = nullptr;
    c->h_batch_bytes = 0;
    CUDA_TRY(cudaMallocHost(&c->h_batch, bytes));
    c->h_batch_bytes = bytes;
    return AWPM_OK;
}

// Copy a batch's per-matrix results to pinned memory.
int copy_batch_results(awpm_ctx *c, const BatchWork &bw)
{
    const int32_t count = bw.count;
    AWPM_TRY(ensure_pinned(c, count));
    char *hb = (char *)c->h_batch;
    CUDA_TRY(cudaMemcpyAsync(hb, bw.miter, sizeof(int32_t) * 3 * (size_t)count,
                             cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(cudaMemcpyAsync(hb + 12 * (size_t)count, bw.mcycles, 8 * (size_t)count,
                             cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(cudaMemcpyAsync(hb + 20 * (size_t)count, bw.mw_in, 16 * (size_t)count,
                             cudaMemcpyDeviceToHost, c->stream));
    return AWPM_OK;
}

size_t batch_i32_bytes(int32_t count)
{
    return sizeof(int32_t) * (5 * (size_t)count + 2 + kSmallClasses);
}

// Device arrays of a batch's results (or a single small solve's).
int batch_arrays(awpm_ctx *c, BatchWork &bw, int32_t count)
{
    AWPM_TRY(ensure(c, c->b_i32, batch_i32_bytes(count)));
    AWPM_TRY(ensure(c, c->b_u64, sizeof(unsigned long long) * 2 * (size_t)count));
    AWPM_TRY(ensure(c, c->b_f64, sizeof(double) * 2 * (size_t)count));
    bw.count = count;
    int32_t *i32 = (int32_t *)c->b_i32.p;
    bw.mdone = i32;
    bw.miter = i32 + count;
    bw.mconv = i32 + 2 * (size_t)count;
    bw.mnnz = i32 + 3 * (size_t)count;
    bw.active = i32 + 5 * (size_t)count;
    bw.tlist_n = i32 + 5 * (size_t)count + 1;
    unsigned long long *u64 = (unsigned long long *)c->b_u64.p;
    bw.mflips = u64;
    bw.mcycles = u64 + count;
    double *f64 = (double *)c->b_f64.p;
    bw.mw_in = f64;
    bw.mw_out = f64 + count;
    return AWPM_OK;
}

// The matrices of a batch by class and, within a class, roughly from the
// largest to the smallest (buckets of an eighth of an octave), so that the
// last blocks to run have the short solves.  False when the offsets are not
// valid or a matrix is too large.
bool small_batch_order(const int32_t *off, int32_t count, int32_t n, std::vector<int32_t> &order,
                       int32_t *per_class)
{
    constexpr int kBuckets = 8 * 16;
    if (off[0] != 0 || off[count] != n)
        return false;
    std::vector<int32_t> at(kBuckets + 1, 0);
    std::vector<uint8_t> of((size_t)count);
    for (int x = 0; x < kSmallClasses; ++x)
        per_class[x] = 0;
    for (int32_t b = 0; b < count; ++b) {
        const int64_t m = (int64_t)off[b + 1] - off[b];
        if (m < 0 || m > kSmallMaxN[0])
            return false;
        ++per_class[small_class((int32_t)m)];
        // octave and the next three bits, largest first
        const int l = ilog2(m > 8 ? m : 8);
        const int bucket = kBuckets - 1 - (8 * (l - 3) + (int)((m >> (l - 3)) & 7));
        // (class limits fall inside a bucket: the class decides first)
        of[(size_t)b] = (uint8_t)bucket;
        ++at[(size_t)bucket + 1];
    }
    for (int x = 0; x < kBuckets; ++x)
        at[(size_t)x + 1] += at[(size_t)x];
    std::vector<int32_t> by((size_t)count);
    for (int32_t b = 0; b < count; ++b)
        by[(size_t)at[of[(size_t)b]]++] = b;
    int32_t next[kSmallClasses] = {0, per_class[0], per_class[0] + per_class[1]};
    order.resize((size_t)count);
    for (int32_t b : by)
        order[(size_t)next[small_class(off[b + 1] - off[b])]++] = b;
    return true;
}

// The entries of a batch of small matrices (valid offsets): their number into
// *nnz, the tiles of each matrix (its own, rounded up) into *load.  Column
// pointers on the device are read by a kernel that writes them to pinned memory
// (a round trip as for nnz alone; copied back, they made it 5 us longer).
int read_batch(awpm_ctx *c, const Request &r, int l_colptr, int l_off, int32_t *nnz,
               BatchLoad *load)
{
    const size_t count = (size_t)r.count;
    const int32_t *off = r.off_host, *at = nullptr;
    std::vector<int32_t> own;
    if (l_colptr == 1) {
        AWPM_TRY(ensure_pinned(c, r.count));
        int32_t *h = (int32_t *)c->h_batch;  // the pointers, then the offsets
        const int32_t *koff = r.n_off;
        if (l_off != 1) {
            std::memcpy(h + count + 1, off, sizeof(int32_t) * (count + 1));
            koff = h + count + 1;
        }
        Sink k;
        k.stream = c->stream;
        launch_small_entries(koff, r.colptr, r.n, r.count, h, k);
        AWPM_TRY(check_sink(k));
        CUDA_TRY(cudaStreamSynchronize(c->stream));
        at = h;
    } else {
        own.resize(count + 1);
        for (size_t b = 0; b <= count; ++b)
            own[b] = r.colptr[off[b]];
        at = own.data();
    }
    *nnz = at[count];
    for (size_t b = 0; b < count; ++b) {
        const int64_t nz = (int64_t)at[b + 1] - at[b];
        load->add(off[b + 1] - off[b], nz > 0 ? (nz + kTile - 1) / kTile : 0);
    }
    return AWPM_OK;
}

int ctx_enqueue_small(awpm_ctx *c, const Request &r, int32_t nnz, const int32_t *per_class,
                      int l_colptr, int l_rowidx, int l_w, int l_mate, int l_out);

int enqueue_once(awpm_ctx *c, const Request &r);

int ctx_enqueue(awpm_ctx *c, const Request &r)
{
    NvtxRange nvtx_range("enqueue");
    c->spares_used = false;
    c->union_tiles = 0;
    int rc = enqueue_once(c, r);
    const bool no_room = rc == AWPM_ERR_BUDGET || (rc == AWPM_ERR_OOM && !c->injected);
    if (no_room && c->spares_used) {
        if (c->stream)
            CUDA_TRY(cudaStreamSynchronize(c->stream));
        cudaGetLastError();
        c->spares_used = false;
        release_spares(c);
        c->least_memory = true;
        rc = enqueue_once(c, r);
        c->least_memory = false;
    } else if (no_room && c->union_tiles > 0) {
        // a batch that would be the faster as a union: the blocks need less
        const int64_t tiles = c->union_tiles;
        ctx_trim(c);
        if (rc == AWPM_ERR_BUDGET && (c->union_full == 0 || tiles < c->union_full))
            c->union_full = tiles;
        c->force_blocks = true;
        rc = enqueue_once(c, r);
        c->force_blocks = false;
    }
    return rc;
}

int enqueue_once(awpm_ctx *c, const Request &r)
{
    Pending &pd = c->pend;
    pd = Pending();
    const int32_t n = r.n;
    if (n < 0 || (n > 0 && (!r.colptr || !r.mate_in)) ||
        (!r.search_only && n > 0 && !r.mate_out) ||
        (r.search_only && n > 0 && (!r.gain_out || !r.row_out)) || r.count < 0 ||
        (r.count > 0 && !r.n_off))
        return AWPM_ERR_INVALID_ARG;
    CUDA_TRY(cudaSetDevice(c->device));
    pd.lookup = (c->opt.lookup == AWPM_LOOKUP_HASH || c->opt.lookup == AWPM_LOOKUP_ROWMARK)
                    ? c->opt.lookup
                    : AWPM_LOOKUP_BSEARCH;
    pd.search_only = r.search_only;
    if (n == 0) {
        pd.active = true;
        pd.trivial = true;
        return AWPM_OK;
    }
    const int l_colptr = where(c, r.colptr), l_rowidx = where(c, r.rowidx),
              l_w = where(c, r.weight), l_mate = where(c, r.mate_in);
    const int l_out = r.search_only ? 0 : where(c, r.mate_out);
    const int l_gain = r.search_only ? where(c, r.gain_out) : 0;
    const int l_row = r.search_only ? where(c, r.row_out) : 0;
    const int l_off = r.count > 0 ? where(c, r.n_off) : 0;
    if (l_colptr < 0 || l_rowidx < 0 || l_w < 0 || l_mate < 0 || l_out < 0 || l_gain < 0 ||
        l_row < 0 || l_off < 0)
        return AWPM_ERR_INVALID_ARG;

    // Small matrices: a block each of a batch, where that pays, or one cluster
    // for a single one, which does not even have its nnz read back first.
    const bool small = c->small_mode && !c->general_only && !c->least_memory && !r.search_only &&
                       !(c->opt.flags & AWPM_FLAG_TIME_SEARCH) &&
                       c->opt.select == AWPM_SELECT_STEP_D &&
                       (c->opt.lookup == AWPM_LOOKUP_AUTO || c->opt.lookup == AWPM_LOOKUP_BSEARCH) &&
                       r.rowidx && r.weight;
    if (small && r.count == 0 && n <= kSmallOneN) {
        const int32_t known = r.nnz >= 0 ? r.nnz : l_colptr == 1 ? -1 : r.colptr[n];
        // (a size class that once had too many entries has them read first)
        if (known <= kSmallOneNnz &&
            (known >= 0 || (l_rowidx == 1 && l_w == 1 && !((c->small_dense >> ilog2(n)) & 1u))))
            return ctx_enqueue_small(c, r, known, nullptr, l_colptr, l_rowidx, l_w, l_mate, l_out);
    }

    int32_t nnz = r.nnz;
    int32_t per_class[kSmallClasses];
    const bool small_batch = small && r.count > 0 && r.off_host &&
                             small_batch_order(r.off_host, r.count, n, pd.order, per_class);
    bool blocks = false;
    if (small_batch) {
        BatchLoad load;
        AWPM_TRY(read_batch(c, r, l_colptr, l_off, &nnz, &load));
        blocks = c->small_mode == 2 || c->force_blocks || load.blocks_pay() ||
                 (c->union_full > 0 && load.all >= c->union_full);
        c->union_tiles = blocks ? 0 : load.all;
    }
    if (nnz < 0 && !small_batch) {
        if (l_colptr == 1) {
            CUDA_TRY(cudaMemcpyAsync(c->h_ctl, r.colptr + n, sizeof(int32_t),
                                     cudaMemcpyDeviceToHost, c->stream));
            CUDA_TRY(cudaStreamSynchronize(c->stream));
            std::memcpy(&nnz, c->h_ctl, sizeof(int32_t));
        } else {
            nnz = r.colptr[n];
        }
    }
    if (nnz < 0 || nnz > kMaxEntries || (nnz > 0 && (!r.rowidx || !r.weight)))
        return AWPM_ERR_INVALID_ARG;
    if (small && r.count == 0 && n <= kSmallMaxN[0] && nnz <= kSmallOneNnz)
        return ctx_enqueue_small(c, r, nnz, nullptr, l_colptr, l_rowidx, l_w, l_mate, l_out);
    if (blocks)
        return ctx_enqueue_small(c, r, nnz, per_class, l_colptr, l_rowidx, l_w, l_mate, l_out);
    const bool timed = (c->opt.flags & AWPM_FLAG_TIME_SEARCH) != 0;
    // launch configuration: given, or the autotuner's (AWPM_LOOKUP_AUTO)
    int lookup = pd.lookup;
    bool wide = c->search_wide;
    if (c->opt.lookup == AWPM_LOOKUP_AUTO && !r.search_only && !timed) {
        const uint64_t key = ((uint64_t)(r.count > 0) << 62) | ((uint64_t)ilog2(n) << 32) |
                             (uint64_t)ilog2(nnz > 0 ? nnz : 1);
        TuneEntry &te = c->tune[key];
        const int cfg = te.chosen >= 0 ? te.chosen : te.trials;
        lookup = kTune[cfg].lookup;
        wide = kTune[cfg].wide;
        if (te.chosen < 0) {
            pd.tune_cfg = cfg;
            pd.tune_key = key;
        }
    }
    // hash slots are addressed as 2 * position in int32
    if (lookup == AWPM_LOOKUP_HASH && nnz > kMaxHashNnz)
        lookup = AWPM_LOOKUP_BSEARCH;
    pd.lookup = lookup;
    const int32_t ntiles = (int32_t)(((int64_t)nnz + kTile - 1) / kTile);
    const int32_t max_passes = c->opt.max_iters > 0 ? c->opt.max_iters : AWPM_PASS_CAP;
    const int32_t count = r.count;

    AWPM_TRY(ensure(c, c->mc, sizeof(int32_t) * n));
    AWPM_TRY(ensure(c, c->mr, sizeof(int32_t) * n));
    AWPM_TRY(ensure(c, c->wm, sizeof(double) * n));
    AWPM_TRY(ensure(c, c->rr, sizeof(RowRange) * n));
    AWPM_TRY(ensure(c, c->rsig, sizeof(unsigned long long) * n));
    AWPM_TRY(ensure(c, c->colsig, sizeof(unsigned long long) * n));
    const void *best_was = c->best.p, *dsel_was = c->dsel.p;
    AWPM_TRY(ensure(c, c->best, sizeof(Rec) * n));
    AWPM_TRY(ensure(c, c->dsel, sizeof(Sel) * n));
    if (c->best.p != best_was || c->dsel.p != dsel_was)
        c->rec_clean = 0;
    AWPM_TRY(ensure(c, c->winbits, sizeof(uint32_t) * ((size_t)n / 32 + 1)));
    AWPM_TRY(ensure(c, c->wkey, sizeof(int32_t) * n));
    AWPM_TRY(ensure(c, c->tile_col, sizeof(int32_t) * ((size_t)ntiles + 1)));
    AWPM_TRY(ensure(c, c->starts, sizeof(uint32_t) * (((size_t)nnz + 31) / 32 + 1)));
    AWPM_TRY(ensure(c, c->ctl, sizeof(Ctl)));
    AWPM_TRY(ensure(c, c->wpart, sizeof(double) * kWsumBlocks));
    const int32_t rs_tiles = (int32_t)(((int64_t)nnz + kRsTile - 1) / kRsTile);
    int32_t rs_passes = 1;
    while (rs_passes < 4 && ((int64_t)(n - 1) >> (8 * rs_passes)) > 0)
        ++rs_passes;
    if (lookup == AWPM_LOOKUP_HASH) {
        AWPM_TRY(ensure(c, c->htab, sizeof(unsigned long long) * 2 * (size_t)nnz));
    } else if (lookup == AWPM_LOOKUP_ROWMARK) {
        const size_t m = (size_t)kRsBins * (size_t)rs_tiles;
        AWPM_TRY(ensure(c, c->rowsig, sizeof(unsigned long long) * n));
        AWPM_TRY(ensure(c, c->trowptr, sizeof(int32_t) * ((size_t)n + 1)));
        AWPM_TRY(ensure(c, c->rs_k0, sizeof(int32_t) * ((size_t)nnz + 1)));
        AWPM_TRY(ensure(c, c->rs_k1, sizeof(int32_t) * ((size_t)nnz + 1)));
        AWPM_TRY(ensure(c, c->rs_v0, sizeof(int32_t) * ((size_t)nnz + 1)));
        AWPM_TRY(ensure(c, c->rs_v1, sizeof(int32_t) * ((size_t)nnz + 1)));
        AWPM_TRY(ensure(c, c->rs_hist, sizeof(int32_t) * (m + 1)));
        AWPM_TRY(ensure(c, c->rs_sums, sizeof(int32_t) * (m / kScanChunk + 2)));
    } else {
        AWPM_TRY(ensure(c, c->bloom, sizeof(uint32_t) * ((size_t)nnz / 4 + 1)));
    }
    const bool ps = c->opt.select == AWPM_SELECT_GREEDY && !r.search_only;
    if (ps) {
        AWPM_TRY(ensure(c, c->psel, sizeof(Sel) * n));
        AWPM_TRY(ensure(c, c->pslive, sizeof(uint32_t) * ((size_t)n / 32 + 1)));
        AWPM_TRY(ensure(c, c->pstaken, sizeof(uint32_t) * ((size_t)n / 32 + 1)));
        AWPM_TRY(ensure(c, c->psused, sizeof(uint32_t) * ((size_t)n / 32 + 1)));
    }

    // Passes after the first search only what the last flips affect, in single
    // solves (a batched solve's passes walk the running matrices' tiles) of at
    // least kIncTiles tiles: below that a whole search is so short that the
    // incremental form's kernel (its bitmaps, one block per SM) costs more.
    // Whole searches against incremental passes, ms per solve: 27-point stencil
    // 0.87 / 0.95 at 0.5 M entries, 1.43 / 1.27 at 2.1 M, 2.16 / 1.79 at 4.2 M,
    // 14.8 / 6.8 at 23 M; 5-point stencil 0.40 / 0.43 at 2.1 M, 0.66 / 0.65 at
    // 4.2 M; banded 0.66 / 0.73 and 1.02 / 1.03; R-MAT 0.24 / 0.25 and 0.40 /
    // 0.39.  Where the budget or the device has no room for them, every pass
    // searches all.
    Shape sh = shape_of(c, count > 0, lookup, wide, ntiles);
    const IncLayout il(n, ntiles);
    if (count == 0 && !r.search_only && max_passes > 1 && ntiles >= inc_min_tiles() &&
        !c->least_memory) {
        c->spares_used = true;
        const int rc = ensure(c, c->incbuf, il.bytes);
        if (rc == AWPM_ERR_OOM && c->injected)
            return rc;
        sh.inc = rc == AWPM_OK;
        sh.large = sh.inc && il.map_bits > 0;
    }

    // the solve graph of this launch shape, built once (before the timed span)
    cudaGraphExec_t gexec = nullptr;
    if (!r.search_only && !timed) {
        cudaGraphExec_t &g = c->g_exec[count > 0 ? 1 : 0][lookup_slot(lookup)]
                                      [wide ? 1 : 0][sh.search_waves - 1][sh.select]
                                      [sh.large ? 2 : sh.inc ? 1 : 0];
        if (!g)
            AWPM_TRY(build_graph(c, sh, &g));
        gexec = g;
    }
    CUDA_TRY(cudaEventRecord(c->ev_a, c->stream));
    Work &wk = *c->h_work;
    std::memset(&wk, 0, sizeof(Work));
    wk.n = n;
    wk.nnz = nnz;
    wk.ntiles = ntiles;
    wk.max_passes = max_passes;
    wk.lookup = lookup;
    AWPM_TRY(stage_in(c, c->s_colptr, r.colptr, (size_t)n + 1, l_colptr, &wk.colptr));
    AWPM_TRY(stage_in(c, c->s_rowidx, r.rowidx, (size_t)nnz, l_rowidx, &wk.rowidx));
    AWPM_TRY(stage_in(c, c->s_w, r.weight, (size_t)nnz, l_w, &wk.w));
    AWPM_TRY(stage_in(c, c->s_mate, r.mate_in, (size_t)n, l_mate, &wk.mate_in));
    wk.mc = (int32_t *)c->mc.p;
    wk.mr = (int32_t *)c->mr.p;
    wk.wm = (double *)c->wm.p;
    wk.rsig = (unsigned long long *)c->rsig.p;
    wk.rrange = (RowRange *)c->rr.p;
    wk.colsig = (unsigned long long *)c->colsig.p;
    wk.htab = lookup == AWPM_LOOKUP_HASH ? (unsigned long long *)c->htab.p : nullptr;
    wk.bloom = lookup == AWPM_LOOKUP_BSEARCH && bloom_enabled() ? (uint32_t *)c->bloom.p : nullptr;
    wk.bloom_min = wk.bloom ? bloom_min(n, nnz) : kNoBloom;
    if (lookup == AWPM_LOOKUP_ROWMARK) {
        wk.rowsig = (unsigned long long *)c->rowsig.p;
        wk.trowptr = (int32_t *)c->trowptr.p;
        wk.rs_key[0] = (int32_t *)c->rs_k0.p;
        wk.rs_key[1] = (int32_t *)c->rs_k1.p;
        wk.rs_val[0] = (int32_t *)c->rs_v0.p;
        wk.rs_val[1] = (int32_t *)c->rs_v1.p;
        wk.rs_hist = (int32_t *)c->rs_hist.p;
        wk.rs_sums = (int32_t *)c->rs_sums.p;
        wk.rs_tiles = rs_tiles;
        wk.rs_passes = rs_passes;
        wk.tpos = wk.rs_val[(rs_passes - 1) & 1];
    }
    if (ps) {
        wk.psel = (Sel *)c->psel.p;
        wk.pslive = (uint32_t *)c->pslive.p;
        wk.pstaken = (uint32_t *)c->pstaken.p;
        wk.psused = (uint32_t *)c->psused.p;
    }
    wk.best = (Rec *)c->best.p;
    wk.dsel = (Sel *)c->dsel.p;
    {
        // solves with Step D's selection (single or batched) leave the
        // Step-C records empty: every pass's flip clears the records of its
        // winners (incremental passes: the last one, which has none); the
        // Step-D records they leave are of older epochs
        const bool keeps_clean = !r.search_only && !ps;
        wk.rec_clean = keeps_clean && (int64_t)n <= c->rec_clean &&
                               c->sel_epoch + max_passes < 0x7fffffff
                           ? 1
                           : 0;
        pd.rec_clean_after = keeps_clean ? std::max<int64_t>(n, wk.rec_clean ? c->rec_clean : 0) : 0;
        pd.rec_clean_capped = sh.inc ? 0 : pd.rec_clean_after;
        pd.epoch0 = wk.rec_clean ? c->sel_epoch : 0;
        wk.epoch0 = (int32_t)pd.epoch0;
        c->rec_clean = 0;
    }
    wk.winbits = (uint32_t *)c->winbits.p;
    wk.wkey = (int32_t *)c->wkey.p;
    wk.tile_col = (int32_t *)c->tile_col.p;
    wk.starts = (uint32_t *)c->starts.p;
    wk.ctl = (Ctl *)c->ctl.p;
    wk.wpart = (double *)c->wpart.p;
    if (sh.inc) {
        unsigned char *p = (unsigned char *)c->incbuf.p;
        wk.inc = 1;
        wk.map_bits = il.map_bits;
        wk.foundbits = (uint32_t *)(p + il.found);
        wk.posbits = (uint32_t *)(p + il.pos);
        wk.mc_old = (int32_t *)(p + il.mc_old);
        for (int x = 0; x < 2; ++x) {
            wk.map_small[x] = (uint32_t *)(p + il.small[x]);
            wk.map_large[x] = (uint32_t *)(p + il.large[x]);
            wk.colfull[x] = (uint32_t *)(p + il.full[x]);
            wk.colpos[x] = (uint32_t *)(p + il.posi[x]);
            wk.tilemark[x] = (uint32_t *)(p + il.mark[x]);
        }
    }
    if (count > 0) {
        BatchWork &bw = wk.bw;
        AWPM_TRY(stage_in(c, c->b_noff, r.n_off, (size_t)count + 1, l_off, &bw.n_off));
        AWPM_TRY(ensure(c, c->b_colmat, sizeof(int32_t) * n));
        AWPM_TRY(ensure(c, c->b_tilemat, sizeof(int32_t) * ((size_t)ntiles + 1)));
        AWPM_TRY(batch_arrays(c, bw, count));
        AWPM_TRY(ensure(c, c->b_tlist, sizeof(int32_t) * ((size_t)ntiles + 1)));
        bw.colmat = (int32_t *)c->b_colmat.p;
        bw.tilemat = (int32_t *)c->b_tilemat.p;
        bw.tlist = (int32_t *)c->b_tlist.p;
        pd.n_off.resize((size_t)count + 1);
        if (r.off_host)
            std::memcpy(pd.n_off.data(), r.off_host, sizeof(int32_t) * (count + 1));
        else if (l_off == 1)
            CUDA_TRY(cudaMemcpyAsync(pd.n_off.data(), r.n_off, sizeof(int32_t) * (count + 1),
                                     cudaMemcpyDeviceToHost, c->stream));
        else
            std::memcpy(pd.n_off.data(), r.n_off, sizeof(int32_t) * (count + 1));
    }
    CUDA_TRY(cudaMemcpyAsync(c->d_work.p, c->h_work, sizeof(Work), cudaMemcpyHostToDevice,
                             c->stream));
    const Work *d = (const Work *)c->d_work.p;

    if (r.search_only) {
        Sink k;
        k.stream = c->stream;
        launch_init(d, sh, k);
        launch_search(d, sh, k);
        double *g = r.gain_out;
        int32_t *row = r.row_out;
        if (l_gain != 1) {
            AWPM_TRY(ensure(c, c->s_gain, sizeof(double) * n));
            g = (double *)c->s_gain.p;
        }
        if (l_row != 1) {
            AWPM_TRY(ensure(c, c->s_row, sizeof(int32_t) * n));
            row = (int32_t *)c->s_row.p;
        }
        launch_export_stepc(d, sh, g, row, k);
        AWPM_TRY(check_sink(k));
        if (l_gain != 1)
            CUDA_TRY(cudaMemcpyAsync(r.gain_out, g, sizeof(double) * n, cudaMemcpyDeviceToHost,
                                     c->stream));
        if (l_row != 1)
            CUDA_TRY(cudaMemcpyAsync(r.row_out, row, sizeof(int32_t) * n, cudaMemcpyDeviceToHost,
                                     c->stream));
    } else if (timed) {
        AWPM_TRY(run_timed(c, sh, max_passes, &pd.passes_enqueued));
    } else {
        CUDA_TRY(cudaGraphLaunch(gexec, c->stream));
    }
    if (!r.search_only)
        CUDA_TRY(cudaMemcpyAsync(r.mate_out, wk.mc, sizeof(int32_t) * n,
                                 l_out == 1 ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                                 c->stream));
    CUDA_TRY(cudaMemcpyAsync(c->h_ctl, wk.ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, c->stream));
    if (count > 0)
        AWPM_TRY(copy_batch_results(c, wk.bw));
    CUDA_TRY(cudaEventRecord(c->ev_b, c->stream));
    pd.active = true;
    pd.timed = timed && !r.search_only;
    pd.n = n;
    pd.nnz = nnz;
    pd.count = count;
    return AWPM_OK;
}

// Enqueue a batch of small matrices (nnz known, per_class given, pd.order
// filled), or a single one (nnz -1: the kernel reads it).
int ctx_enqueue_small(awpm_ctx *c, const Request &r, int32_t nnz, const int32_t *per_class,
                      int l_colptr, int l_rowidx, int l_w, int l_mate, int l_out)
{
    Pending &pd = c->pend;
    const int32_t n = r.n, count = r.count > 0 ? r.count : 1;
    const int32_t cap = nnz >= 0 ? nnz : kSmallOneNnz;
    const int32_t max_passes = c->opt.max_iters > 0 ? c->opt.max_iters : AWPM_PASS_CAP;
    const size_t words = (size_t)cap / 32 + (size_t)count + 1;
    c->spares_used = true;
    AWPM_TRY(ensure(c, c->wm, sizeof(double) * n));
    const void *best_was = c->best.p, *dsel_was = c->dsel.p;
    AWPM_TRY(ensure(c, c->best, sizeof(Rec) * n));
    AWPM_TRY(ensure(c, c->dsel, sizeof(Sel) * n));
    if (c->best.p != best_was || c->dsel.p != dsel_was)
        c->rec_clean = 0;
    AWPM_TRY(ensure(c, c->wkey, sizeof(int32_t) * n));
    AWPM_TRY(ensure(c, c->ctl, sizeof(Ctl)));
    AWPM_TRY(ensure(c, c->smallbuf, 3 * sizeof(uint32_t) * words));
    if (l_out != 1)
        AWPM_TRY(ensure(c, c->mc, sizeof(int32_t) * n));
    CUDA_TRY(cudaEventRecord(c->ev_a, c->stream));
    Work &wk = *c->h_work;
    std::memset(&wk, 0, sizeof(Work));
    wk.n = n;
    wk.nnz = nnz;
    wk.max_passes = max_passes;
    wk.lookup = AWPM_LOOKUP_BSEARCH;
    AWPM_TRY(stage_in(c, c->s_colptr, r.colptr, (size_t)n + 1, l_colptr, &wk.colptr));
    AWPM_TRY(stage_in(c, c->s_rowidx, r.rowidx, (size_t)(nnz > 0 ? nnz : 0), l_rowidx, &wk.rowidx));
    AWPM_TRY(stage_in(c, c->s_w, r.weight, (size_t)(nnz > 0 ? nnz : 0), l_w, &wk.w));
    AWPM_TRY(stage_in(c, c->s_mate, r.mate_in, (size_t)n, l_mate, &wk.mate_in));
    wk.wm = (double *)c->wm.p;
    wk.best = (Rec *)c->best.p;
    wk.dsel = (Sel *)c->dsel.p;
    wk.wkey = (int32_t *)c->wkey.p;
    wk.ctl = (Ctl *)c->ctl.p;
    wk.rec_clean =
        (int64_t)n <= c->rec_clean && c->sel_epoch + max_passes < 0x7fffffff ? 1 : 0;
    pd.rec_clean_after = std::max<int64_t>(n, wk.rec_clean ? c->rec_clean : 0);
    pd.rec_clean_capped = 0;
    pd.epoch0 = wk.rec_clean ? c->sel_epoch : 0;
    wk.epoch0 = (int32_t)pd.epoch0;
    c->rec_clean = 0;
    wk.small_cap = cap;
    wk.small_fb = (uint32_t *)c->smallbuf.p;
    wk.small_pb = wk.small_fb + words;
    wk.small_c0 = (int32_t *)(wk.small_pb + words);
    wk.small_out = l_out == 1 ? r.mate_out : (int32_t *)c->mc.p;
    for (int x = 0; x <= kSmallClasses; ++x)
        wk.small_smem[x] = (int32_t)small_class_smem(x);
    AWPM_TRY(batch_arrays(c, wk.bw, count));
    wk.small_next = (int32_t *)c->b_i32.p + 5 * (size_t)count + 2;
    const Work *d = (const Work *)c->d_work.p;
    Sink k;
    k.stream = c->stream;
    if (r.count > 0) {
        pd.n_off.assign(r.off_host, r.off_host + count + 1);
        AWPM_TRY(ensure(c, c->b_order, sizeof(int32_t) * (2 * (size_t)count + 1)));
        int32_t *dord = (int32_t *)c->b_order.p;
        // the offsets and the order in one copy
        pd.order.insert(pd.order.end(), pd.n_off.begin(), pd.n_off.end());
        CUDA_TRY(cudaMemcpyAsync(dord, pd.order.data(), sizeof(int32_t) * pd.order.size(),
                                 cudaMemcpyHostToDevice, c->stream));
        wk.small_order = dord;
        wk.bw.n_off = dord + count;
        for (int x = 0, at = 0; x < kSmallClasses; at += per_class[x++]) {
            wk.small_first[x] = at;
            wk.small_count[x] = per_class[x];
        }
        CUDA_TRY(cudaMemcpyAsync(c->d_work.p, &wk, sizeof(Work), cudaMemcpyHostToDevice,
                                 c->stream));
        Shape sh;
        sh.num_sms = c->num_sms;
        if (!c->small_streams.fork) {
            SmallStreams ss;
            for (cudaStream_t &s : ss.side)
                CUDA_TRY(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
            for (cudaEvent_t &e : ss.join)
                CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
            CUDA_TRY(cudaEventCreateWithFlags(&ss.fork, cudaEventDisableTiming));
            c->small_streams = ss;
        }
        launch_small_batch(d, sh, per_class, c->small_streams, k);
    } else {
        AWPM_TRY(ensure(c, c->winbits, sizeof(uint32_t) * ((size_t)n / 32 + 1)));
        AWPM_TRY(ensure(c, c->colsig, sizeof(unsigned long long) * n));
        wk.winbits = (uint32_t *)c->winbits.p;
        wk.small_sig = (uint32_t *)c->colsig.p;
        wk.small_off[1] = n;
        wk.bw.n_off = (const int32_t *)((const char *)d + offsetof(Work, small_off));
        if (nnz < 0)
            wk.small_nnz = wk.colptr + n;
        const size_t need = small_smem(n, kSmallWarps[kSmallOne], true) + 1024;
        if (need < small_class_smem(kSmallOne))
            wk.small_smem[kSmallOne] = (int32_t)need;
        CUDA_TRY(cudaMemcpyAsync(c->d_work.p, &wk, sizeof(Work), cudaMemcpyHostToDevice,
                                 c->stream));
        launch_small_one(d, wk.small_smem[kSmallOne], k);
    }
    AWPM_TRY(check_sink(k));
    if (l_out != 1)
        CUDA_TRY(cudaMemcpyAsync(r.mate_out, wk.small_out, sizeof(int32_t) * n,
                                 cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(cudaMemcpyAsync(c->h_ctl, wk.ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, c->stream));
    if (r.count > 0)
        AWPM_TRY(copy_batch_results(c, wk.bw));
    CUDA_TRY(cudaEventRecord(c->ev_b, c->stream));
    pd.active = true;
    pd.small = true;
    pd.req = r;
    pd.lookup = AWPM_LOOKUP_BSEARCH;
    pd.n = n;
    pd.nnz = nnz;
    pd.count = r.count;
    return AWPM_OK;
}

int ctx_finish(awpm_ctx *c, awpm_stats *st, awpm_stats *per_matrix)
{
    NvtxRange nvtx_range("finish");
    Pending &pd = c->pend;
    if (!pd.active)
        return AWPM_ERR_INVALID_ARG;
    pd.active = false;
    awpm_stats S;
    std::memset(&S, 0, sizeof(S));
    S.lookup_used = pd.lookup;
    if (pd.trivial) {
        S.iterations = pd.search_only ? 0 : 1;
        S.converged = 1;
        if (st)
            *st = S;
        return AWPM_OK;
    }
    CUDA_TRY(cudaEventSynchronize(c->ev_b));
    c->spares_used = false;
    const Ctl &h = *c->h_ctl;
    if (pd.small && h.err) {
        // the general path names the error (or solves what was not for the
        // small-matrix kernel)
        Request again = pd.req;
        if (again.count == 0 && pd.nnz < 0 && small_too_many(h.small_nnz))
            c->small_dense |= 1u << ilog2(pd.n);
        const std::vector<int32_t> off = pd.n_off;
        if (again.off_host)
            again.off_host = off.data();
        c->general_only = true;
        int rc = ctx_enqueue(c, again);
        c->general_only = false;
        if (rc != AWPM_OK) {
            cudaStreamSynchronize(c->stream);
            cudaGetLastError();
            c->pend.active = false;
            return rc;
        }
        return ctx_finish(c, st, per_matrix);
    }
    if (pd.small && pd.count == 0)
        pd.nnz = h.small_nnz;
    const int rc = code_of(h.err);
    if (rc != AWPM_OK)
        return rc;
    c->rec_clean = h.converged ? pd.rec_clean_after : pd.rec_clean_capped;
    c->sel_epoch = pd.epoch0 + h.iterations;
    double ms_search = 0.0;
    if (pd.timed) {
        for (int t = 0; t < h.iterations && t < pd.passes_enqueued; ++t) {
            float ms = 0.f;
            CUDA_TRY(cudaEventElapsedTime(&ms, c->tev[2 * t], c->tev[2 * t + 1]));
            ms_search += ms;
        }
    }
    float ms_total = 0.f;
    CUDA_TRY(cudaEventElapsedTime(&ms_total, c->ev_a, c->ev_b));
    if (pd.tune_cfg >= 0) {
        TuneEntry &te = c->tune[pd.tune_key];
        if (te.chosen < 0 && pd.tune_cfg == te.trials) {
            te.ms[te.trials++] = ms_total;
            if (te.trials == kTuneConfigs) {
                int best = 0;
                for (int k = 1; k < kTuneConfigs; ++k)
                    if (te.ms[k] < te.ms[best])
                        best = k;
                te.chosen = best;
            }
        }
        pd.tune_cfg = -1;
    }
    S.iterations = h.iterations;
    S.converged = h.converged;
    S.cycles_applied = (int64_t)h.cycles;
    S.edge_checks = (int64_t)(pd.nnz - pd.n) * (int64_t)(pd.search_only ? 1 : h.iterations);
    S.candidates = (int64_t)h.candidates;
    S.closing_found = (int64_t)h.found;
    S.positive = (int64_t)h.positive;
    S.weight_in = h.weight_in;
    S.weight_out = pd.search_only ? h.weight_in : h.weight_out;
    S.ms_total = ms_total;
    S.ms_search = ms_search;
    if (pd.count > 0) {
        const int32_t count = pd.count;
        const char *hb = (const char *)c->h_batch;
        const int32_t *miter = (const int32_t *)hb;
        const int32_t *mconv = miter + count;
        const int32_t *mnnz = miter + 2 * (size_t)count;
        const unsigned long long *mcyc = (const unsigned long long *)(hb + 12 * (size_t)count);
        const double *mwi = (const double *)(hb + 20 * (size_t)count);
        const double *mwo = mwi + count;
        int all_conv = 1;
        S.edge_checks = 0;
        for (int32_t b = 0; b < count; ++b) {
            const int64_t ec = (int64_t)(mnnz[b] - (pd.n_off[b + 1] - pd.n_off[b])) * miter[b];
            S.edge_checks += ec;
            all_conv &= mconv[b];
            if (!per_matrix)
                continue;
            awpm_stats &m = per_matrix[b];
            std::memset(&m, 0, sizeof(m));
            m.iterations = miter[b];
            m.converged = mconv[b];
            m.cycles_applied = (int64_t)mcyc[b];
            m.edge_checks = ec;
            m.weight_in = mwi[b];
            m.weight_out = mwo[b];
            m.ms_total = ms_total;
            m.lookup_used = pd.lookup;
        }
        S.converged = all_conv;
    }
    if (st)
        *st = S;
    return AWPM_OK;
}

}  // namespace awpm

extern "C" {

const char *awpm_strerror(int code)
{
    switch (code) {
    case AWPM_OK: return "ok";
    case AWPM_ERR_INVALID_ARG: return "invalid argument";
    case AWPM_ERR_NOT_PERFECT: return "mate_in is not a perfect matching of stored entries";
    case AWPM_ERR_UNSORTED_OR_DUP: return "rows not strictly increasing within a column";
    case AWPM_ERR_NONFINITE: return "non-finite weight";
    case AWPM_ERR_OOM: return "out of memory";
    case AWPM_ERR_BUDGET: return "device memory budget exceeded";
    case AWPM_ERR_CUDA: return "CUDA error";
    case AWPM_ERR_TIMEOUT: return "a bounded device-side retry or loop gave up";
    case AWPM_ERR_NOT_FOUND: return "unknown ticket";
    case AWPM_ERR_TOO_LARGE: return "problem exceeds the fixed scratch of awpm_search_noalloc";
    case AWPM_ERR_INTERNAL: return "internal consistency check failed (library bug)";
    case AWPM_ERR_CANCELLED: return "request cancelled before it started";
    default: return "unknown error";
    }
}

const char *awpm_last_error(void)
{
    return g_last_error;
}

void awpm_default_options(awpm_options *opt)
{
    if (!opt)
        return;
    std::memset(opt, 0, sizeof(*opt));
    opt->device = -1;
    opt->max_iters = 0;
    opt->lookup = AWPM_LOOKUP_AUTO;
    opt->flags = 0;
    opt->stream = nullptr;
    opt->mem_budget_bytes = 0;
    opt->slots = 0;
    opt->select = AWPM_SELECT_STEP_D;
}

int awpm_create(awpm_ctx **out, const awpm_options *opt)
{
    if (!out)
        return AWPM_ERR_INVALID_ARG;
    *out = nullptr;
    awpm_ctx *c = new (std::nothrow) awpm_ctx();
    if (!c)
        return AWPM_ERR_OOM;
    int rc = setup_ctx(c, opt);
    if (rc != AWPM_OK) {
        teardown_ctx(c);
        delete c;
        return rc;
    }
    *out = c;
    return AWPM_OK;
}

void awpm_server_shutdown(awpm_ctx *ctx);

int awpm_destroy(awpm_ctx *ctx)
{
    if (!ctx)
        return AWPM_OK;
    awpm_server_shutdown(ctx);
    {
        std::lock_guard<std::mutex> lk(ctx->mu);
        cudaSetDevice(ctx->device);
        teardown_ctx(ctx);
    }
    delete ctx;
    return AWPM_OK;
}

int awpm_inject_alloc_failure(awpm_ctx *ctx, int32_t after)
{
    if (!ctx || after < -1)
        return AWPM_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(ctx->mu);
    ctx->fail_after = after;
    return AWPM_OK;
}

void awpm_server_memory(awpm_ctx *ctx, size_t *held, size_t *peak);

int awpm_bytes_needed(awpm_ctx *ctx, int32_t n, int32_t nnz, int32_t host_inputs, size_t *bytes)
{
    if (!ctx || !bytes || n < 0 || nnz < 0)
        return AWPM_ERR_INVALID_ARG;
    *bytes = ctx_bytes_needed(n, nnz, host_inputs != 0, ctx->opt.lookup, ctx->opt.select,
                              false);
    return AWPM_OK;
}

int awpm_memory_held(awpm_ctx *ctx, size_t *held, size_t *peak)
{
    if (!ctx || !held || !peak)
        return AWPM_ERR_INVALID_ARG;
    size_t h, p;
    {
        std::lock_guard<std::mutex> lk(ctx->mu);
        h = ctx->held;
        p = ctx->peak;
    }
    size_t sh = 0, sp = 0;
    awpm_server_memory(ctx, &sh, &sp);
    *held = h + sh;
    *peak = p > sp ? p : sp;
    return AWPM_OK;
}

static int solve_sync(awpm_ctx *c, const Request &r, awpm_stats *st, awpm_stats *per_matrix)
{
    std::lock_guard<std::mutex> lk(c->mu);
    int rc;
    try {
        rc = ctx_enqueue(c, r);
        if (rc == AWPM_OK)
            return ctx_finish(c, st, per_matrix);
    } catch (const std::bad_alloc &) {  // (host memory: offsets and order of a batch)
        c->general_only = c->force_blocks = c->least_memory = false;
        rc = AWPM_ERR_OOM;
    }
    if (c->stream)
        cudaStreamSynchronize(c->stream);
    cudaGetLastError();
    c->pend.active = false;
    c->spares_used = false;
    return rc;
}

int awpm_improve_ctx(awpm_ctx *ctx, int32_t n, const int32_t *colptr, const int32_t *rowidx,
                     const double *weight, const int32_t *mate_in, int32_t *mate_out,
                     awpm_stats *stats)
{
    NvtxRange nvtx_range("awpm_improve");
    if (!ctx)
        return AWPM_ERR_INVALID_ARG;
    Request r;
    r.n = n;
    r.colptr = colptr;
    r.rowidx = rowidx;
    r.weight = weight;
    r.mate_in = mate_in;
    r.mate_out = mate_out;
    if (!mate_in && n > 0) {
        // no matching given: start from the greedy maximal matching
        if (!mate_out)
            return AWPM_ERR_INVALID_ARG;
        int32_t *gm = nullptr;
        {
            std::lock_guard<std::mutex> lk(ctx->mu);
            CUDA_TRY(cudaSetDevice(ctx->device));
            AWPM_TRY(ensure(ctx, ctx->gmate, sizeof(int32_t) * (size_t)n));
            gm = (int32_t *)ctx->gmate.p;
        }
        awpm_greedy_stats gs;
        AWPM_TRY(awpm_greedy(ctx, n, colptr, rowidx, weight, gm, &gs));
        int32_t card = gs.cardinality;
        if (card != n) {
            // greedy is not perfect: complete it with augmenting paths
            awpm_mcm_stats ms;
            AWPM_TRY(awpm_mcm(ctx, n, colptr, rowidx, weight, gm, &ms));
            card = ms.cardinality;
        }
        if (card != n) {
            std::lock_guard<std::mutex> lk(ctx->mu);
            const int l_out = where(ctx, mate_out);
            if (l_out < 0)
                return AWPM_ERR_INVALID_ARG;
            CUDA_TRY(cudaMemcpyAsync(mate_out, gm, sizeof(int32_t) * (size_t)n,
                                     l_out == 1 ? cudaMemcpyDeviceToDevice
                                                : cudaMemcpyDeviceToHost,
                                     ctx->stream));
            CUDA_TRY(cudaStreamSynchronize(ctx->stream));
            return AWPM_ERR_NOT_PERFECT;
        }
        r.mate_in = gm;
    }
    return solve_sync(ctx, r, stats, nullptr);
}

int awpm_improve(int32_t n, const int32_t *colptr, const int32_t *rowidx, const double *weight,
                 const int32_t *mate_in, int32_t *mate_out, awpm_stats *stats)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) {
        note_cuda_error(e, "cudaGetDevice", __LINE__);
        return AWPM_ERR_CUDA;
    }
    awpm_ctx *c = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_default_mu);
        auto it = g_default.find(dev);
        if (it == g_default.end()) {
            awpm_options o;
            awpm_default_options(&o);
            o.device = dev;
            int rc = awpm_create(&c, &o);
            if (rc != AWPM_OK)
                return rc;
            g_default[dev] = c;
        } else {
            c = it->second;
        }
    }
    return awpm_improve_ctx(c, n, colptr, rowidx, weight, mate_in, mate_out, stats);
}

int awpm_improve_batch(awpm_ctx *ctx, int32_t count, const int32_t *n_off, const int32_t *colptr,
                       const int32_t *rowidx, const double *weight, const int32_t *mate_in,
                       int32_t *mate_out, awpm_stats *per_matrix, awpm_stats *total)
{
    NvtxRange nvtx_range("awpm_improve_batch");
    if (!ctx || count < 0 || (count > 0 && !n_off))
        return AWPM_ERR_INVALID_ARG;
    if (count == 0) {
        if (total) {
            std::memset(total, 0, sizeof(*total));
            total->converged = 1;
        }
        return AWPM_OK;
    }
    std::vector<int32_t> off;
    try {
        off.resize((size_t)count + 1);
    } catch (const std::bad_alloc &) {
        return AWPM_ERR_OOM;
    }
    {
        std::lock_guard<std::mutex> lk(ctx->mu);
        cudaError_t e = cudaSetDevice(ctx->device);
        if (e == cudaSuccess && where(ctx, n_off) == 1)
            e = cudaMemcpy(off.data(), n_off, sizeof(int32_t) * off.size(),
                           cudaMemcpyDeviceToHost);
        else if (e == cudaSuccess)
            std::memcpy(off.data(), n_off, sizeof(int32_t) * off.size());
        if (e != cudaSuccess) {
            note_cuda_error(e, "reading the batch offsets", __LINE__);
            return AWPM_ERR_CUDA;
        }
    }
    const int32_t n = off[(size_t)count];
    if (n <= 0)
        return AWPM_ERR_INVALID_ARG;
    Request r;
    r.n = n;
    r.off_host = off.data();
    r.colptr = colptr;
    r.rowidx = rowidx;
    r.weight = weight;
    r.mate_in = mate_in;
    r.mate_out = mate_out;
    r.count = count;
    r.n_off = n_off;
    return solve_sync(ctx, r, total, per_matrix);
}

int awpm_greedy(awpm_ctx *ctx, int32_t n, const int32_t *colptr, const int32_t *rowidx,
                const double *weight, int32_t *mate_out, awpm_greedy_stats *stats)
{
    NvtxRange nvtx_range("awpm_greedy");
    if (!ctx || n < 0 || (n > 0 && (!colptr || !mate_out)))
        return AWPM_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(ctx->mu);
    awpm_ctx *c = ctx;
    awpm_greedy_stats S;
    std::memset(&S, 0, sizeof(S));
    if (n == 0) {
        S.rounds = 1;  // one round, which matches nothing
        if (stats)
            *stats = S;
        return AWPM_OK;
    }
    CUDA_TRY(cudaSetDevice(c->device));
    const int l_colptr = where(c, colptr), l_rowidx = where(c, rowidx), l_w = where(c, weight),
              l_out = where(c, mate_out);
    if (l_colptr < 0 || l_rowidx < 0 || l_w < 0 || l_out < 0)
        return AWPM_ERR_INVALID_ARG;
    int32_t nnz = 0;
    if (l_colptr == 1) {
        CUDA_TRY(cudaMemcpyAsync(c->h_ctl, colptr + n, sizeof(int32_t), cudaMemcpyDeviceToHost,
                                 c->stream));
        CUDA_TRY(cudaStreamSynchronize(c->stream));
        std::memcpy(&nnz, c->h_ctl, sizeof(int32_t));
    } else {
        nnz = colptr[n];
    }
    if (nnz < 0 || nnz > kMaxEntries || (nnz > 0 && (!rowidx || !weight)))
        return AWPM_ERR_INVALID_ARG;
    const int32_t ntiles = (int32_t)(((int64_t)nnz + kTile - 1) / kTile);
    AWPM_TRY(ensure(c, c->mc, sizeof(int32_t) * n));
    // (the records share the maximum matching's buffers: the two run one after
    // the other)
    AWPM_TRY(ensure(c, c->mroff, sizeof(Off) * n));
    AWPM_TRY(ensure(c, c->mtend, sizeof(Off) * n));
    AWPM_TRY(ensure(c, c->gdead, (size_t)ntiles / 8 + 1));
    AWPM_TRY(ensure(c, c->tile_col, sizeof(int32_t) * ((size_t)ntiles + 1)));
    AWPM_TRY(ensure(c, c->starts, sizeof(uint32_t) * (((size_t)nnz + 31) / 32 + 1)));
    AWPM_TRY(ensure(c, c->ctl, sizeof(Ctl)));
    AWPM_TRY(ensure(c, c->wpart, sizeof(double) * kWsumBlocks));
    Shape sh = shape_of(c, false, AWPM_LOOKUP_BSEARCH, true, ntiles);
    sh.cluster = c->clusters && ntiles <= kGmClusterTiles;
    sh.greedy = true;
    // AWPM_FLAG_TIME_SEARCH: a host loop over the rounds (every kernel a
    // separate stream launch, visible to profilers) instead of the graph
    const bool host_loop = (c->opt.flags & AWPM_FLAG_TIME_SEARCH) != 0;
    cudaGraphExec_t g = nullptr;
    if (!host_loop) {
        cudaGraphExec_t &gg = c->g_greedy[sh.cluster ? 2 : sh.search_waves - 1];
        if (!gg)
            AWPM_TRY(build_greedy_graph(c, sh, &gg));
        g = gg;
    }
    CUDA_TRY(cudaEventRecord(c->ev_a, c->stream));
    Work &wk = *c->h_work;
    std::memset(&wk, 0, sizeof(Work));
    wk.n = n;
    wk.nnz = nnz;
    wk.ntiles = ntiles;
    // at most n rounds match something, then one matches nothing
    wk.max_passes = n < 0x7fffffff ? n + 1 : n;
    wk.lookup = AWPM_LOOKUP_BSEARCH;
    AWPM_TRY(stage_in(c, c->s_colptr, colptr, (size_t)n + 1, l_colptr, &wk.colptr));
    AWPM_TRY(stage_in(c, c->s_rowidx, rowidx, (size_t)nnz, l_rowidx, &wk.rowidx));
    AWPM_TRY(stage_in(c, c->s_w, weight, (size_t)nnz, l_w, &wk.w));
    wk.mc = (int32_t *)c->mc.p;
    wk.tile_col = (int32_t *)c->tile_col.p;
    wk.starts = (uint32_t *)c->starts.p;
    wk.ctl = (Ctl *)c->ctl.p;
    wk.wpart = (double *)c->wpart.p;
    wk.grow = (Off *)c->mroff.p;
    wk.gcol = (Off *)c->mtend.p;
    wk.gdead = (uint8_t *)c->gdead.p;
    CUDA_TRY(cudaMemcpyAsync(c->d_work.p, c->h_work, sizeof(Work), cudaMemcpyHostToDevice,
                             c->stream));
    if (host_loop) {
        const Work *d = (const Work *)c->d_work.p;
        Sink k;
        k.stream = c->stream;
        launch_greedy_init(d, sh, k);
        for (int32_t round = 0; round < wk.max_passes; ++round) {
            launch_greedy_round(d, sh, false, cudaGraphConditionalHandle(), k);
            AWPM_TRY(check_sink(k));
            CUDA_TRY(cudaMemcpyAsync(c->h_ctl, wk.ctl, sizeof(Ctl), cudaMemcpyDeviceToHost,
                                     c->stream));
            CUDA_TRY(cudaStreamSynchronize(c->stream));
            if (!c->h_ctl->active)
                break;
        }
        launch_weight_sum(d, sh, true, k);
        AWPM_TRY(check_sink(k));
    } else {
        CUDA_TRY(cudaGraphLaunch(g, c->stream));
    }
    CUDA_TRY(cudaMemcpyAsync(mate_out, wk.mc, sizeof(int32_t) * n,
                             l_out == 1 ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                             c->stream));
    CUDA_TRY(cudaMemcpyAsync(c->h_ctl, wk.ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(cudaEventRecord(c->ev_b, c->stream));
    CUDA_TRY(cudaEventSynchronize(c->ev_b));
    const Ctl &h = *c->h_ctl;
    const int rc = code_of(h.err);
    if (rc != AWPM_OK)
        return rc;
    float ms = 0.f;
    CUDA_TRY(cudaEventElapsedTime(&ms, c->ev_a, c->ev_b));
    S.rounds = h.iterations;
    S.cardinality = (int32_t)h.cycles;
    S.weight = h.weight_out;
    S.ms_total = ms;
    if (stats)
        *stats = S;
    return AWPM_OK;
}

int awpm_mcm(awpm_ctx *ctx, int32_t n, const int32_t *colptr, const int32_t *rowidx,
             const double *weight, int32_t *mate, awpm_mcm_stats *stats)
{
    NvtxRange nvtx_range("awpm_mcm");
    if (!ctx || n < 0 || (n > 0 && (!colptr || !mate)))
        return AWPM_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(ctx->mu);
    awpm_ctx *c = ctx;
    awpm_mcm_stats S;
    std::memset(&S, 0, sizeof(S));
    if (n == 0) {
        S.phases = 1;
        if (stats)
            *stats = S;
        return AWPM_OK;
    }
    CUDA_TRY(cudaSetDevice(c->device));
    const int l_colptr = where(c, colptr), l_rowidx = where(c, rowidx), l_w = where(c, weight),
              l_m = where(c, mate);
    if (l_colptr < 0 || l_rowidx < 0 || l_w < 0 || l_m < 0)
        return AWPM_ERR_INVALID_ARG;
    int32_t nnz = 0;
    if (l_colptr == 1) {
        CUDA_TRY(cudaMemcpyAsync(c->h_ctl, colptr + n, sizeof(int32_t), cudaMemcpyDeviceToHost,
                                 c->stream));
        CUDA_TRY(cudaStreamSynchronize(c->stream));
        std::memcpy(&nnz, c->h_ctl, sizeof(int32_t));
    } else {
        nnz = colptr[n];
    }
    if (nnz < 0 || nnz > kMaxEntries || (nnz > 0 && (!rowidx || !weight)))
        return AWPM_ERR_INVALID_ARG;
    const int32_t ntiles = (int32_t)(((int64_t)nnz + kTile - 1) / kTile);
    const size_t words = (size_t)n / 32 + 1;
    AWPM_TRY(ensure(c, c->mc, sizeof(int32_t) * n));
    AWPM_TRY(ensure(c, c->mr, sizeof(int32_t) * n));
    AWPM_TRY(ensure(c, c->mroot, sizeof(int32_t) * n));
    AWPM_TRY(ensure(c, c->mrpar, sizeof(int32_t) * n));
    AWPM_TRY(ensure(c, c->mroff, sizeof(Off) * n));
    AWPM_TRY(ensure(c, c->mtend, sizeof(Off) * n));
    AWPM_TRY(ensure(c, c->mtouch, sizeof(int32_t) * n));
    AWPM_TRY(ensure(c, c->mfront, sizeof(uint32_t) * (words + 1)));
    AWPM_TRY(ensure(c, c->mreach, sizeof(uint32_t) * (words + 1)));
    AWPM_TRY(ensure(c, c->mtmark, sizeof(uint32_t) * ((size_t)ntiles / 32 + 1)));
    AWPM_TRY(ensure(c, c->mfl, sizeof(int32_t) * n));
    AWPM_TRY(ensure(c, c->mcolof, sizeof(int32_t) * ((size_t)nnz + 1)));
    // the level's tile list: every tile at most once
    AWPM_TRY(ensure(c, c->mtiles, sizeof(int32_t) * ((size_t)ntiles + 1)));
    AWPM_TRY(ensure(c, c->tile_col, sizeof(int32_t) * ((size_t)ntiles + 1)));
    AWPM_TRY(ensure(c, c->starts, sizeof(uint32_t) * (((size_t)nnz + 31) / 32 + 1)));
    AWPM_TRY(ensure(c, c->ctl, sizeof(Ctl)));
    int32_t *dmate = mate;
    if (l_m != 1) {
        AWPM_TRY(ensure(c, c->mstage, sizeof(int32_t) * n));
        dmate = (int32_t *)c->mstage.p;
        CUDA_TRY(cudaMemcpyAsync(dmate, mate, sizeof(int32_t) * n, cudaMemcpyHostToDevice,
                                 c->stream));
    }
    Shape sh = shape_of(c, false, AWPM_LOOKUP_BSEARCH, true, ntiles);
    sh.cluster = c->clusters && mcm_cluster(ntiles, n);
    CUDA_TRY(cudaEventRecord(c->ev_a, c->stream));
    Work &wk = *c->h_work;
    std::memset(&wk, 0, sizeof(Work));
    wk.n = n;
    wk.nnz = nnz;
    wk.ntiles = ntiles;
    AWPM_TRY(stage_in(c, c->s_colptr, colptr, (size_t)n + 1, l_colptr, &wk.colptr));
    AWPM_TRY(stage_in(c, c->s_rowidx, rowidx, (size_t)nnz, l_rowidx, &wk.rowidx));
    AWPM_TRY(stage_in(c, c->s_w, weight, (size_t)nnz, l_w, &wk.w));
    wk.mc = (int32_t *)c->mc.p;
    wk.mr = (int32_t *)c->mr.p;
    wk.tile_col = (int32_t *)c->tile_col.p;
    wk.starts = (uint32_t *)c->starts.p;
    wk.ctl = (Ctl *)c->ctl.p;
    wk.mroot = (int32_t *)c->mroot.p;
    wk.mrpar = (int32_t *)c->mrpar.p;
    wk.mfront = (uint32_t *)c->mfront.p;
    wk.mreach = (uint32_t *)c->mreach.p;
    wk.mtmark = (uint32_t *)c->mtmark.p;
    wk.mfl = (int32_t *)c->mfl.p;
    wk.mroff = (Off *)c->mroff.p;
    wk.mtend = (Off *)c->mtend.p;
    wk.mtouch = (int32_t *)c->mtouch.p;
    wk.mmate = dmate;
    wk.mcolof = (int32_t *)c->mcolof.p;
    wk.mtiles = (int32_t *)c->mtiles.p;
    wk.mtiles_cap = ntiles;
    CUDA_TRY(cudaMemcpyAsync(c->d_work.p, c->h_work, sizeof(Work), cudaMemcpyHostToDevice,
                             c->stream));
    const Work *d = (const Work *)c->d_work.p;
    Ctl *dctl = (Ctl *)c->ctl.p;
    if (!(c->opt.flags & AWPM_FLAG_TIME_SEARCH)) {
        // the whole search in one graph launch (loops on the device)
        cudaGraphExec_t &g = c->g_mcm[sh.cluster ? 2 : sh.search_waves - 1];
        if (!g)
            AWPM_TRY(build_mcm_graph(c, sh, &g));
        CUDA_TRY(cudaGraphLaunch(g, c->stream));
        if (l_m != 1)
            CUDA_TRY(cudaMemcpyAsync(mate, dmate, sizeof(int32_t) * n, cudaMemcpyDeviceToHost,
                                     c->stream));
        CUDA_TRY(cudaMemcpyAsync(c->h_ctl, dctl, sizeof(Ctl), cudaMemcpyDeviceToHost,
                                 c->stream));
        CUDA_TRY(cudaEventRecord(c->ev_b, c->stream));
        CUDA_TRY(cudaEventSynchronize(c->ev_b));
        const int rc = code_of(c->h_ctl->err);
        if (rc != AWPM_OK)
            return rc;
        float gms = 0.f;
        CUDA_TRY(cudaEventElapsedTime(&gms, c->ev_a, c->ev_b));
        S.phases = c->h_ctl->iterations;
        S.cardinality = (int32_t)c->h_ctl->cycles;
        S.levels = (int64_t)c->h_ctl->levels;
        S.ms_total = gms;
        if (stats)
            *stats = S;
        return AWPM_OK;
    }
    // AWPM_FLAG_TIME_SEARCH: levels and phases driven from the host
    Sink k;
    k.stream = c->stream;
    launch_mcm_load(d, sh, k);
    AWPM_TRY(check_sink(k));
    // read one counter of the control block, then zero it on the device
    auto take = [&](void *field, size_t bytes, void *host) -> int {
        CUDA_TRY(cudaMemcpyAsync(host, field, bytes, cudaMemcpyDeviceToHost, c->stream));
        CUDA_TRY(cudaMemcpyAsync(&c->h_ctl->err, &dctl->err, sizeof(unsigned),
                                 cudaMemcpyDeviceToHost, c->stream));
        CUDA_TRY(cudaStreamSynchronize(c->stream));
        CUDA_TRY(cudaMemsetAsync(field, 0, bytes, c->stream));
        return code_of(c->h_ctl->err);
    };
    unsigned long long have = 0;
    AWPM_TRY(take(&dctl->cycles, sizeof(unsigned long long), &have));
    unsigned long long total = have;
    for (int32_t phase = 0; phase <= n; ++phase) {
        S.phases += 1;
        launch_mcm_phase(d, sh, k);
        AWPM_TRY(check_sink(k));
        for (int32_t level = 0; level <= n; ++level) {
            int32_t live = 0;
            AWPM_TRY(take(&dctl->live, sizeof(int32_t), &live));
            if (live <= 0)
                break;
            S.levels += 1;
            launch_mcm_level(d, sh, k);
            AWPM_TRY(check_sink(k));
        }
        launch_mcm_augment(d, sh, k);
        AWPM_TRY(check_sink(k));
        unsigned long long aug = 0;
        AWPM_TRY(take(&dctl->pass_flips, sizeof(unsigned long long), &aug));
        total += aug;
        if (aug == 0)
            break;
    }
    launch_mcm_store(d, sh, k);
    AWPM_TRY(check_sink(k));
    if (l_m != 1)
        CUDA_TRY(cudaMemcpyAsync(mate, dmate, sizeof(int32_t) * n, cudaMemcpyDeviceToHost,
                                 c->stream));
    CUDA_TRY(cudaEventRecord(c->ev_b, c->stream));
    CUDA_TRY(cudaEventSynchronize(c->ev_b));
    float ms = 0.f;
    CUDA_TRY(cudaEventElapsedTime(&ms, c->ev_a, c->ev_b));
    S.cardinality = (int32_t)total;
    S.ms_total = ms;
    if (stats)
        *stats = S;
    return AWPM_OK;
}

static int weights_once(awpm_ctx *ctx, int32_t n, const int32_t *colptr, const int32_t *rowidx,
                        const double *values, int32_t mode, double *weight_out, bool thin)
{
    awpm_ctx *c = ctx;
    CUDA_TRY(cudaSetDevice(c->device));
    const int l_colptr = where(c, colptr), l_rowidx = where(c, rowidx), l_a = where(c, values),
              l_out = where(c, weight_out);
    if (l_colptr < 0 || l_rowidx < 0 || l_a < 0 || l_out < 0)
        return AWPM_ERR_INVALID_ARG;
    int32_t nnz = 0;
    if (l_colptr == 1) {
        CUDA_TRY(cudaMemcpyAsync(c->h_ctl, colptr + n, sizeof(int32_t), cudaMemcpyDeviceToHost,
                                 c->stream));
        CUDA_TRY(cudaStreamSynchronize(c->stream));
        std::memcpy(&nnz, c->h_ctl, sizeof(int32_t));
    } else {
        nnz = colptr[n];
    }
    if (nnz < 0 || nnz > kMaxEntries || (nnz > 0 && (!rowidx || !values || !weight_out)))
        return AWPM_ERR_INVALID_ARG;
    const int32_t ntiles = (int32_t)(((int64_t)nnz + kTile - 1) / kTile);
    const bool small = c->clusters && weights_cluster(ntiles, n);
    thin = thin || small || weights_thin(ntiles, n);
    AWPM_TRY(ensure(c, c->wt_max, sizeof(unsigned long long) * n));
    if (!thin) {
        AWPM_TRY(ensure(c, c->wt_scale, sizeof(Scale) * n));
        AWPM_TRY(ensure(c, c->tile_col, sizeof(int32_t) * ((size_t)ntiles + 1)));
        AWPM_TRY(ensure(c, c->starts, sizeof(uint32_t) * (((size_t)nnz + 31) / 32 + 1)));
    }
    AWPM_TRY(ensure(c, c->ctl, sizeof(Ctl)));
    double *dout = weight_out;
    if (l_out != 1) {
        AWPM_TRY(ensure(c, c->wt_stage, sizeof(double) * (size_t)nnz));
        dout = (double *)c->wt_stage.p;
    }
    Shape sh = shape_of(c, false, AWPM_LOOKUP_BSEARCH, true, ntiles);
    sh.cluster = small;
    Work &wk = *c->h_work;
    std::memset(&wk, 0, sizeof(Work));
    wk.n = n;
    wk.nnz = nnz;
    wk.ntiles = ntiles;
    AWPM_TRY(stage_in(c, c->s_colptr, colptr, (size_t)n + 1, l_colptr, &wk.colptr));
    AWPM_TRY(stage_in(c, c->s_rowidx, rowidx, (size_t)nnz, l_rowidx, &wk.rowidx));
    AWPM_TRY(stage_in(c, c->s_w, values, (size_t)nnz, l_a, &wk.wt_a));
    wk.wt_out = dout;
    wk.wt_max = (unsigned long long *)c->wt_max.p;
    if (!thin) {
        wk.wt_scale = (Scale *)c->wt_scale.p;
        wk.tile_col = (int32_t *)c->tile_col.p;
        wk.starts = (uint32_t *)c->starts.p;
    }
    wk.wt_mode = mode;
    wk.ctl = (Ctl *)c->ctl.p;
    CUDA_TRY(cudaMemcpyAsync(c->d_work.p, c->h_work, sizeof(Work), cudaMemcpyHostToDevice,
                             c->stream));
    Sink k;
    k.stream = c->stream;
    launch_weights((const Work *)c->d_work.p, sh, thin, k);
    AWPM_TRY(check_sink(k));
    if (l_out != 1 && nnz > 0)
        CUDA_TRY(cudaMemcpyAsync(weight_out, dout, sizeof(double) * (size_t)nnz,
                                 cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(cudaMemcpyAsync(c->h_ctl, wk.ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, c->stream));
    CUDA_TRY(cudaStreamSynchronize(c->stream));
    // a column without entries is no error here (no matching is asked for)
    return code_of(c->h_ctl->err & ~kErrNotPerfect);
}

int awpm_weights(awpm_ctx *ctx, int32_t n, const int32_t *colptr, const int32_t *rowidx,
                 const double *values, int32_t mode, double *weight_out)
{
    NvtxRange nvtx_range("awpm_weights");
    if (!ctx || n < 0 || (n > 0 && !colptr) ||
        (mode != AWPM_WEIGHTS_SUM && mode != AWPM_WEIGHTS_PRODUCT))
        return AWPM_ERR_INVALID_ARG;
    if (n == 0)
        return AWPM_OK;
    std::lock_guard<std::mutex> lk(ctx->mu);
    int rc = weights_once(ctx, n, colptr, rowidx, values, mode, weight_out, false);
    if (rc == AWPM_ERR_BUDGET || (rc == AWPM_ERR_OOM && !ctx->injected)) {
        // no room for the columns' scales and the tiles' columns: the form
        // that keeps only the row maxima
        CUDA_TRY(cudaStreamSynchronize(ctx->stream));
        release(ctx, ctx->wt_scale);
        release(ctx, ctx->tile_col);
        release(ctx, ctx->starts);
        rc = weights_once(ctx, n, colptr, rowidx, values, mode, weight_out, true);
    }
    return rc;
}

int awpm_search(awpm_ctx *ctx, int32_t n, const int32_t *colptr, const int32_t *rowidx,
                const double *weight, const int32_t *mate, double *stepc_gain, int32_t *stepc_row,
                awpm_stats *stats)
{
    NvtxRange nvtx_range("awpm_search");
    if (!ctx)
        return AWPM_ERR_INVALID_ARG;
    Request r;
    r.n = n;
    r.colptr = colptr;
    r.rowidx = rowidx;
    r.weight = weight;
    r.mate_in = mate;
    r.search_only = true;
    r.gain_out = stepc_gain;
    r.row_out = stepc_row;
    return solve_sync(ctx, r, stats, nullptr);
}

}  // extern "C"

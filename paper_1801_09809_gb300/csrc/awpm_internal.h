// Internal declarations shared by the kernels and the host side of libawpm.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "awpm.h"
#include "awpm_fixed.h"
#include "awpm_rules.h"

namespace awpm {

// Error bits raised on the device; the host maps them to the public code
// (priority INVALID > UNSORTED > NONFINITE > NOTPERF > INTERNAL > TIMEOUT).
constexpr unsigned kErrInvalid = 1u;
constexpr unsigned kErrUnsorted = 2u;
constexpr unsigned kErrNonfinite = 4u;
constexpr unsigned kErrNotPerfect = 8u;
constexpr unsigned kErrInternal = 16u;  // a consistency check of the library's own state failed
constexpr unsigned kErrTimeout = 32u;   // a bounded retry loop or level loop gave up
constexpr unsigned kErrBounds = 64u;    // AWPM_DEBUG_BOUNDS builds: an index check failed
constexpr unsigned kErrRetry = 128u;    // small-matrix kernel: something is wrong with the
                                        // input (or it is not for this kernel); the general
                                        // path is to solve it

// Public code of a set of device error bits (host side).
inline int awpm_code_of_bits(unsigned err)
{
    if (err & kErrInvalid)
        return AWPM_ERR_INVALID_ARG;
    if (err & kErrUnsorted)
        return AWPM_ERR_UNSORTED_OR_DUP;
    if (err & kErrNonfinite)
        return AWPM_ERR_NONFINITE;
    if (err & kErrNotPerfect)
        return AWPM_ERR_NOT_PERFECT;
    if (err & (kErrInternal | kErrBounds))
        return AWPM_ERR_INTERNAL;
    if (err & kErrTimeout)
        return AWPM_ERR_TIMEOUT;
    if (err)
        return AWPM_ERR_INTERNAL;
    return AWPM_OK;
}

// Step-C record of a root column j (Algorithm 5): best positive gain, the
// position p of (i, j) in column j and the position q of the closing entry
// (m_j, m_i) in column m_i.  g == 0 means "no cycle".
struct alignas(16) Rec {
    double g;
    int32_t p;
    int32_t q;
};

// Per-row view of the column matched to row i (m_i), in two arrays:
//   rsig[i]   a 64-bit signature of column m_i's rows (the bits sig_mask(r)
//             set for every stored row r): a clear bit proves that the
//             closing entry (m_j, m_i) is absent without touching the column;
//             every candidate gathers these 8 bytes;
//   rrange[i] where column m_i's rows sit in the CSC arrays and the matched
//             weight w(i, m_i): read only for the candidates that pass.
// Both are rewritten whenever row i changes mate.
struct alignas(16) RowRange {
    int32_t s;
    int32_t e;
    double w;
};

// Maximum matching: the best offer a row received at this level (order key
// of the edge weight, then the lowest column), or a tree's end (order key of
// its last edge, then the lowest row); one 128-bit compare-and-swap updates
// both fields together.
struct alignas(16) Off {
    long long key;
    int32_t who;
    int32_t pad;
};

// Step-D selection at a key column k (Algorithm 6): best gain and its root j,
// and the pass that wrote it (Work::epoch0 + passes run + 1): a record of
// another pass counts as empty, so none has to be cleared.
struct alignas(16) Sel {
    double g;
    int32_t j;
    int32_t epoch;
};

// Device-resident control block of one solve.
struct Ctl {
    unsigned int err;            // kErr* bits
    int32_t active;              // 1 while the pass loop continues; maximum matching: the
                                 // next step is one cluster's
    int32_t iterations;          // passes run
    int32_t converged;           // last pass flipped nothing
    int32_t max_passes;          // cap on passes
    int32_t live;                // greedy selection: winners still undecided
    int32_t ps_done;             // greedy selection: the pass was decided by k_ps_small
    int32_t ps_count;            // its winners, then those undecided
    int32_t nonempty;            // maximum matching: no column is empty
    int32_t phase_levels;        // maximum matching: levels of the running phase
    // maximum matching: tiles and columns listed for the next level (counted
    // with one 64-bit atomic), columns of the running one
    alignas(8) int32_t level_tiles;
    int32_t front_next;
    int32_t front_n;
    uint32_t flip_done;          // blocks done with the pass's flip (graph form)
    uint32_t level_done;         // maximum matching: blocks done with the level's last step
    int32_t touched;             // maximum matching: rows listed in mtouch this level
    unsigned long long levels;   // maximum matching: search levels run
    unsigned long long pass_flips;   // cycles flipped in the running pass
    unsigned long long cycles;       // cycles flipped in total
    unsigned long long candidates;   // Step A requests (i > m_j)
    unsigned long long found;        // closing edge present
    unsigned long long positive;     // closing edge present and g > 0
    // incremental passes: this pass's changes of the three counts (signed),
    // the counts of the last pass, and the cycles it flipped
    unsigned long long d_candidates, d_found, d_positive;
    unsigned long long cur_candidates, cur_found, cur_positive;
    unsigned long long last_flips;
    double weight_in;
    double weight_out;
    int32_t small_nnz;           // small single solve: nonzeros
    int32_t small_pad;
};

// Batched solve of many independent matrices as one block-diagonal union
// (count > 0).  Matrix b owns columns and rows [n_off[b], n_off[b+1]).
struct BatchWork {
    int32_t count;
    int32_t pad;
    const int32_t *n_off;   // count + 1 offsets
    int32_t *colmat;        // matrix of each column
    int32_t *tilemat;       // matrix of each tile's first nonzero | kTileSingle
    int32_t *mdone;         // matrix finished (converged or pass cap)
    int32_t *miter;         // passes run per matrix
    int32_t *mconv;         // converged per matrix
    int32_t *mnnz;          // nonzeros per matrix
    unsigned long long *mflips;   // cycles flipped in the running pass
    unsigned long long *mcycles;  // cycles flipped in total
    double *mw_in;
    double *mw_out;
    int32_t *active;        // matrices still running after a pass
    int32_t *tlist;         // tiles the next pass searches (running matrices,
                            // and every tile spanning two matrices)
    int32_t *tlist_n;       // their number
};

// Tile whose nonzeros all belong to one matrix.
constexpr int32_t kTileSingle = (int32_t)0x80000000;

// Rows whose mate the last pass changed, as folded bitmaps: bit r mod 2^17 of
// the small one, bit r mod 2^k of the large one (2^k >= n, at most 2^20; only
// kept for n > 2^17, and then searched instead of the small one after a pass
// of more than kSmallFlips flips).
constexpr int kMapSmallBits = 1 << 17;
constexpr int kMapLargeBits = 1 << 20;
constexpr unsigned kSmallFlips = 1024;

// Solves of small matrices by one block each (classes: kSmallMaxN): the shared
// memory that a matrix needs with `warps` warps, with or without the columns'
// signatures (the rings; the column pointers; four bitmaps; signatures; three
// 16-bit arrays).
constexpr int kSmallOne = kSmallClasses;  // the single matrix's class
constexpr int kSmallWarps[kSmallClasses + 1] = {32, 16, 8, 16};
__host__ __device__ constexpr size_t small_smem(int32_t n, int warps, bool sigs)
{
    return (size_t)warps * 512 + 4 * ((size_t)n + 1) + 16 * ((size_t)n / 32 + 1) +
           (sigs ? 4 * (size_t)n : 0) + 6 * (size_t)n + 4;
}
// Dynamic shared memory of a class's blocks (the largest class keeps no
// signatures above about 14,700 columns).
constexpr size_t small_class_smem(int c)
{
    // (and room for the bitmap of marked tiles)
    return c == 0 || c == kSmallOne
               ? small_smem(kSmallMaxN[0], kSmallWarps[c], false) + 2560
               : small_smem(kSmallMaxN[c], kSmallWarps[c], true) + 512;
}

// Descriptor of one solve.  It lives in device memory and every kernel reads
// it from there, so launch configurations do not depend on the problem and
// one instantiated CUDA graph serves every problem of a context: a new
// problem only rewrites the descriptor before the graph launch.
struct Work {
    int32_t n;
    int32_t nnz;
    int32_t ntiles;
    int32_t max_passes;
    int32_t lookup;     // AWPM_LOOKUP_BSEARCH, _HASH or _ROWMARK
    int32_t rec_clean;  // the Step-C and Step-D records of columns [0, n) are all empty
    int32_t inc;        // passes after the first search only what the last flips affect
    int32_t epoch0;     // Step-D records of this solve's passes: epochs epoch0 + 1, ...
    int32_t map_bits;   // bits of the large folded bitmap (0: none kept)
    int32_t bloom_min;  // columns with more rows than this have a Bloom filter
    const int32_t *colptr;
    const int32_t *rowidx;
    const double *w;
    const int32_t *mate_in;
    int32_t *mc;        // row matched to column j
    int32_t *mr;        // column matched to row i
    double *wm;         // w(mc[j], j)
    unsigned long long *rsig;  // per row i: signature of the rows of column mr[i]
    RowRange *rrange;          // per row i: that column's range and w(i, mr[i])
    unsigned long long *colsig;  // per column: signature of its rows
    unsigned long long *htab;    // per-column hash tables (2 slots per nonzero), or null
    uint32_t *bloom;    // blocked Bloom filters of the long columns (a word per 4 nonzeros), or null
    Rec *best;          // Step-C records
    Sel *dsel;          // Step-D selections
    uint32_t *winbits;  // bit j: column j holds a Step-C winner this pass
    int32_t *wkey;      // key column k of winner j (set by Step D), ~k if dropped
    // small matrices: numbers of matrices by class (order, first and count of
    // each class), the classes' queues, found and positive bits of the
    // matrices' tiles (tile x of matrix b at (p0 >> 5) + b + x, p0 its first
    // entry), most nonzeros; single solves: where nnz is
    const int32_t *small_order;
    int32_t small_first[kSmallClasses];
    int32_t small_count[kSmallClasses];
    int32_t small_smem[kSmallClasses + 1];
    int32_t small_cap;
    int32_t *small_next;
    uint32_t *small_fb;
    uint32_t *small_pb;
    int32_t *small_c0;      // columns of the tiles' first entries
    uint32_t *small_sig;    // single solves: the columns' signatures
    const int32_t *small_nnz;
    int32_t *small_out;     // the matchings (global rows)
    int32_t small_off[2];   // single solves: their n_off
    // incremental passes: per entry, a bit each for "closing entry found" and
    // "positive gain" at its last evaluation; per column whose mate changed
    // the row matched to it before; two sets (of alternate passes) of bitmaps:
    // changed rows (folded), columns to search whole, columns to search by
    // their entries of positive gain, tiles of either
    uint32_t *foundbits;
    uint32_t *posbits;
    int32_t *mc_old;
    uint32_t *map_small[2];
    uint32_t *map_large[2];
    uint32_t *colfull[2];
    uint32_t *colpos[2];
    uint32_t *tilemark[2];
    int32_t *tile_col;  // column holding the first nonzero of each tile
    uint32_t *starts;   // bit p set when a column starts at nonzero p
    Ctl *ctl;
    double *wpart;      // partial sums of the weight reduction
    BatchWork bw;       // batched solve (bw.count > 0), else zero
    // greedy maximal matching: per row the best free entry (order key, column,
    // round; kMatched once the row is matched), per column (order key,
    // position, round)
    Off *grow;
    Off *gcol;
    uint8_t *gdead;     // per group of eight tiles: the tiles without a free entry
    // greedy (Pettie-Sanders) selection: per column the first remaining
    // winner touching it; bitmaps of undecided and kept winners and of the
    // columns of kept cycles
    Sel *psel;
    uint32_t *pslive;
    uint32_t *pstaken;
    uint32_t *psused;
    // weights from matrix values: values, output, the columns' and then the
    // rows' maxima (bit patterns of positive doubles), the same with their
    // reciprocals, mode (0 scaled magnitude, 1 its log)
    const double *wt_a;
    double *wt_out;
    unsigned long long *wt_max;
    Scale *wt_scale;
    int32_t wt_mode;
    int32_t wt_pad;
    // maximum cardinality matching: tree of a column, column that reached a
    // row, bitmaps and lists of the levels, per row the best offer (key,
    // column), per tree its end (key of the last edge, row); mate in/out
    int32_t *mroot;
    int32_t *mrpar;
    uint32_t *mfront;   // bit c: column c is in the frontier
    uint32_t *mreach;   // bit r: row r was reached in this phase
    uint32_t *mtmark;   // bit t: tile t, shared by columns, is listed
    int32_t *mfl;       // columns of the frontier
    Off *mroff;         // per row: the level's best offer (key, column)
    Off *mtend;         // per tree (root column): its end (key of the last edge, row)
    int32_t *mtouch;    // rows offered something at this level (each once), then
                        // the columns matched to them
    int32_t *mmate;
    int32_t *mcolof;    // column of every entry
    int32_t *mtiles;    // tiles holding a frontier column, this level
    int64_t mtiles_cap; // capacity of mtiles
    // row marking: per row the mark of its columns (a signature), the
    // transpose (row pointers; CSC positions row by row, ascending), the
    // radix sort that builds it (keys and values in two buffers each, digit
    // counts per block tile, then their offsets; sums per scan chunk)
    unsigned long long *rowsig;
    int32_t *trowptr;
    int32_t *tpos;
    int32_t *rs_key[2];
    int32_t *rs_val[2];
    int32_t *rs_hist;
    int32_t *rs_sums;
    int32_t rs_tiles;   // block tiles of kRsTile entries
    int32_t rs_passes;  // 8-bit digits of the largest row index (at least 1)
};

// Radix sort of the transpose: 256 threads, 8 entries each per block tile,
// 8-bit digits; scans run over chunks of 2048 counts.
constexpr int kRsThreads = 256;
constexpr int kRsItems = 8;
constexpr int kRsTile = kRsThreads * kRsItems;
constexpr int kRsBins = 256;
constexpr int kScanChunk = kRsThreads * 8;

// Launch shape of a context: fixed grids sized by the GPU, not the problem.
struct Shape {
    int num_sms;
    int search_bps;     // resident blocks per SM of the chosen search kernel
    int lookup;         // AWPM_LOOKUP_BSEARCH, _HASH or _ROWMARK
    bool batch;
    bool wide;          // search kernel takes four tiles per warp round (else one)
    int search_waves;   // size class: 2 when there are at least 64 tiles per resident
                        // search warp, else 1 (keys the cached graphs; Step D's grid)
    int select;         // AWPM_SELECT_STEP_D or AWPM_SELECT_GREEDY
    bool cluster = false;  // greedy and maximum matching: loops run in one cluster
    bool greedy = false;   // greedy matching: the matched weights are in gcol
    bool inc = false;   // passes after the first are incremental
    bool large = false; // n > kMapSmallBits: the incremental search's large form
};

constexpr int kWsumBlocks = 1024;
constexpr int kWsumThreads = 256;

// Rows above which a column has a Bloom filter, by the matrix's size, and the
// value that gives none to any.
int32_t bloom_min(int32_t n, int32_t nnz);
constexpr int32_t kNoBloom = 0x7fffffff;

// Where launches go: a stream (launched at once, asynchronously) or a graph
// (appended as kernel nodes, each depending on the previous one).  Graphs are
// built node by node rather than by stream capture, so building one never
// interacts with work other threads submit meanwhile.
struct Sink {
    cudaStream_t stream = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphNode_t last = nullptr;
    cudaError_t err = cudaSuccess;
    void launch(const void *func, unsigned grid, unsigned block, void **args, unsigned smem = 0);
};

// Solves of small matrices: a batch (counts: matrices per class), or one
// matrix (smem: its Work::small_smem).
cudaError_t small_setup();
struct SmallStreams {
    cudaStream_t side[kSmallClasses - 1] = {};
    cudaEvent_t fork = nullptr, join[kSmallClasses - 1] = {};
};
void launch_small_batch(const Work *d, const Shape &sh, const int32_t *counts,
                        const SmallStreams &ss, Sink &k);
void launch_small_one(const Work *d, int32_t smem, Sink &k);
// The column pointers at count + 1 offsets in [0, n], into at[].
void launch_small_entries(const int32_t *off, const int32_t *colptr, int32_t n, int32_t count,
                          int32_t *at, Sink &k);

// Launch sequences; `d` is the device copy of the Work.
void launch_init(const Work *d, const Shape &sh, Sink &k);
void launch_weight_sum(const Work *d, const Shape &sh, bool out, Sink &k);
void launch_search(const Work *d, const Shape &sh, Sink &k);
// The search of a pass after the first with Shape::inc.
void launch_search_inc(const Work *d, const Shape &sh, Sink &k);
// Allow the incremental search kernels their shared memory (once per device).
cudaError_t search_inc_setup();
void launch_select_and_flip(const Work *d, const Shape &sh, Sink &k);
// Graph form for single problems with Step D: the selection and the flip,
// whose last block also ends the pass (no separate control kernel).
void launch_select_flip_control_graph(const Work *d, const Shape &sh,
                                      cudaGraphConditionalHandle h, Sink &k);
// Greedy selection: the kernels before the rounds (keys, undecided set,
// condition of the rounds' loop), one round (the loop condition is set at
// its end), and the kernels after (records for the flip).  With graph ==
// false the conditions are not set; the host reads Ctl::live instead.
void launch_greedy_select_begin(const Work *d, const Shape &sh, bool graph,
                                cudaGraphConditionalHandle h, Sink &k);
void launch_greedy_select_round(const Work *d, const Shape &sh, bool graph,
                                cudaGraphConditionalHandle h, Sink &k);
void launch_greedy_select_end_and_flip(const Work *d, const Shape &sh, Sink &k);
// The checks of the pattern and the entries, and the start marks.
void launch_check_colptr(const Work *d, const Shape &sh, Sink &k);
void launch_mark_starts(const Work *d, const Shape &sh, Sink &k);
void launch_check_entries(const Work *d, const Shape &sh, Sink &k);
// The column-pointer check with the start marks (k_check_mark).
void launch_check_mark(const Work *d, const Shape &sh, Sink &k);
// Weights from matrix values (equilibration, Options A / B).
// thin: the form without wt_scale, tile_col and starts.
void launch_weights(const Work *d, const Shape &sh, bool thin, Sink &k);
// Maximum cardinality matching: load and check the starting matching; start
// a phase (Ctl::live = free columns); one level of the searches (Ctl::live =
// next frontier); augment (Ctl::pass_flips = paths augmented); write back.
void launch_mcm_load(const Work *d, const Shape &sh, Sink &k);
void launch_mcm_phase(const Work *d, const Shape &sh, Sink &k);
void launch_mcm_level(const Work *d, const Shape &sh, Sink &k);
// Graph form of a level: small levels in one cluster, then the steps, the last
// one also setting the level loop's condition.
void launch_mcm_level_graph(const Work *d, const Shape &sh, cudaGraphConditionalHandle h,
                            Sink &k);
// The phases and levels of a small problem in one kernel.
void launch_mcm_cluster(const Work *d, const Shape &sh, Sink &k);
void launch_mcm_augment(const Work *d, const Shape &sh, Sink &k);
void launch_mcm_store(const Work *d, const Shape &sh, Sink &k);
// Graph forms: the condition of the level loop (undecided frontier left),
// and the end of a phase (count it, continue while it augmented).
void launch_mcm_cond_level(const Work *d, const Shape &sh, cudaGraphConditionalHandle h, Sink &k);
void launch_mcm_cond_phase(const Work *d, const Shape &sh, cudaGraphConditionalHandle h, Sink &k);
void launch_control(const Work *d, const Shape &sh, bool graph, cudaGraphConditionalHandle h,
                    Sink &k);
void launch_export_stepc(const Work *d, const Shape &sh, double *gain, int32_t *row, Sink &k);
// Greedy maximal matching: state reset and input checks; one round (the
// control kernel ends the loop after a round that matched nothing).
void launch_greedy_init(const Work *d, const Shape &sh, Sink &k);
// The rounds of a small problem in one kernel.
void launch_greedy_cluster(const Work *d, const Shape &sh, Sink &k);
void launch_greedy_round(const Work *d, const Shape &sh, bool graph, cudaGraphConditionalHandle h,
                         Sink &k);
// Resident blocks per SM of the search kernel for a lookup strategy.
int search_blocks_per_sm(int lookup, bool batch, bool wide);
// Waves of the search grid for a problem of ntiles tiles: 2 once every warp
// of a single wave would take at least 64 tiles (more blocks than resident
// slots shorten the tail of uneven warps), else 1.
int search_waves(int num_sms, int search_bps, int32_t ntiles);
// Whether the search kernel takes four tiles per warp round (default on; the
// environment variable AWPM_SEARCH_WIDE=0/1 overrides it, a tuning knob).
bool default_search_wide();
// Whether single-problem searches use the pipelined kernel (default on; the
// environment variable AWPM_SEARCH_PIPE=0/1 overrides it, a tuning knob).
bool search_pipe();

}  // namespace awpm

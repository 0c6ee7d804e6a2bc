// Index arithmetic and size rules in plain C++, with host and device forms, so
// that both are tested on the CPU.
#pragma once

#include <stdint.h>

#include "awpm_fixed.h"

namespace awpm {

// Nonzeros handled by one warp per tile of the edge-parallel kernels; tiles
// start at multiples of kTile, so tile t owns word t of the column-start
// bitmap.
constexpr int kTile = 32;

// Largest nnz: the positions of all tiles' lanes, and of those of one tile past
// the last, stay in int32.
constexpr int32_t kMaxEntries = 0x7fffffff - 63;

// Position of a lane's entry in tile t.  A kernel that looks ahead asks for
// tiles past the last one: they get the positions of tile ntiles, which are at
// or past nnz and never wrap (the product t * kTile does, close to kMaxEntries).
AWPM_HD int32_t tile_pos(int32_t t, int32_t ntiles, int lane)
{
    return (t < ntiles ? t : ntiles) * kTile + lane;
}

// Most tiles of a problem whose greedy rounds run in one cluster (no column is
// empty, so they bound n).  us per call, loops in the graph against one cluster:
// 16,000 entries 229 / 172, 64,000 248 / 184, 130,000 235 / 237, 260,000 244 /
// 357 (random; the others alike).
constexpr int32_t kGmClusterTiles = 3584;

// Whether the phases and levels of a maximum matching run in one cluster.  Each
// phase walks all columns, which may be empty, 32 by 32, as its levels do the
// tiles.  us per call, loops in the graph against one cluster: random, 8,000
// columns and 100,000 entries 993 / 824, 16,000 and 190,000 1,106 / 1,067, 32,000
// and 190,000 2,536 / 2,793, 65,536 and 100,000 1,353 / 1,458, 131,072 and 10,000
// 292 / 289, 262,144 and 10,000 318 / 399, 4 M and 10,000 590 / 2,950.
constexpr int64_t kMcClusterTiles = 6656;
inline bool mcm_cluster(int32_t ntiles, int32_t n)
{
    return ntiles + (int64_t)n / 32 <= kMcClusterTiles;
}

// Forms of the weights: one cluster (a warp per column), the thin form (a warp
// per column, no scales and tile map to build, five launches), the full one.  us
// per call, full / thin / cluster (and three warp-per-column kernels on the FP64
// units, the former form): random, 8 entries a column, 8,000 entries 73 / 55 / 49
// (57), 30,000 73 / 55 / 67 (69), 120,000 71 / 55 / 161 (98), 250,000 76 / 67 /
// 296 (156), 1 M 96 / 108 / 1,049 (458); R-MAT 8,000 73 / 56 / 41 (69), 120,000
// 74 / 68 / 136 (191), 250,000 75 / 87 / 235 (313); 27-point stencil 8,000 72 /
// 55 / 40 (56).  Mostly empty columns, thin / cluster: 8,000 columns and 1,000
// entries 62 / 62, 32,000 and 1,000 62 / 98, 4,000 and 10,000 62 / 72, 4 M and
// 1,000 433 / 6,494 (the former form 1,777); 100,000 entries thin, 190,000 full:
// 131,072 columns 90, 92, 262,144 111, 92, 4 M 460, 222.
constexpr int64_t kWtClusterTiles = 384;
constexpr int32_t kWtThinTiles = 4096;
inline bool weights_cluster(int32_t ntiles, int32_t n)
{
    return ntiles + (int64_t)n / 32 <= kWtClusterTiles;
}
inline bool weights_thin(int32_t ntiles, int32_t n)
{
    return ntiles <= kWtThinTiles && n / 32 <= kWtThinTiles;
}

// Solves of small matrices by one block each: classes of sizes (the largest
// first) and the largest n of each.
constexpr int kSmallClasses = 3;
constexpr int32_t kSmallMaxN[kSmallClasses] = {20096, 7168, 2048};

// Class of a matrix of n columns, n at most kSmallMaxN[0].
inline int small_class(int32_t n)
{
    return n <= kSmallMaxN[2] ? 2 : n <= kSmallMaxN[1] ? 1 : 0;
}

// Most entries of a single solve by the small-matrix kernel (one cluster of
// eight blocks).  us per solve, by the kernel against the general path: random
// n = 300 70 / 138, n = 2,000 with 18,000 entries 75 / 139, 72,000 entries 111
// / 138, 180,000 entries 158 / 123; banded (19 passes) 4,400 entries 225 / 379,
// 30,000 entries 423 / 491, 60,000 entries 581 / 500; 5-point 39,000 entries
// 174 / 188; 27-point 22,000 entries 434 / 546, 51,000 entries 647 / 640.
constexpr int32_t kSmallOneNnz = 40960;

// Whether a solve that came back undone from that kernel, which had read the
// number of entries itself, had too many (and not an input to be refused): then
// the next ones of its size have the number read first.
inline bool small_too_many(int32_t nnz)
{
    return nnz > kSmallOneNnz;
}

// Whether a batch of small matrices is solved by a block per matrix, rather than
// as a union over the whole GPU.  A block has one SM at most, so the call lasts
// as long as its slowest matrix there, however idle the other SMs are; the union
// spreads all tiles over the GPU, but launches its kernels again for every pass.
// Both go with the number of passes, which nobody knows beforehand, so the
// rule compares what a pass costs, in ns:
//   a matrix in its block: 14,000 + 100, 58 or 34 per tile by class (256, 512 or
//     1,024 threads);
//   the union: 44,000 + 0.42 per tile still searched.  With matrices alike all
//     are to the last pass; with mixed sizes most converge before the largest.
//     Where the average has a small share of the largest's tiles, 0.4 of them
//     count.
// ms per call, union / blocks: banded, 2,000 columns (562 tiles each), 4
// matrices 0.61 / 0.91, 64 0.86 / 1.00, 256 1.86 / 1.31; banded, 20,000 (5,624),
// 16 matrices 1.15 / 2.90, 64 3.08 / 3.52; banded, 16,371 (3,581), 96 2.69 /
// 2.05; 5-point, 2,000 (311), 1 matrix 0.341 / 0.347; 27-point, 1,728 (1,228), 64
// 1.74 / 3.33, 256 4.82 / 4.33; random, 300 (83), 4 matrices 0.250 / 0.127, 2,000
// (562), 64 0.322 / 0.285 (the rule's loss: few passes); random with 100 entries
// a column, 10,000 (31,400), 4 matrices 1.26 / 11.4; sizes from 200 to 20,000, 32
// matrices 0.83 / 3.07, 512 3.58 / 6.89, 1,024 6.45 / 7.77, 2,048 12.1 / 9.43.
struct BatchLoad {
    int64_t count = 0, all = 0, largest = 0;  // matrices, their tiles, the most of one
    double block_ns = 0;                      // the slowest matrix's pass in its block
    void add(int32_t n, int64_t tiles)
    {
        constexpr double kTileNs[kSmallClasses] = {34, 58, 100};
        const double ns = 14000 + kTileNs[small_class(n)] * (double)tiles;
        ++count;
        all += tiles;
        largest = largest > tiles ? largest : tiles;
        block_ns = block_ns > ns ? block_ns : ns;
    }
    double union_ns() const
    {
        const double share = largest > 0 ? (double)all / ((double)count * (double)largest) : 1.0;
        return 44000 + 0.42 * (0.4 + 0.6 * share) * (double)all;
    }
    bool blocks_pay() const { return block_ns <= union_ns(); }
};

}  // namespace awpm

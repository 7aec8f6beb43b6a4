// Cell-sorted sampling (bf16 storage): pieces shared by the kernels of dsa3d_cells.cu.
//
// A sample reads (and its gradient writes) the eight corner rows of the grid cell it falls into.  All samples of a cell,
// whichever query they belong to, share those eight rows.  So the samples are first sorted by key cell: then the dot
// products of 16 samples with their eight corners are one m16n8k16 product chain (16 query rows x 8 key rows), the
// dK / dV contributions of 16 samples another (corners, the weights in three bf16 parts, x 16 query rows), and the
// row traffic per sample falls from eight key rows to one query row.  Nothing depends on how far the offsets reach.
// (The groups are 16 samples of one cell, so the warp-level product is the one that fits: a tcgen05 tile would hold
// 128 rows of which a cell fills 27.)
//
// Queries come in tiles of 4 x 4 x 6 (t, y, x) of one head, cells in blocks of 4 x 4 x 3 whose rows are a box of
// 5 x 5 x 4 positions.  Three cells along x: their corners are 4 x 4 rows, the sixteen rows of one product tile of
// the dK / dV sums.  cells_bin_kernel sorts the samples of a tile by the block they fall into, relative to the tile
// (bins); a block finds its samples as one segment per (tile, bin), and cells_sort_kernel lays them down cell after cell.
#pragma once
#include "dsa3d_common.cuh"
#include "dsa3d_gather.cuh"

namespace dsa3d {
namespace cells {

constexpr int kTileX = 6, kRows = 4 * 4 * kTileX; // queries per tile
constexpr int kReach = 12;                        // bins reach this far below and above the tile on every axis
constexpr int kBlockX = 3;                        // cells of a block along x (4 along t and y)
constexpr int kBinsT = 7, kBinsY = 7, kBinsX = (kTileX + 2 * kReach) / kBlockX;   // blocks of the bin grid
constexpr int kBins = kBinsT * kBinsY * kBinsX;   // 490; the bin after them takes the samples beyond
constexpr int kSegsX = kBinsX / 2, kSegs = kBinsT * kBinsY * kSegsX;   // tiles whose bins can hold a given block: 245
constexpr int kBox = 100;                         // rows of a box
constexpr int kRuns = 16, kCells = kRuns * kBlockX;   // runs of cells along x, cells of a block

// The part of a problem one pass takes: heads [m0, m0 + heads), frames [f0, f1) of queries.  Tiles are numbered
// ((head * tiles_t + tt) * tiles_y + ty) * tiles_x + tx, tile tt starts at frame f0 + 4 tt.
struct Slab {
    int m0, heads, f0, f1;
    int tiles_t, tiles_y, tiles_x;
    int blocks_t, blocks_y, blocks_x;             // blocks that samples of these queries can fall into: block b starts at cell
    int bt0;                                      // f0 + 4 (b + bt0) along t, 4 (b - 1) along y, 3 (b - 1) along x
    uint4* geo;                                   // [tile][kRows * P]: {token, ft, fy, fx}
    uint16_t* meta;                               // [tile][kRows * P]: sample | cell in its block << 8
    uint32_t* seg;                                // [tile][kBins + 1]: start | count << 16
    float4* sorted;                               // samples in the order of (block, cell): {ft, fy, fx, token (bits)}
    uint32_t* place;                              // of the same sample in stats and coef
    uint32_t* first;                              // [block][kCells + 1]: where the samples of a cell begin in `sorted`
    uint32_t* used;                               // samples laid down so far
    float* stats;                                 // [head][frame of the slab][y][x][P][8]
    float2* coef;                                 // [head][...][P]: scale dS, alpha (sign bit: marked, see cells_query_kernel)
    int* marked;                                  // is any sample marked
};

// Place of sample p of token n in stats / coef (in samples).
__device__ __forceinline__ long long sample_at(const Slab& s, const Problem& pr, int m, int n, int p) {
    const long long frame = static_cast<long long>(pr.H) * pr.W;
    return ((m - s.m0) * (frame * (s.f1 - s.f0)) + (n - frame * s.f0)) * pr.P + p;
}

// Cell (t, y, x) of a block is number (4 t + y) * 3 + x; box rows likewise, 5 x 5 x 4.
__device__ __forceinline__ int cell_t(int cell) { return cell / 12; }
__device__ __forceinline__ int cell_y(int cell) { return (cell / 3) & 3; }
__device__ __forceinline__ int cell_x(int cell) { return cell % 3; }
__device__ __forceinline__ int box_row(int cell) { return cell_t(cell) * 20 + cell_y(cell) * 4 + cell_x(cell); }
__device__ __forceinline__ int box_step(int corner) { return (corner >> 2) * 20 + ((corner >> 1) & 1) * 4 + (corner & 1); }

}  // namespace cells
}  // namespace dsa3d

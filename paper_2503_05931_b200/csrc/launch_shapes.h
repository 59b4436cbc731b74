// The shape of the tensor-core vocabulary projection: row tile, ring and shared memory.  Plain C++ (no CUDA), so that the
// sizes are also checked on the host, over every row count and model width.
#pragma once
#include <algorithm>
#include <cstddef>

namespace aed {
namespace tc {

constexpr int kBlockK = 64;                    // bf16 elements per k-block = one 128-byte swizzle row
constexpr int kTileM = 128;
constexpr int kATileBytes = kTileM * kBlockK * 2;
constexpr int kMaxStages = 8;
constexpr int kProducerWarps = 8;              // (a k-block is three copies)
constexpr int kRowPitch = kTileM + 4;          // floats between the rows of an accumulator tile in shared memory (bank spread)
constexpr int kTcSmemBudget = 200 * 1024;

}  // namespace tc

// MMA N (a multiple of 16) for rows_ub rows in tiles of at most `most`: as few tiles as possible, of equal size, because
// a tile's operand traffic and tensor time go with its N whether its rows are real or padding.  (Tiles of a power of two
// against this, per step of the 24-layer model: 72 rows 1387 -> 1278 us, 136 rows 2109 -> 1856, 192 rows 2323 -> 2120.)
inline int tc_n_tile(int rows_ub, int most)
{
    const int tiles = (rows_ub + most - 1) / most;
    return std::max(16, ((rows_ub + tiles - 1) / tiles + 15) / 16 * 16);
}

struct VocabShape {
    int n_tile, row_tiles, stages, producers;
    size_t smem;                               // dynamic shared memory, the alignment of the ring included
};
inline VocabShape vocab_shape(int rows_ub, int k_blocks)
{
    VocabShape s;
    s.n_tile = tc_n_tile(rows_ub, 256);
    s.row_tiles = (rows_ub + s.n_tile - 1) / s.n_tile;
    const int stage_bytes = tc::kATileBytes + 2 * s.n_tile * tc::kBlockK * 2;
    s.stages = std::min({tc::kTcSmemBudget / stage_bytes, tc::kMaxStages, k_blocks});
    // every ring stage belongs to one issuing thread: as many producers as stages (at most one per producer warp)
    s.producers = std::min(s.stages, tc::kProducerWarps);
    s.stages -= s.stages % s.producers;
    // The ring, then over the same memory the accumulator's rows.  These need more than the ring where that has one stage only
    // (d_model 64, row tiles of 64 and more: 528 bytes a row against 16 KB + 256 bytes a row).
    s.smem = std::max((size_t)s.stages * stage_bytes, (size_t)s.n_tile * tc::kRowPitch * sizeof(float)) + 1024;
    return s;
}

}  // namespace aed

// Launch shapes that depend on sizes alone: row tile, ring and shared memory of the tensor-core vocabulary projection; warps of a
// cross-attention block; rows of the warp-level projections.  Plain C++ (no CUDA), so that they are also checked on the host,
// over every row count and model width.
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdlib>

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

// The same for pairs of blocks, each with half of the rows, in 16s.
inline int tc_pair_tile(int rows_ub, int most)
{
    const int tiles = (rows_ub + most - 1) / most;
    return std::max(32, ((rows_ub + tiles - 1) / tiles + 31) / 32 * 32);
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

// Most rows that the warp-level projections take (two halves of three row tiles of 8, step_gemv.cuh), and what AED_DEC_GEMV_ROWS makes of
// it: fewer, from 1 on.  A setting of more rows means all that there are; none, or none of these, the default.
constexpr int kFewRows = 48;
inline int few_row_setting(const char *text)
{
    const int rows = text ? std::atoi(text) : 0;
    return rows >= 1 ? std::min(rows, kFewRows) : kFewRows;
}

// The encoder outputs of the rows of a step, as far as the host knows them.
struct EncoderFrames {
    int rows = 0, longest = 0;
    long long sum = 0;
    void add(int frames)
    {
        ++rows;
        longest = std::max(longest, frames);
        sum += frames;
    }
    void add(const EncoderFrames &o)
    {
        rows += o.rows;
        longest = std::max(longest, o.longest);
        sum += o.sum;
    }
};

// Cross-attention of many rows with short encoder outputs: 4 warps per (row, head) instead of 8.  pairs: (row, head) pairs of the grid.
// With more than 4 blocks of 8 warps per SM the blocks come in waves, and each wave pays for a block's start, its statistics and its
// merge; blocks of half the size make half as many waves.  Two things speak against it.
//  * Long rows in general: an SM has as many loads in flight either way, and the rows that are left at the end of a launch are done
//    sooner with 8.  So the mean is limited, to more frames where a frame is half the bytes.  24 layers, 16 heads, us per step, 8 -> 4
//    warps, 128 / 200 / 400 rows of one length: 130 frames 1535 / 1964 / 2914 -> 1450 / 1873 / 2607, 192 frames 1594 / 2068 / 3076 -> 1561 /
//    2051 / 3038, 220 frames 1633 / 2122 / 3272 -> 1644 / 2176 / 3220; 8-bit store, 250 frames 1567 / 2004 / 3081 -> 1511 / 1926 / 2876,
//    384 frames 1722 / 2240 / 3638 -> 1707 / 2200 / 3496.
//  * One long row among few: it decides when the launch ends, and takes twice as long with 4.  How long it may be grows with the blocks
//    that an SM has to work through meanwhile: 30 frames per block, until beyond 10 blocks per SM the longest that were tried (500) cost
//    2 % at most.  bf16 / 8-bit store, change of the step in %: log-normal lengths (sigma 0.7, median 130, longest 408 to 500) at 40 / 48 /
//    64 / 80 / 96 / 112 / 128 rows +7.7 / +8.3 / +6.1 / +1.9 / -0.9 / -2.5 / -4.4 and +9.0 / +9.1 / +5.3 / +1.9 / -0.7 / -2.2 / -3.7; uniform up
//    to 250 frames +4.8 / +3.8 / +0.7 / -2.5 / -4.5 / -5.0 / -6.1 and +6.1 / +6.0 / +1.1 / -1.8 / -4.4 / -5.9 / -6.9; half 40 and half 190 +1.6 /
//    +0.5 / -1.0 / -4.6 / -5.9 / -6.2 / -7.1 and +3.3 / +2.0 / -0.6 / -4.3 / -5.7 / -6.8 / -7.5; all 130 -2.5 / -3.9 / -4.0 / -3.5 / -4.2 / -4.9 /
//    -5.6 and -0.6 / -2.5 / -4.1 / -4.0 / -4.8 / -6.3 / -6.6.  (The mean alone, as it was, lost up to 17 % below 96 rows.)
inline bool few_cross_warps(long long pairs, int sm_count, const EncoderFrames &f, bool eight_bit_store)
{
    return pairs > 4ll * sm_count && f.sum <= (eight_bit_store ? 384ll : 192ll) * f.rows &&
           (pairs > 10ll * sm_count || (long long)f.longest * sm_count <= 30 * pairs);
}

}  // namespace aed

// Host check of launch_shapes.h (no GPU): whatever the row count and the model width, the dynamic shared memory of the
// vocabulary projection holds both things that live in it one after the other, the ring and the accumulator's rows.  And the
// rule for smaller cross-attention blocks, on batches whose step times on either side of it are known.
#include <cstdio>

#include "../paper_2503_05931_b200/csrc/launch_shapes.h"

using namespace aed;

// rows utterances, every n-th of them of `b` frames and the others of `a`
static bool smaller(int rows, int a, int b, int n, bool eight_bit)
{
    EncoderFrames f;
    for (int u = 0; u < rows; ++u) f.add(u % n == 0 ? b : a);
    return few_cross_warps(16ll * rows, 148, f, eight_bit);
}

static bool cross_warps_ok()
{
    bool ok = true;
    for (bool eight_bit : {false, true}) {
        ok = ok && smaller(64, 130, 130, 1, eight_bit) && smaller(128, 130, 130, 1, eight_bit) && smaller(400, 130, 130, 1, eight_bit);
        // at most 4 blocks per SM
        ok = ok && !smaller(36, 10, 10, 1, eight_bit) && smaller(40, 10, 10, 1, eight_bit);
        // half short, half long; a few very long ones: longest against the blocks per SM, not the mean
        ok = ok && !smaller(40, 60, 300, 2, eight_bit) && !smaller(64, 60, 300, 2, eight_bit) && smaller(128, 60, 300, 2, eight_bit);
        ok = ok && !smaller(48, 100, 500, 16, eight_bit) && !smaller(64, 100, 500, 16, eight_bit) && !smaller(88, 100, 500, 16, eight_bit) &&
             smaller(128, 100, 500, 16, eight_bit);
        // a longer longest, or a longer mean, never brings the smaller block back
        for (int rows = 1; rows <= 512; ++rows) {
            bool before = true;
            for (int frames = 1; frames <= 600; ++frames) {
                const bool now = smaller(rows, 1, frames, 4, eight_bit);
                ok = ok && (before || !now);
                before = now;
            }
        }
    }
    // long on average
    ok = ok && smaller(128, 192, 192, 1, false) && !smaller(128, 193, 193, 1, false) && !smaller(400, 250, 250, 1, false);
    ok = ok && smaller(128, 384, 384, 1, true) && !smaller(128, 385, 385, 1, true);
    return ok;
}

// Row tiles of the pairs of blocks: whole 32s (halves of 16 rows, an MMA of a multiple of 64 columns, at most 256), as many as needed, none empty.
static bool pair_tiles_ok()
{
    bool ok = true;
    for (int rows = 1; rows <= 2048; ++rows) {
        const int n = tc_pair_tile(rows, 128), tiles = (rows + n - 1) / n;
        ok = ok && n % 32 == 0 && n >= 32 && n <= 128 && tiles * n >= rows && (tiles - 1) * n < rows && tiles == (rows + 127) / 128;
    }
    return ok;
}

int main()
{
    if (!pair_tiles_ok()) { std::printf("row tiles of pairs\n"); return 1; }
    const bool setting_ok = few_row_setting(nullptr) == 48 && few_row_setting("") == 48 && few_row_setting("0") == 48 && few_row_setting("-3") == 48 &&
                            few_row_setting("1") == 1 && few_row_setting("32") == 32 && few_row_setting("48") == 48 && few_row_setting("49") == 48 &&
                            few_row_setting("64") == 48 && few_row_setting("1000") == 48;
    if (!setting_ok) { printf("few_row_setting\n"); return 1; }
    if (!cross_warps_ok()) { printf("few_cross_warps\n"); return 1; }
    for (int k_blocks = 1; k_blocks <= 128; ++k_blocks)          // d_model 64 .. 8192
        for (int rows = 1; rows <= 2100; ++rows) {
            const VocabShape s = vocab_shape(rows, k_blocks);
            const size_t ring = (size_t)s.stages * (128 * 64 * 2 + 2 * s.n_tile * 64 * 2), epilogue = (size_t)s.n_tile * tc::kRowPitch * 4;
            const bool shape_ok = s.n_tile % 16 == 0 && s.n_tile >= 16 && s.n_tile <= 256 && s.row_tiles * s.n_tile >= rows &&
                                  (s.row_tiles - 1) * s.n_tile < rows && s.stages >= 1 && s.stages <= tc::kMaxStages &&
                                  s.producers >= 1 && s.producers <= tc::kProducerWarps && s.stages % s.producers == 0;
            const bool room = s.smem >= ring + 1024 && s.smem >= epilogue + 1024 && s.smem <= tc::kTcSmemBudget + 1024;
            if (!shape_ok || !room) {
                printf("%d rows, %d k-blocks: n_tile %d, %d stages, %d producers, %zu bytes; ring %zu, epilogue %zu\n", rows, k_blocks, s.n_tile,
                       s.stages, s.producers, s.smem, ring, epilogue);
                return 1;
            }
        }
    printf("ok\n");
    return 0;
}

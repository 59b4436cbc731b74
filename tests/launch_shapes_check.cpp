// Host check of launch_shapes.h (no GPU): whatever the row count and the model width, the dynamic shared memory of the
// vocabulary projection holds both things that live in it one after the other, the ring and the accumulator's rows.
#include <cstdio>

#include "../paper_2503_05931_b200/csrc/launch_shapes.h"

using namespace aed;

int main()
{
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

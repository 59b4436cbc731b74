// Tensor-core GEMM for sm_100a: TMA-fed tcgen05.mma with the accumulator in tensor memory.
//
//   D[128 x N] (fp32, TMEM) = sum over the k-blocks of  A_tile[128 x 64] . B_tile[N x 64]^T
//
// Both operands are K-major bf16 in global memory and arrive in shared memory through
// cp.async.bulk.tensor (no multicast) with the 128-byte swizzle the MMA descriptors name.
// One CTA = one (128-row tile of A, N-row tile of B).  Warp roles: warps 0..7 issue TMA (the k-blocks are
// shared out round robin, a ring stage per warp), warp 8 owns the TMEM allocation and issues the MMAs; at the end all warps but that
// one drain the accumulator (warp w reads TMEM lanes 32*(w%4) .. +31) into the ring's memory, rows first, and then take
// a row each.
//
// Used by the vocabulary projection ("weights as A"): A = output matrix [vocab, K], B = the final LayerNorm output
// [rows, K] as a bf16 high plane and a low (residual) plane accumulated into the same D, so that activations keep ~16
// mantissa bits; the greedy argmax is taken in the epilogue.  The rows-first epilogue is there because an argmax straight
// from the accumulator (a lane per vocabulary entry) needs four warp reductions and four atomics per row and tile, one
// row after the other, and took longer than the product: 16384 entries x 128 rows 38 us, now 20; 512 rows 109, now 57.
//
// Every wait on an mbarrier is bounded: on expiry the CTA raises the error word in the decode state, stops
// issuing work, waits (bounded) for its own TMA copies, frees its TMEM and returns.
#pragma once
#include <cuda.h>

#include "bounded_wait.h"
#include "common.cuh"
#include "launch_shapes.h"

namespace aed {
namespace tc {

constexpr int kThreads = 416;                    // 8 producer warps, 1 MMA warp, 4 more for the epilogue
constexpr long long kWaitCycles = 2000000000ll;   // about a second at B200 clocks
constexpr int kErrTimeout = 2;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

// One lane of a converged warp.  MMAs and commits are issued behind this and not behind `lane == 0`: they take their operands from uniform
// registers, and under a branch that the compiler has to take for divergent each of them cost 70 to 200 cycles (a k-block of four MMAs
// with its wait and commit 530; four MMAs behind this 126).  Copies show no such difference (8 of 16 KB issue in 571 cycles from lane 0
// and in 361 from an elected lane, one from each of 8 warps in 144 and 244); they stand behind this where the warp issues in a loop.
__device__ __forceinline__ bool elect_one()
{
    uint32_t yes;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(yes));
    return yes != 0;
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// The lanes of a warp agree on how a wait ends (see bounded_wait.h).
struct WarpVote {
    __device__ __forceinline__ bool operator()(bool p) const { return __all_sync(0xffffffffu, p) != 0; }
};
// Bounded wait of a whole warp, with one result for all lanes: false if the phase did not complete in time or another role already
// gave up.  (The polling loop is kept out of line: the common case is that the phase has already completed.)
__device__ __noinline__ bool mbar_wait_poll(uint64_t *bar, uint32_t parity, volatile int *abort_flag)
{
    return bounded_poll([&] { return mbar_try_wait(bar, parity); }, [] { return clock64(); }, kWaitCycles, abort_flag, WarpVote());
}
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag)
{
    if (WarpVote()(mbar_try_wait(bar, parity))) return true;
    return mbar_wait_poll(bar, parity, abort_flag);
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int c_inner, int c_outer, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(c_inner), "r"(c_outer), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap *map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// K-major operand tile in shared memory, rows of 128 bytes, 128-byte swizzle, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr)
{
    uint64_t desc = static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
    desc |= static_cast<uint64_t>(1) << 16;            // leading byte offset (unused for swizzled K-major), 16 B
    desc |= static_cast<uint64_t>(1024 >> 4) << 32;    // stride byte offset between 8-row groups
    desc |= static_cast<uint64_t>(1) << 46;            // descriptor version of this architecture
    desc |= static_cast<uint64_t>(2) << 61;            // 128-byte swizzle
    return desc;
}
// bf16 x bf16 -> fp32, both operands K-major, M = 128, N = n
__device__ __forceinline__ uint32_t instr_desc_bf16(int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(kTileM >> 4) << 24);
}
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t desc_a, uint64_t desc_b, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(desc_a), "l"(desc_b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// 16 consecutive fp32 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Twice 16 columns with one wait.
__device__ __forceinline__ void tmem_ld16x2(uint32_t ta, uint32_t tb, float (&a)[16], float (&b)[16])
{
    uint32_t r[16], q[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%33];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(q[0]), "=r"(q[1]), "=r"(q[2]), "=r"(q[3]), "=r"(q[4]), "=r"(q[5]), "=r"(q[6]), "=r"(q[7]), "=r"(q[8]),
          "=r"(q[9]), "=r"(q[10]), "=r"(q[11]), "=r"(q[12]), "=r"(q[13]), "=r"(q[14]), "=r"(q[15])
        : "r"(ta), "r"(tb) : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) { a[i] = __uint_as_float(r[i]); b[i] = __uint_as_float(q[i]); }
}

struct TcParams {
    int a_rows;          // valid rows of A (output features, or frames)
    int n_tile;          // rows of B per CTA = MMA N (multiple of 16, at most 256)
    int k_blocks;
    int rows_fixed;      // >= 0: number of valid B rows; < 0: read it from the decode state
    const __nv_bfloat16 *bias;         // over the columns of D's first dimension (vocabulary / K-V features), may be null
    float *logits_out;                 // [batch, vocab] by utterance or nullptr
    int from_state;                    // logits_out stands in the decode state (steps that are replayed as a graph)
    unsigned long long *keys;          // [rows]
    const int32_t *active_list;
    DecState *state;
};

// grid: x = 128-row tiles of A, z = N-row tiles of B.  Dynamic shared memory: see vocab_shape.
__global__ void __launch_bounds__(kThreads, 1)
tc_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
               const __grid_constant__ CUtensorMap map_b_lo, TcParams p, int stages, int producers)
{
    // `stages` is a multiple of `producers` (1..kProducerWarps): every ring stage is refilled by one warp only, so
    // a producer is never more than one phase ahead of the barrier it waits on (a parity wait cannot tell more).
    extern __shared__ uint8_t smem_dyn[];
    __shared__ __align__(8) uint64_t bar_full[kMaxStages];
    __shared__ __align__(8) uint64_t bar_empty[kMaxStages];
    __shared__ __align__(8) uint64_t bar_done;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;

    AED_TRACE_BEGIN(p.state, 17);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row0 = blockIdx.z * p.n_tile;
    // Only row tiles after the first can be empty; the first one skips this read so that set-up and the first
    // loads do not wait on it (the epilogue reads the row count when it needs it).
    if (blockIdx.z > 0 && row0 >= (p.rows_fixed >= 0 ? p.rows_fixed : p.state->n_active)) return;
    const int a0 = blockIdx.x * kTileM;
    const int n_kb = p.k_blocks;

    uint8_t *tiles = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~static_cast<uintptr_t>(1023));
    const int b_bytes = p.n_tile * kBlockK * 2;
    const int stage_bytes = kATileBytes + 2 * b_bytes;
    // Up to 128 rows the low plane's tile, which stands right behind the high plane's, is multiplied by the same MMAs (N of twice the
    // rows; the two products of a row meet in the epilogue): what an MMA of a few rows costs is its issue.  (us per step of the 4-layer
    // model, 24 / 32 / 64 / 128 rows: 120.9 / 135.7 / 180.3 / 261.0 -> 119.5 / 134.1 / 179.0 / 259.7.  In plane_gemm.cuh, where an MMA has 96 rows
    // and more, the same changed nothing: 200 / 512 rows 1785 / 2873 against 1786 / 2879.)
    const bool stacked = p.n_tile <= 128;
    const int n_cols = stacked ? 2 * p.n_tile : p.n_tile;
    uint32_t tmem_cols = 32;
    while (tmem_cols < static_cast<uint32_t>(n_cols)) tmem_cols <<= 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) { mbar_init(&bar_full[s], 1); mbar_init(&bar_empty[s], 1); }
        mbar_init(&bar_done, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kProducerWarps) tmem_alloc(&tmem_slot, tmem_cols);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = tmem_slot;
    if (threadIdx.x == 0) AED_TRACE_MARK(p.state, 32);      // set-up done
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp < kProducerWarps) {
        if (warp < producers) {
            int issued = 0;
            bool waited = false;
            for (int i = warp; i < n_kb; i += producers) {
                const int s = i % stages;
                if (i >= stages && !mbar_wait(&bar_empty[s], ((i / stages) - 1) & 1, &abort_flag)) break;
                uint8_t *st = tiles + static_cast<size_t>(s) * stage_bytes;
                const int kc = i * kBlockK;
                if (elect_one()) {
                    mbar_expect_tx(&bar_full[s], stage_bytes);
                    tma_load_2d(st, &map_a, kc, a0, &bar_full[s]);
                }
                __syncwarp();
                // A is static (a weight matrix): its first tile is requested while the previous kernel still runs;
                // B is that kernel's output
                if (!waited) { asm volatile("griddepcontrol.wait;" ::: "memory"); waited = true; }
                if (elect_one()) {
                    tma_load_2d(st + kATileBytes, &map_b, kc, row0, &bar_full[s]);
                    tma_load_2d(st + kATileBytes + b_bytes, &map_b_lo, kc, row0, &bar_full[s]);
                }
                __syncwarp();
                issued = i + 1;
            }
            if (abort_flag && issued > 0) {
                // give this warp's last copies a bounded chance to land before the CTA's memory goes away
                const int i = issued - 1;
                const long long start = clock64();
                while (!mbar_try_wait(&bar_full[i % stages], (i / stages) & 1) && clock64() - start < kWaitCycles / 8) {}
            }
        }
    } else if (warp == kProducerWarps) {
        {
            const uint32_t idesc = instr_desc_bf16(n_cols);
            int s = 0;
            uint32_t phase = 0;
            for (int i = 0; i < n_kb; ++i) {
                if (!mbar_wait(&bar_full[s], phase, &abort_flag)) break;
                tc_fence_after_sync();
                const uint32_t sa = smem_u32(tiles + static_cast<size_t>(s) * stage_bytes);
                const uint64_t da = smem_desc_sw128(sa), db = smem_desc_sw128(sa + kATileBytes), dl = smem_desc_sw128(sa + kATileBytes + b_bytes);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < kBlockK / 16; ++k)
                        mma_bf16(tmem_base, da + 2 * k, db + 2 * k, idesc, (i > 0 || k > 0) ? 1u : 0u);
                    if (!stacked) {
#pragma unroll
                        for (int k = 0; k < kBlockK / 16; ++k) mma_bf16(tmem_base, da + 2 * k, dl + 2 * k, idesc, 1u);
                    }
                    mma_commit(&bar_empty[s]);      // the stage may be refilled once these MMAs have read it
                    if (i == n_kb - 1) mma_commit(&bar_done);      // accumulator complete
                }
                __syncwarp();
                if (++s == stages) { s = 0; phase ^= 1; }
            }
        }
    }
    // ---- epilogue: all warps but the one that issues the MMAs (the producers have nothing left to do) -------------
    if (warp != kProducerWarps) {
        constexpr int kPitch = kRowPitch;
        const int ew = warp < kProducerWarps ? warp : warp - 1;      // 0..11
        const int quarter = warp & 3;                                // tensor memory lanes this warp can reach
        const int third = warp < 4 ? 0 : warp < kProducerWarps ? 1 : 2;      // three warps per quarter share the rows in 16s
        float *trans = reinterpret_cast<float *>(tiles);             // T[row][feature] over the ring's memory
        __syncwarp();
        const int n_rows = p.rows_fixed >= 0 ? p.rows_fixed : p.state->n_active;
        float *const logits_out = p.from_state ? p.state->step_logits : p.logits_out;
        const bool ok = mbar_wait(&bar_done, 0, &abort_flag);        // every MMA has completed: the ring is free
        tc_fence_after_sync();
        if (threadIdx.x == (kProducerWarps + 1) * 32) AED_TRACE_MARK(p.state, 34);  // accumulator complete
        const int rows_here = min(p.n_tile, max(n_rows - row0, 0));
        if (ok) {
            const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
            for (int c0 = 16 * third; c0 < rows_here; c0 += 48) {
                float v[16], low[16];
                tmem_ld16x2(taddr + c0, taddr + (stacked ? p.n_tile : 0) + c0, v, low);
#pragma unroll
                for (int j = 0; j < 16; ++j) trans[(c0 + j) * kPitch + quarter * 32 + lane] = stacked ? v[j] + low[j] : v[j];
            }
        }
        asm volatile("bar.sync 1, %0;" ::"n"(kThreads - 32) : "memory");
        if (ok) {
            // a warp per row, 4 consecutive vocabulary entries per lane
            const int o = a0 + lane * 4;
            float bias[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) bias[j] = p.bias && o + j < p.a_rows ? to_f32(p.bias[o + j]) : 0.f;
            const bool vec = o + 3 < p.a_rows && p.a_rows % 4 == 0 && (reinterpret_cast<uintptr_t>(logits_out) & 15) == 0;
#pragma unroll 2
            for (int rl = ew; rl < rows_here; rl += kThreads / 32 - 1) {
                const int r = row0 + rl;
                float4 t = *reinterpret_cast<const float4 *>(trans + rl * kPitch + lane * 4);
                const float z[4] = {t.x + bias[0], t.y + bias[1], t.z + bias[2], t.w + bias[3]};
                if (logits_out) {
                    float *dst = logits_out + static_cast<size_t>(p.active_list[r]) * p.a_rows + o;
                    if (vec) *reinterpret_cast<float4 *>(dst) = make_float4(z[0], z[1], z[2], z[3]);
                    else {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (o + j < p.a_rows) dst[j] = z[j];
                    }
                }
                // the lane's best entry, the warp's best key, then the lowest lane that has it: the lowest index among equals
                int which;
                const uint32_t k32 = best_of(z, p.a_rows - o, which), best = static_cast<uint32_t>(o + which);
                const uint32_t kmax = __reduce_max_sync(0xffffffffu, k32);
                const uint32_t winners = __ballot_sync(0xffffffffu, k32 == kmax);
                if (kmax != 0u && lane == __ffs(winners) - 1)
                    atomicMax(p.keys + r, (static_cast<unsigned long long>(kmax) << 32) | (0xFFFFFFFFu - best));
            }
        }
    }
    if (threadIdx.x == (kProducerWarps + 1) * 32) AED_TRACE_MARK(p.state, 35);      // epilogue issued
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kProducerWarps) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, tmem_cols);
    }
    if (threadIdx.x == 0 && abort_flag) atomicExch(&p.state->error, kErrTimeout);
}

}  // namespace tc
}  // namespace aed

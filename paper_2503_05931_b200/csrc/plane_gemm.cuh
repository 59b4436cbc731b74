// Projections of steps with many rows: both operands ready-made, fetched by TMA, on pairs of blocks (tcgen05 cta_group::2).
//
//   out[r, o] (+)= sum_k (high[r, k] + low[r, k]) * W[o, k]   (+ bias[o])
//
// The activation rows come as two bf16 planes (value = high + low), the weights are the A operand (128 features per block,
// 256 per pair), the rows are N.  What bounds it is what an SM takes in, about 50 bytes a cycle: a block alone with 128
// features x 128 rows takes 48 KB in per k-block of 64 (16 KB of weights, 32 KB of planes).  In a pair each block fetches
// its own features and half of the rows, 32 KB, and the tensor cores read the other half from the peer's shared memory.
//
// Per step of the 24-layer model, with one block per tile before and with pairs: 256 rows 2587 -> 2371 us, 304 rows
// 2870 -> 2601, 512 rows 3772 -> 3495; that includes FFN1's epilogue, which writes the activation planes of FFN2 itself.  An L2
// prefetch of the next projection's weights and more ring stages changed nothing.
//
// Warp roles: 0..7 the copies, a ring stage each (the first weights before the dependency wait), 8 the MMAs (in the pair's
// first block); then all but warp 8 the epilogue: accumulator -> shared memory, rows first -> 16-byte accesses of global
// memory.  Every wait is bounded; on expiry the block raises the sticky error word, lets its
// copies land, frees its tensor memory and returns.
#pragma once
#include "crosskv_gemm.cuh"
#include "step_gemm.cuh"

namespace aed {
namespace pg {

using namespace tc;

constexpr int kPgThreads = 416, kPgMmaWarp = 8, kPgStages = 8;

enum PlaneEpi { PG_ADD = 0, PG_STORE = 1, PG_RELU_PLANES = 2 };

struct PlaneGemmParams {
    int a_rows, k_blocks, n_tile, stages;      // n_tile: rows per pair, a multiple of 32, at most 256
    int epi;
    float *out;                                // PG_ADD: accumulated into (k-splits, residual stream); PG_STORE: written
    int ldo;
    const __nv_bfloat16 *bias;                 // added by k-split 0, may be null
    // PG_RELU_PLANES (one k-split): planes of relu(rstd * (value - mean * c1) + c2)
    const float *c1, *c2;
    const float2 *stats;
    __nv_bfloat16 *out_hi, *out_lo;
    DecState *state;
};

// grid: x = 128-feature tiles (an even number), y = k-splits, z = row tiles.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPgThreads, 1)
plane_gemm_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_hi, const __grid_constant__ CUtensorMap map_lo,
                  const __grid_constant__ PlaneGemmParams p)
{
    extern __shared__ uint8_t smem_dyn[];
    __shared__ __align__(8) uint64_t bar_full[kPgStages], bar_empty[kPgStages], bar_done;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = ckv::cluster_rank();
    const int a0 = blockIdx.x * kTileM, row0 = blockIdx.z * p.n_tile;
    const int kb_begin = static_cast<int>(p.k_blocks * blockIdx.y / gridDim.y);
    const int kb_end = static_cast<int>(p.k_blocks * (blockIdx.y + 1) / gridDim.y);
    const int n_kb = kb_end - kb_begin, S = p.stages;
    uint8_t *tiles = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~static_cast<uintptr_t>(1023));
    const int plane_bytes = p.n_tile / 2 * kBlockK * 2, stage_bytes = kATileBytes + 2 * plane_bytes;
    uint32_t tmem_cols = 32;
    while (tmem_cols < static_cast<uint32_t>(p.n_tile)) tmem_cols <<= 1;

    sg::pdl_launch_dependents();
    if (threadIdx.x == 0) {
        for (int s = 0; s < kPgStages; ++s) { mbar_init(&bar_full[s], 1); mbar_init(&bar_empty[s], 1); }
        mbar_init(&bar_done, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kPgMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before_sync();
    __syncthreads();
    ckv::cluster_meet();                               // the peer's barriers exist before anything reports to them
    tc_fence_after_sync();
    const uint32_t tmem_base = tmem_slot;

    if (warp < kPgMmaWarp) {
        // a ring stage per warp; both blocks' copies report to the first block's barrier
        const int s = warp;
        if (s < S) {
            if (elect_one()) {
                prefetch_tensormap(&map_w);
                prefetch_tensormap(&map_hi);
                prefetch_tensormap(&map_lo);
            }
            __syncwarp();
            const uint32_t full0 = ckv::map_to_rank(&bar_full[s], 0);
            uint8_t *const st = tiles + static_cast<size_t>(s) * stage_bytes;
            const int rows_at = row0 + static_cast<int>(rank) * (p.n_tile / 2);
            bool ok = true;
            uint32_t fills = 0;
            for (int i = s; i < n_kb; i += S, ++fills) {
                if (fills > 0 && !mbar_wait(&bar_empty[s], (fills - 1) & 1, &abort_flag)) { ok = false; break; }
                const int kc = (kb_begin + i) * kBlockK;
                if (elect_one()) {
                    if (rank == 0) mbar_expect_tx(&bar_full[s], 2 * stage_bytes);
                    ckv::tma_load_2d_pair(st, &map_w, kc, a0, full0);
                }
                __syncwarp();
                if (fills == 0) sg::pdl_wait();        // the weights are static
                if (elect_one()) {
                    ckv::tma_load_2d_pair(st + kATileBytes, &map_hi, kc, rows_at, full0);
                    ckv::tma_load_2d_pair(st + kATileBytes + plane_bytes, &map_lo, kc, rows_at, full0);
                }
                __syncwarp();
            }
            // the last MMAs that read this stage must have done so before its memory is used again
            if (ok && fills > 0) ok = mbar_wait(&bar_empty[s], (fills - 1) & 1, &abort_flag);
            if (!ok) {
                // gave up: copies in flight land within microseconds; leave them a millisecond
                const long long start = clock64();
                while (clock64() - start < 2000000ll) {}
            }
        }
        __syncwarp();
    } else if (warp == kPgMmaWarp) {
        if (rank == 0) {
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(p.n_tile >> 3) << 17) |
                                   (static_cast<uint32_t>(2 * kTileM >> 4) << 24);
            bool ok = true;
            int s = 0;
            uint32_t phase = 0;
            for (int i = 0; i < n_kb && ok; ++i) {
                ok = mbar_wait(&bar_full[s], phase, &abort_flag);
                if (!ok) break;
                tc_fence_after_sync();
                const uint32_t sa = smem_u32(tiles + static_cast<size_t>(s) * stage_bytes);
                const uint64_t da = smem_desc_sw128(sa), dh = smem_desc_sw128(sa + kATileBytes), dl = smem_desc_sw128(sa + kATileBytes + plane_bytes);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < kBlockK / 16; ++k) ckv::mma_bf16_pair(tmem_base, da + 2 * k, dh + 2 * k, idesc, (i > 0 || k > 0) ? 1u : 0u);
#pragma unroll
                    for (int k = 0; k < kBlockK / 16; ++k) ckv::mma_bf16_pair(tmem_base, da + 2 * k, dl + 2 * k, idesc, 1u);
                    ckv::mma_commit_pair(&bar_empty[s]);
                    if (i == n_kb - 1) ckv::mma_commit_pair(&bar_done);
                }
                __syncwarp();
                if (++s == S) { s = 0; phase ^= 1; }
            }
        }
    }
    // ---- epilogue ----------------------------------------------------------------------------------------------------
    if (warp != kPgMmaWarp) {
        constexpr int kPitch = kTileM + 4;
        sg::pdl_wait();
        const int n_rows = p.state->n_active, rows_here = min(p.n_tile, max(n_rows - row0, 0));
        const int ew = warp < kPgMmaWarp ? warp : warp - 1;          // 0..11
        const int quarter = warp & 3;                                // tensor memory lanes this warp can reach
        const int third = warp < 4 ? 0 : warp < kPgMmaWarp ? 1 : 2;      // three warps per quarter share the rows in 16s
        float *trans = reinterpret_cast<float *>(tiles);             // T[row][feature] over the ring's memory
        const int o = a0 + lane * 4;
        const bool o_ok = o < p.a_rows;                              // (feature counts are multiples of 64)
        float bias[4] = {0.f, 0.f, 0.f, 0.f};
        float4 c1 = make_float4(0.f, 0.f, 0.f, 0.f), c2 = c1;
        if (o_ok && blockIdx.y == 0 && p.bias) {
#pragma unroll
            for (int j = 0; j < 4; ++j) bias[j] = to_f32(p.bias[o + j]);
        }
        if (o_ok && p.epi == PG_RELU_PLANES) {
            c1 = *reinterpret_cast<const float4 *>(p.c1 + o);
            c2 = *reinterpret_cast<const float4 *>(p.c2 + o);
        }
        const bool ok = mbar_wait(&bar_done, 0, &abort_flag);        // every MMA has completed: the ring is free
        tc_fence_after_sync();
        if (ok) {
            const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
            for (int c0 = 16 * third; c0 < rows_here; c0 += 48) {
                float v[16];
                tmem_ld16(taddr + c0, v);
#pragma unroll
                for (int j = 0; j < 16; ++j) trans[(c0 + j) * kPitch + quarter * 32 + lane] = v[j];
            }
        }
        asm volatile("bar.sync 1, %0;" ::"n"(kPgThreads - 32) : "memory");
        if (ok && o_ok) {
#pragma unroll 4
            for (int rl = ew; rl < rows_here; rl += kPgThreads / 32 - 1) {
                const size_t r = row0 + rl;
                float4 v = *reinterpret_cast<const float4 *>(trans + rl * kPitch + lane * 4);
                if (p.epi == PG_RELU_PLANES) {
                    const float2 st = p.stats[r];
                    const float y[4] = {fmaxf(fmaf(st.y, v.x - st.x * c1.x, c2.x), 0.f), fmaxf(fmaf(st.y, v.y - st.x * c1.y, c2.y), 0.f),
                                        fmaxf(fmaf(st.y, v.z - st.x * c1.z, c2.z), 0.f), fmaxf(fmaf(st.y, v.w - st.x * c1.w, c2.w), 0.f)};
                    uint32_t h[2], l[2];
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const __nv_bfloat162 hi = __floats2bfloat162_rn(y[2 * j], y[2 * j + 1]);
                        h[j] = *reinterpret_cast<const uint32_t *>(&hi);
                        l[j] = sg::pack_bf16(y[2 * j] - __bfloat162float(hi.x), y[2 * j + 1] - __bfloat162float(hi.y));
                    }
                    *reinterpret_cast<uint2 *>(p.out_hi + r * p.ldo + o) = make_uint2(h[0], h[1]);
                    *reinterpret_cast<uint2 *>(p.out_lo + r * p.ldo + o) = make_uint2(l[0], l[1]);
                } else {
                    v.x += bias[0]; v.y += bias[1]; v.z += bias[2]; v.w += bias[3];
                    float *const dst = p.out + r * p.ldo + o;
                    if (p.epi == PG_STORE) *reinterpret_cast<float4 *>(dst) = v;
                    else sg::red_add_v4(dst, v);
                }
            }
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    ckv::cluster_meet();                               // neither block ends while the other may still report to it
    if (warp == kPgMmaWarp) {
        tc_fence_after_sync();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
    }
    if (threadIdx.x == 0 && abort_flag) atomicExch(&p.state->error, kErrTimeout);
}

}  // namespace pg
}  // namespace aed

// Final LayerNorm + vocabulary projection + greedy argmax for steps of at most 16 rows, in one kernel.
//
//   z[r, o] = rstd_r * (sum_k (gamma[k] x[r, k]) Wout[o, k] - mean_r * c1[o]) + c2[o]
//   c1[o] = sum_k gamma[k] Wout[o, k],  c2[o] = sum_k beta[k] Wout[o, k] + b_out[o]      (built at create)
//
// which is LayerNorm(x) Wout^T + b_out with the normalisation folded as in the layer projections (step_gemm.cuh).  With
// few rows the separate normalisation kernel and the tcgen05 projection are two links of the step's dependency chain
// whose work is a few microseconds of weight streaming; here one CTA per 128 vocabulary rows
//   * streams its 128 x d weight tile through a ring of 16 KB stages from the moment it becomes resident (the weights
//     do not depend on the step),
//   * after the dependency wait lets every warp load one row of x into registers, all of it at once, compute its (mean, rstd) and
//     write gamma * x as bf16 high and low planes into shared memory (gain and fold constants, which come from DRAM, are loaded
//     ahead of the wait),
//   * multiplies by warp-level MMAs (m16n8k16; 16 vocabulary rows a warp, the step's rows as one or two N = 8 tiles; two sets of
//     8 warps take the even and the odd k-blocks, because a warp's chain of fragments and MMAs is latency),
//   * and finishes each row: logits for the caller if asked, and one 64-bit atomicMax per row and CTA on the packed
//     (value, lowest index) key that the step's last kernel decodes.
// With 8 warps, rows read twice a few loads at a time and constants loaded where they are used, the time from dependency to end was
// 10 to 12 us (5 to 7 of them the rows); per step of the 4-layer model 1 / 4 / 8 / 16 rows 86 / 94 / 98 / 105 us, now 82 / 90 / 93 / 101.
#pragma once
#include "step_gemv.cuh"

namespace aed {
namespace vg {

using namespace tc;

constexpr int kVgHalf = 8, kVgComputeWarps = 2 * kVgHalf, kVgProducers = 4;      // warps w and w + kVgHalf: the same vocabulary rows, even and odd k-blocks
constexpr int kVgThreads = (kVgComputeWarps + kVgProducers) * 32;
constexpr int kVgStages = 8;                       // multiple of the producers: every stage has one owner
constexpr int kVgRows = 16;

struct VocabGemvParams {
    int vocab, d_model;
    const float *x;                    // [rows, d_model] residual stream after the last layer
    const __nv_bfloat16 *gamma;        // final LayerNorm gain [d_model]
    const float *c1, *c2;              // fold constants [vocab] each
    float eps;
    float *logits_out;                 // [batch, vocab] by utterance, or nullptr
    int from_state;                    // logits_out stands in the decode state (steps that are replayed as a graph)
    unsigned long long *keys;          // [rows]
    const int32_t *active_list;
    DecState *state;
};

__host__ __device__ constexpr int vg_pitch(int d_model) { return d_model * 2 + 16; }       // bytes per row of a plane
__host__ __device__ constexpr int vg_smem(int d_model) { return kVgStages * kATileBytes + 2 * kVgRows * vg_pitch(d_model) + 1024; }

// grid: one CTA per 128 vocabulary rows.  kNT: step rows in eights.
template <int kNT>
__global__ void __launch_bounds__(kVgThreads, 1)
vocab_gemv_kernel(const __grid_constant__ CUtensorMap map_w, VocabGemvParams p)
{
    extern __shared__ uint8_t smem_dyn[];
    __shared__ __align__(8) uint64_t bar_full[kVgStages];
    __shared__ __align__(8) uint64_t bar_empty[kVgStages];
    __shared__ int abort_flag;
    __shared__ float2 s_stats[kVgRows];
    __shared__ __align__(16) float s_t[kVgHalf][8][16 + 4];
    __shared__ unsigned long long s_keys[kVgHalf][kVgRows];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int a0 = blockIdx.x * kTileM;
    const int k_blocks = p.d_model / kBlockK;
    const int pitch = vg_pitch(p.d_model);
    uint8_t *tiles = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~static_cast<uintptr_t>(1023));
    uint8_t *plane_hi = tiles + kVgStages * kATileBytes, *plane_lo = plane_hi + kVgRows * pitch;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kVgStages; ++s) { mbar_init(&bar_full[s], 1); mbar_init(&bar_empty[s], kVgHalf); }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    sg::pdl_launch_dependents();

    if (warp >= kVgComputeWarps) {
        // ---- weight tiles: static data, streamed from the start ---------------------------------------------------
        const int me = warp - kVgComputeWarps;
        int issued = -1;
        for (int i = me; i < k_blocks; i += kVgProducers) {
            const int s = i % kVgStages;
            if (i >= kVgStages && !mbar_wait(&bar_empty[s], ((i / kVgStages) - 1) & 1, &abort_flag)) break;
            if (elect_one()) {
                mbar_expect_tx(&bar_full[s], kATileBytes);
                tma_load_2d(tiles + static_cast<size_t>(s) * kATileBytes, &map_w, i * kBlockK, a0, &bar_full[s]);
            }
            __syncwarp();
            issued = i;
        }
        if (abort_flag && issued >= 0) {
            const long long start = clock64();
            while (!mbar_try_wait(&bar_full[issued % kVgStages], (issued / kVgStages) & 1) && clock64() - start < kWaitCycles / 8) {}
        }
        return;
    }

    // ---- static data of the lanes, before the dependency wait: the gain, the fold constants of the epilogue ---------------
    constexpr int kHeld = 8;                                  // 16-byte pieces of a row per lane that stay in registers (d_model 1024)
    const bool gamma_aligned = aligned16(p.gamma);
    const int per_lane = p.d_model / 128;                     // 16-byte loads per lane and row (d_model is a multiple of 128 here)
    const bool has_row = warp < 8 * kNT;
    float gain[kHeld][4];
    if (has_row) {
#pragma unroll
        for (int i = 0; i < kHeld; ++i)
            if (i < per_lane) load_vec(p.gamma + (lane + 32 * i) * 4, gamma_aligned, gain[i]);
    }
    const int fw = warp & (kVgHalf - 1), f4 = (lane & 3) * 4, o = a0 + fw * 16 + f4;      // the epilogue's 4 vocabulary rows of this lane
    float c1[4], c2[4];
    if (warp < kVgHalf) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            c1[j] = o + j < p.vocab ? p.c1[o + j] : 0.f;
            c2[j] = o + j < p.vocab ? p.c2[o + j] : 0.f;
        }
    }
    // ---- row `warp`: statistics and planes, read once -----------------------------------------------------------------
    const int n_rows = p.state->n_active;
    sg::pdl_wait();
    float *const logits_out = p.from_state ? p.state->step_logits : p.logits_out;
    if (has_row && warp < n_rows) {                           // (rows past the last: planes and statistics that nobody reads the results of)
        const int r = warp;
        const float *xr = p.x + static_cast<size_t>(r) * p.d_model;
        float4 v[kHeld];
        float s = 0.f, q = 0.f;
        auto load = [&](int i) { return *reinterpret_cast<const float4 *>(xr + (lane + 32 * i) * 4); };
#pragma unroll
        for (int i = 0; i < kHeld; ++i) v[i] = i < per_lane ? load(i) : make_float4(0.f, 0.f, 0.f, 0.f);
        auto planes = [&](int i, float4 u, const float (&g)[4]) {
            const int k = (lane + 32 * i) * 4;
            uint32_t h0, l0, h1, l1;
            sv::split2(u.x * g[0], u.y * g[1], h0, l0);
            sv::split2(u.z * g[2], u.w * g[3], h1, l1);
            *reinterpret_cast<uint2 *>(plane_hi + r * pitch + k * 2) = make_uint2(h0, h1);
            *reinterpret_cast<uint2 *>(plane_lo + r * pitch + k * 2) = make_uint2(l0, l1);
        };
#pragma unroll
        for (int i = 0; i < kHeld; ++i)
            if (i < per_lane) { planes(i, v[i], gain[i]); s += (v[i].x + v[i].y) + (v[i].z + v[i].w); }
        for (int i = kHeld; i < per_lane; ++i) {
            const float4 u = load(i);
            float g[4];
            load_vec(p.gamma + (lane + 32 * i) * 4, gamma_aligned, g);
            planes(i, u, g);
            s += (u.x + u.y) + (u.z + u.w);
        }
        const float mean = warp_sum(s) / p.d_model;
        auto spread = [&](float4 u) {
            const float d0 = u.x - mean, d1 = u.y - mean, d2 = u.z - mean, d3 = u.w - mean;
            q += (d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3);
        };
#pragma unroll
        for (int i = 0; i < kHeld; ++i)
            if (i < per_lane) spread(v[i]);
        for (int i = kHeld; i < per_lane; ++i) spread(load(i));
        q = warp_sum(q);
        if (lane == 0) s_stats[r] = make_float2(mean, rsqrtf(q / p.d_model + p.eps));
    }
    asm volatile("bar.sync 2, %0;" ::"n"(kVgComputeWarps * 32) : "memory");           // planes and statistics complete

    // ---- 16 vocabulary rows per warp x 8 kNT step rows, every other k-block -------------------------------------------------
    float acc_h[kNT][4], acc_l[kNT][4];
#pragma unroll
    for (int nt = 0; nt < kNT; ++nt)
#pragma unroll
        for (int j = 0; j < 4; ++j) { acc_h[nt][j] = 0.f; acc_l[nt][j] = 0.f; }
    const uint32_t b_off = static_cast<uint32_t>(((lane & 7) + ((lane >> 4) << 3)) * pitch + ((lane >> 3) & 1) * 16);
    const uint32_t b_one = static_cast<uint32_t>((lane & 7) * pitch + ((lane >> 3) & 1) * 16);
    const uint32_t hi_base = smem_u32(plane_hi), lo_base = smem_u32(plane_lo);
    bool ok = true;
    for (int i = warp / kVgHalf; i < k_blocks; i += 2) {
        const int s = i % kVgStages;
        ok = mbar_wait(&bar_full[s], (i / kVgStages) & 1, &abort_flag);
        if (!ok) break;
        const uint32_t wt = smem_u32(tiles + static_cast<size_t>(s) * kATileBytes);
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
            uint32_t a[4];
            sv::ldmatrix_x4(wt + sv::swz(fw * 16 + (lane & 15), ks * 2 + (lane >> 4)), a);
            const uint32_t kbyte = static_cast<uint32_t>((i * kBlockK + ks * 16) * 2);
            if (kNT == 2) {
                uint32_t bh[4], bl[4];
                sv::ldmatrix_x4(hi_base + b_off + kbyte, bh);
                sv::ldmatrix_x4(lo_base + b_off + kbyte, bl);
                sv::mma_16816(acc_h[0], a, bh[0], bh[1]);
                sv::mma_16816(acc_l[0], a, bl[0], bl[1]);
                sv::mma_16816(acc_h[kNT - 1], a, bh[2], bh[3]);
                sv::mma_16816(acc_l[kNT - 1], a, bl[2], bl[3]);
            } else {                                            // both planes in one ldmatrix
                uint32_t b[4];
                sv::ldmatrix_x4((lane >> 4 ? lo_base : hi_base) + b_one + kbyte, b);
                sv::mma_16816(acc_h[0], a, b[0], b[1]);
                sv::mma_16816(acc_l[0], a, b[2], b[3]);
            }
        }
        __syncwarp();                                           // every lane has read the stage
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&bar_empty[s])) : "memory");
    }
    if (!ok && threadIdx.x % 32 == 0) atomicExch(&p.state->error, kErrTimeout);
    // the odd k-blocks' sums to the warps of the even ones, over the planes' memory
#pragma unroll
    for (int nt = 0; nt < kNT; ++nt)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc_h[nt][j] += acc_l[nt][j];
    asm volatile("bar.sync 2, %0;" ::"n"(kVgComputeWarps * 32) : "memory");
    float4 *const part = reinterpret_cast<float4 *>(plane_hi) + (fw * kNT) * 32 + lane;
    if (warp >= kVgHalf) {
#pragma unroll
        for (int nt = 0; nt < kNT; ++nt) part[nt * 32] = make_float4(acc_h[nt][0], acc_h[nt][1], acc_h[nt][2], acc_h[nt][3]);
    }
    asm volatile("bar.sync 2, %0;" ::"n"(kVgComputeWarps * 32) : "memory");
    if (warp >= kVgHalf) return;
    // ---- per row: fold, logits, argmax key ----------------------------------------------------------------------------
    const int kq = (lane & 3) * 2;
#pragma unroll
    for (int nt = 0; nt < kNT; ++nt) {
        float (*t)[16 + 4] = s_t[warp];
        const float4 odd = part[nt * 32];
        __syncwarp();
        t[kq][lane >> 2] = acc_h[nt][0] + odd.x;
        t[kq + 1][lane >> 2] = acc_h[nt][1] + odd.y;
        t[kq][(lane >> 2) + 8] = acc_h[nt][2] + odd.z;
        t[kq + 1][(lane >> 2) + 8] = acc_h[nt][3] + odd.w;
        __syncwarp();
        const int rr = lane >> 2;                               // row of the tile
        const float4 raw = *reinterpret_cast<const float4 *>(&t[rr][f4]);
        const int r = nt * 8 + rr;
        const float2 st = s_stats[r];
        const float rawv[4] = {raw.x, raw.y, raw.z, raw.w};
        float z[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) z[j] = o + j < p.vocab ? fmaf(st.y, rawv[j] - st.x * c1[j], c2[j]) : 0.f;
        int which;
        const uint32_t k32 = best_of(z, r < n_rows ? p.vocab - o : 0, which);
        unsigned long long key = k32 ? (static_cast<unsigned long long>(k32) << 32) | (0xFFFFFFFFu - static_cast<uint32_t>(o + which)) : 0ull;
        if (r < n_rows && logits_out) {
            float *dst = logits_out + static_cast<size_t>(p.active_list[r]) * p.vocab + o;
            if (o + 3 < p.vocab && (reinterpret_cast<uintptr_t>(dst) & 15) == 0) *reinterpret_cast<float4 *>(dst) = make_float4(z[0], z[1], z[2], z[3]);
            else {
#pragma unroll
                for (int j = 0; j < 4; ++j) if (o + j < p.vocab) dst[j] = z[j];
            }
        }
        // the 4 lanes that share a row, then this warp's entry for the row
        unsigned long long other = __shfl_xor_sync(0xffffffffu, key, 1);
        key = other > key ? other : key;
        other = __shfl_xor_sync(0xffffffffu, key, 2);
        key = other > key ? other : key;
        if ((lane & 3) == 0) s_keys[warp][r] = key;
    }
    asm volatile("bar.sync 3, %0;" ::"n"(kVgHalf * 32) : "memory");
    if (threadIdx.x < 8 * kNT && static_cast<int>(threadIdx.x) < n_rows) {
        unsigned long long key = 0ull;
#pragma unroll
        for (int w = 0; w < kVgHalf; ++w) key = s_keys[w][threadIdx.x] > key ? s_keys[w][threadIdx.x] : key;
        if (key != 0ull) atomicMax(p.keys + threadIdx.x, key);
    }
}

}  // namespace vg
}  // namespace aed

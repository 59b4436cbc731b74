// Decode-step projections for steps of at most 48 rows.
//
//   out[r, o] += sum_k B(r, k) * W[o, k]      (+ bias[o] from the CTA of the first k-split)
//
// Same contract, parameters and side jobs as step_gemm.cuh (B_PLAIN / B_GAMMA / B_LN_RELU, two weight matrices per
// launch), different mechanics.  With a handful of rows a projection launch is a chain of dependent hand-overs, not
// arithmetic: in the tcgen05 form the activation rows go registers -> shared memory -> proxy fence -> barrier -> MMA
// warp -> tensor memory -> registers -> reductions.  Here the rows are the N = 8 columns of warp-level MMAs (m16n8k16, bf16 x
// bf16 -> fp32).  After the dependency wait the 256 compute threads load the rows' k range once (coalesced 16-byte loads), and
// while those loads are on their way each warp waits for the weight tiles (TMA, requested before the wait) and reads its A
// fragments, so that nothing of the weights stands in the chain.  The rows are transformed, written as bf16 high and low
// planes [row][k] into shared memory (row pitch padded against bank conflicts), one named barrier, B fragments by ldmatrix, MMAs,
// and each 16 x 8 result is transposed through shared memory into 16-byte reductions.
//
// What bounds it: up to 8 rows latency (cycles at 4 rows, two k-blocks: rows there 700, planes complete 320, multiplied 340,
// reduced 200).  Beyond, the warp-level MMAs: 1024 MACs a cycle and SM by these marks (with two CTAs per SM and two k-blocks 340, 640,
// 1090 and 1540 cycles for 1, 2, 4 and 6 MMAs of 8 columns per 16 k), so a tile of padding costs as much as one of rows, and the last
// four rows of a launch are one MMA for both planes, not two.  us per step of the 24-layer model, 1 / 2 / 4 / 8 / 12 / 16 / 20 / 24 / 32 /
// 40 / 48 rows: 421 / 427 / 463 / 464 / 492 / 510 / 603 / 622 / 707 / 832 / 853 before, 378 / 388 / 396 / 424 / 481 / 507 / 591 / 608 /
// 679 / 778 / 824 with this form.  Before, barrier, fragments and MMAs of a k-block followed those of the one before, steps of at
// most four rows had every warp load its B fragments from global memory (16 loads per thread, 8 times the sectors: 2100 to 3300 cycles for
// two k-blocks against 940 for one), and row tiles came in whole 8s.
//
// A CTA covers 128 output features x at most 2 k-blocks of 64 (4 in launches of 33 to 48 rows); the host picks the k-splits
// accordingly and falls back to the tcgen05 kernel otherwise.
#pragma once
#include "step_gemm.cuh"

namespace aed {
namespace sv {

using namespace tc;
using sg::StepGemmParams;
using sg::B_PLAIN;
using sg::B_GAMMA;
using sg::B_LN_RELU;

constexpr int kSvThreads = 320;       // warps 0..7: 16 output features each; warps 8..9: weight copies and side jobs
constexpr int kSvMaxKb = 2;

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// byte offset of the 16-byte chunk `chunk` of row `row` in a 128-byte-swizzled tile of 128-byte rows
__device__ __forceinline__ uint32_t swz(int row, int chunk) { return static_cast<uint32_t>(row * 128 + ((chunk ^ (row & 7)) << 4)); }

// two values -> packed bf16 high parts and packed bf16 low parts (value - high)
__device__ __forceinline__ void split2(float a, float b, uint32_t &hi, uint32_t &lo)
{
    hi = sg::pack_bf16(a, b);
    lo = sg::pack_bf16(a - __uint_as_float(hi << 16), b - __uint_as_float(hi & 0xFFFF0000u));
}

// A fragments of M x 16 features from feature f on, from the weight tiles of k-blocks first .. first + N - 1 (those below n_kb), once they have come
template <int N, int M>
__device__ __forceinline__ bool load_weight_fragments(const uint8_t *tiles, uint64_t *bars, int first, int n_kb, int f, int lane, int *abort_flag,
                                                      uint32_t (&a)[N][4][M][4])
{
    bool ok = true;
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (ok && first + i < n_kb) ok = mbar_wait(&bars[first + i], 0, abort_flag);
    if (!ok) return false;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        if (first + i >= n_kb) break;
        const uint32_t wt = smem_u32(tiles + static_cast<size_t>(first + i) * kATileBytes);
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
#pragma unroll
            for (int m = 0; m < M; ++m) ldmatrix_x4(wt + swz(f + m * 16 + (lane & 15), ks * 2 + (lane >> 4)), a[i][ks][m]);
    }
    return true;
}

// kRows: rows of a CTA, a multiple of 4 up to 32; launches of 33 to 48 rows put two halves on grid.z.  Row tiles are 8 rows, one MMA for the
// high and one for the low plane; the eight columns of a last tile of four rows are their high planes and their low planes, one MMA for both.
// (Which of the two a last tile is must be known to the compiler: chosen in the kernel, from the device's row count, the code of both
// is fetched, and 4 / 24 / 32 rows took 406 / 637 / 724 us a step instead of 396 / 608 / 679.)
// kKB: most k-blocks per CTA (2, or 4 for the launches of 33 to 48 rows, which halve the k-splits: the same number of CTAs, half
// the reduction traffic).
// From 20 rows on a warp has 32 features and four of the eight multiply: half the reads of the planes (24 / 32 rows 622 / 709 -> 607 / 678
// us a step; at 16 rows the same eight warps are as fast, 510 against 516).
__host__ __device__ constexpr int sv_pitch(int kb) { return kb * kBlockK * 2 + 16; }          // bytes per row of a plane: the CTA's k range in bf16 + pad
__host__ __device__ constexpr int sv_smem(int rows, int kb = kSvMaxKb) { return kb * kATileBytes + 2 * ((rows + 7) / 8 * 8) * sv_pitch(kb) + 1024; }

// grid: x = 128-feature tiles, y = k-splits, z = row tiles of kRows rows.
template <int MODE, int kRows, int kKB = kSvMaxKb>
__global__ void __launch_bounds__(kSvThreads, 2)
step_gemv_staged_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_w2, StepGemmParams p)
{
    extern __shared__ uint8_t smem_dyn[];
    __shared__ __align__(8) uint64_t bar_a[kKB];
    __shared__ int abort_flag;
    __shared__ __align__(16) float s_g[kKB * kBlockK], s_c1[kKB * kBlockK], s_c2[kKB * kBlockK];
    __shared__ __align__(16) float s_t[8][8][16 + 4];          // per 16 features: 8 rows (+ pad), for the transposition

    static_assert(kRows % 4 == 0 && kRows <= 32, "whole row tiles of 8 and at most one of 4");
    constexpr int kNT = kRows / 8, kTiles = (kRows + 7) / 8;      // whole row tiles, and with that of four rows
    constexpr bool kFour = kRows % 8 != 0;
    constexpr int kM = kRows >= 20 ? 2 : 1, kMmaWarps = 8 / kM;    // 16-feature tiles of a warp; warps that multiply
    constexpr int kSvPitch = sv_pitch(kKB), kF4 = kKB * kBlockK / 4;      // kF4: 16-byte loads per row
    const int row0 = blockIdx.z * kRows;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool second_w = p.tiles_first > 0 && static_cast<int>(blockIdx.x) >= p.tiles_first;
    const CUtensorMap *mw = second_w ? &map_w2 : &map_w;
    const int a0 = (second_w ? static_cast<int>(blockIdx.x) - p.tiles_first : static_cast<int>(blockIdx.x)) * kTileM;
    const int a_rows = second_w ? p.a_rows2 : p.a_rows;
    const int kb_begin = static_cast<int>(p.k_blocks * blockIdx.y / gridDim.y);
    const int kb_end = static_cast<int>(p.k_blocks * (blockIdx.y + 1) / gridDim.y);
    const int n_kb = min(kb_end - kb_begin, kKB);
    uint8_t *tiles = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~static_cast<uintptr_t>(1023));
    uint8_t *plane_hi = tiles + kKB * kATileBytes, *plane_lo = plane_hi + kTiles * 8 * kSvPitch;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kKB; ++s) mbar_init(&bar_a[s], 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (!p.after_rows) sg::pdl_launch_dependents();

    if (warp >= 8) {
        if (warp == 8 && lane == 0) {
            prefetch_tensormap(mw);
            for (int i = 0; i < n_kb; ++i) {
                mbar_expect_tx(&bar_a[i], kATileBytes);
                tma_load_2d(tiles + static_cast<size_t>(i) * kATileBytes, mw, (kb_begin + i) * kBlockK, a0, &bar_a[i]);
            }
        }
        const int cta = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
        const int n_cta = gridDim.x * gridDim.y * gridDim.z;
        sg::side_prefetch(p, cta * 2 + warp - 8, n_cta * 2, lane);
        int n_rows = p.after_rows ? 0 : p.state->n_active;
        sg::pdl_wait();
        if (p.after_rows) { n_rows = p.state->n_active; sg::pdl_launch_dependents(); }
        sg::side_after_wait(p, n_rows, cta + n_cta * (warp - 8), n_cta * 2, lane);
        return;
    }

    const __nv_bfloat16 *const gamma = second_w ? p.gamma2 : p.gamma;
    for (int i = threadIdx.x; i < n_kb * kBlockK; i += 256) {
        const int k = kb_begin * kBlockK + i;
        if (MODE == B_GAMMA) s_g[i] = to_f32(gamma[k]);
        if (MODE == B_LN_RELU) { s_c1[i] = p.c1[k]; s_c2[i] = p.c2[k]; }
    }
    const int f_warp = warp * 16 * kM;                        // this warp's first feature of the tile
    float bias_lo[kM], bias_hi[kM];                           // of features 16 m + lane / 4 and 8 more
#pragma unroll
    for (int m = 0; m < kM; ++m) {
        const int f_lo = a0 + f_warp + m * 16 + (lane >> 2);
        bias_lo[m] = bias_hi[m] = 0.f;
        if (blockIdx.y != 0 || warp >= kMmaWarps) continue;
        if (second_w) {
            if (p.bias2) { if (f_lo < a_rows) bias_lo[m] = p.bias2[f_lo]; if (f_lo + 8 < a_rows) bias_hi[m] = p.bias2[f_lo + 8]; }
        } else if (p.bias) {
            if (f_lo < a_rows) bias_lo[m] = to_f32(p.bias[f_lo]);
            if (f_lo + 8 < a_rows) bias_hi[m] = to_f32(p.bias[f_lo + 8]);
        }
    }
    float *const out = second_w ? p.out2 : p.out;
    const int ldo = second_w ? p.ldo2 : p.ldo;
    asm volatile("bar.sync 2, 256;" ::: "memory");

    int n_rows = p.after_rows ? 0 : p.state->n_active;
    sg::pdl_wait();
    if (p.after_rows) { n_rows = p.state->n_active; sg::pdl_launch_dependents(); }
    // ---- the rows' k range -> planes: element e of the tile is row e / kF4, floats 4 (e % kF4) .. + 3 ------------------
    constexpr int kPer = (kRows * kF4 + 255) / 256;            // 16-byte loads per thread
    float4 xv[kPer];
    float2 st[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int e = threadIdx.x + 256 * j, rl = e / kF4, r = row0 + rl, c4 = e % kF4;
        const bool live = r < n_rows && rl < kRows && c4 * 4 < n_kb * kBlockK;
        xv[j] = live ? *reinterpret_cast<const float4 *>(p.src + static_cast<size_t>(r) * p.ld_src + kb_begin * kBlockK + c4 * 4)
                     : make_float4(0.f, 0.f, 0.f, 0.f);
        st[j] = (MODE == B_LN_RELU && r < n_rows) ? p.stats_in[r] : make_float2(0.f, 0.f);
    }
    // the first two k-blocks' weight fragments while the rows are on their way
    constexpr int kHeld = kRows <= 16 ? 2 : 1;
    uint32_t a[kHeld][4][kM][4];
    bool ok = warp >= kMmaWarps || load_weight_fragments<kHeld, kM>(tiles, bar_a, 0, n_kb, f_warp, lane, &abort_flag, a);
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int e = threadIdx.x + 256 * j, rl = e / kF4, r = row0 + rl, c4 = e % kF4;
        if (kRows * kF4 % 256 != 0 && rl >= kRows) break;
        float y[4] = {xv[j].x, xv[j].y, xv[j].z, xv[j].w};
        if (MODE == B_GAMMA) {
            const float4 g = *reinterpret_cast<const float4 *>(&s_g[c4 * 4]);
            y[0] *= g.x; y[1] *= g.y; y[2] *= g.z; y[3] *= g.w;
        } else if (MODE == B_LN_RELU) {
            const float4 c1 = *reinterpret_cast<const float4 *>(&s_c1[c4 * 4]), c2 = *reinterpret_cast<const float4 *>(&s_c2[c4 * 4]);
            const float cc1[4] = {c1.x, c1.y, c1.z, c1.w}, cc2[4] = {c2.x, c2.y, c2.z, c2.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) y[q] = (r < n_rows) ? fmaxf(fmaf(st[j].y, y[q] - st[j].x * cc1[q], cc2[q]), 0.f) : 0.f;
        }
        uint32_t h0, l0, h1, l1;
        split2(y[0], y[1], h0, l0);
        split2(y[2], y[3], h1, l1);
        *reinterpret_cast<uint2 *>(plane_hi + rl * kSvPitch + c4 * 8) = make_uint2(h0, h1);
        *reinterpret_cast<uint2 *>((kFour && rl >= kNT * 8 ? plane_hi + 4 * kSvPitch : plane_lo) + rl * kSvPitch + c4 * 8) = make_uint2(l0, l1);
    }
    asm volatile("bar.sync 2, 256;" ::: "memory");           // planes complete

    if (warp >= kMmaWarps) return;
    constexpr int kSums = kRows < 16 ? 2 : 1;                   // chains per result: the planes' products apart where there are few
    float acc[kSums][kM][kTiles][4];
#pragma unroll
    for (int m = 0; m < kM; ++m)
#pragma unroll
        for (int nt = 0; nt < kTiles; ++nt)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[0][m][nt][j] = acc[kSums - 1][m][nt][j] = 0.f;
    // ldmatrix addresses of the B fragments: matrices (rows 0-7, k 0-7), (rows 0-7, k 8-15), (rows 8-15, k 0-7), (rows 8-15, k 8-15);
    // of a row tile alone: k 0-7, 8-15 of both planes, or k 0-31 of four rows
    const uint32_t b_off = static_cast<uint32_t>(((lane & 7) + ((lane >> 4) << 3)) * kSvPitch + ((lane >> 3) & 1) * 16);
    const uint32_t b_last = static_cast<uint32_t>((lane & 7) * kSvPitch + ((lane >> 3) & 1) * 16);
    const uint32_t b_long = static_cast<uint32_t>((lane & 7) * kSvPitch + (lane >> 3) * 16);
    const uint32_t hi_base = smem_u32(plane_hi), lo_base = smem_u32(plane_lo);
#pragma unroll
    for (int i = 0; i < kKB; ++i) {
        if (i >= n_kb || !ok) break;
        if (i > 0 && i % kHeld == 0) ok = load_weight_fragments<kHeld, kM>(tiles, bar_a, i, n_kb, f_warp, lane, &abort_flag, a);
        if (!ok) break;
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
            const uint32_t (&af)[kM][4] = a[i % kHeld][ks];
            const uint32_t kbyte = static_cast<uint32_t>((i * kBlockK + ks * 16) * 2);
            if constexpr (kFour) {                              // four rows: both planes are columns of one tile; two steps per ldmatrix
                if (ks % 2 == 0) {
                    uint32_t b[4];
                    ldmatrix_x4(hi_base + kNT * 8 * kSvPitch + b_long + kbyte, b);
#pragma unroll
                    for (int m = 0; m < kM; ++m) {
                        mma_16816(acc[0][m][kNT], af[m], b[0], b[1]);
                        mma_16816(acc[kSums - 1][m][kNT], a[i % kHeld][ks + 1][m], b[2], b[3]);
                    }
                }
            }
#pragma unroll
            for (int np = 0; np + 1 < kNT; np += 2) {            // two row tiles of 8 per ldmatrix
                uint32_t bh[4], bl[4];
                ldmatrix_x4(hi_base + np * 8 * kSvPitch + b_off + kbyte, bh);
                ldmatrix_x4(lo_base + np * 8 * kSvPitch + b_off + kbyte, bl);
#pragma unroll
                for (int m = 0; m < kM; ++m) {
                    mma_16816(acc[0][m][np], af[m], bh[0], bh[1]);
                    mma_16816(acc[0][m][np + 1], af[m], bh[2], bh[3]);
                }
#pragma unroll
                for (int m = 0; m < kM; ++m) {
                    mma_16816(acc[kSums - 1][m][np], af[m], bl[0], bl[1]);
                    mma_16816(acc[kSums - 1][m][np + 1], af[m], bl[2], bl[3]);
                }
            }
            if constexpr (kNT % 2) {                            // an odd row tile: both planes in one ldmatrix
                uint32_t b[4];
                ldmatrix_x4((lane >> 4 ? lo_base : hi_base) + (kNT - 1) * 8 * kSvPitch + b_last + kbyte, b);
#pragma unroll
                for (int m = 0; m < kM; ++m) {
                    mma_16816(acc[0][m][kNT - 1], af[m], b[0], b[1]);
                    mma_16816(acc[kSums - 1][m][kNT - 1], af[m], b[2], b[3]);
                }
            }
        }
    }
    if (!ok) {
        if (lane == 0 && warp == 0) {
            for (int i = 0; i < n_kb; ++i) {
                const long long start = clock64();
                while (!mbar_try_wait(&bar_a[i], 0) && clock64() - start < kWaitCycles / 8) {}
            }
            atomicExch(&p.state->error, kErrTimeout);
        }
        return;
    }
    // ---- 16 features x 8 rows per warp -> [row][feature] in shared memory -> one 16-byte reduction per lane ----------
    // accumulator element j of a thread: feature (lane / 4) + 8 (j / 2), column 2 (lane % 4) + (j % 2)
    const int kq = (lane & 3) * 2;
#pragma unroll
    for (int nt = 0; nt < kTiles; ++nt) {
        __syncwarp();
#pragma unroll
        for (int m = 0; m < kM; ++m) {
            float (*t)[16 + 4] = s_t[warp * kM + m];
            // (in the tile of four rows the columns from 4 on are low planes: the bias once per row)
            const bool again = kFour && nt == kNT && kq >= 4;
            const float lo = again ? 0.f : bias_lo[m], hi = again ? 0.f : bias_hi[m];
            auto sum = [&](int j) { return kSums == 2 ? acc[0][m][nt][j] + acc[kSums - 1][m][nt][j] : acc[0][m][nt][j]; };
            t[kq][lane >> 2] = sum(0) + lo;
            t[kq + 1][lane >> 2] = sum(1) + lo;
            t[kq][(lane >> 2) + 8] = sum(2) + hi;
            t[kq + 1][(lane >> 2) + 8] = sum(3) + hi;
        }
        __syncwarp();
        const int rr = lane >> 2, f4 = (lane & 3) * 4;         // row of the tile, first of 4 consecutive features
#pragma unroll
        for (int m = 0; m < kM; ++m) {
            float (*t)[16 + 4] = s_t[warp * kM + m];
            float4 v = *reinterpret_cast<const float4 *>(&t[rr][f4]);
            if (kFour && nt == kNT) {
                const float4 l = *reinterpret_cast<const float4 *>(&t[(rr & 3) + 4][f4]);
                v.x += l.x; v.y += l.y; v.z += l.z; v.w += l.w;
            }
            const int r = row0 + nt * 8 + rr, o = a0 + f_warp + m * 16 + f4;
            if (r < n_rows && nt * 8 + rr < kRows) {
                float *dst = out + static_cast<size_t>(r) * ldo + o;
                if (o + 3 < a_rows) sg::red_add_v4(dst, v);
                else {
                    if (o + 0 < a_rows) atomicAdd(dst + 0, v.x);
                    if (o + 1 < a_rows) atomicAdd(dst + 1, v.y);
                    if (o + 2 < a_rows) atomicAdd(dst + 2, v.z);
                }
            }
        }
    }
}

}  // namespace sv
}  // namespace aed

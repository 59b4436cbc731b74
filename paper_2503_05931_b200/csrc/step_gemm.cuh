// Decode-step projection on tensor cores with the activation operand built in the kernel, for steps of 49 to 128 rows (fewer
// rows: step_gemv.cuh, more: plane_gemm.cuh).
//
//   out[r, o] += sum_k B(r, k) * W[o, k]      (+ bias[o] from the CTA of the first k-split)
//
// Pairs of CTAs (tcgen05 cta_group::2): a CTA has 128 output features, up to four k-blocks of 64 at a time and makes the activation tiles of
// half of the rows; the tensor cores read the other half from the peer's shared memory.  The weight tiles (bf16, TMA) do not depend on
// earlier kernels and are requested before the programmatic-dependency wait.  The activation tiles are made by 16 warps from
// the fp32 source in the 128-byte-swizzled layout the MMA reads, as a bf16 high plane and a bf16 low plane
// (value - high) behind each other, so that one MMA of twice the rows multiplies both; with one of three transforms fused:
//   B_PLAIN    B = src                                   (attention output -> output projection)
//   B_GAMMA    B = gamma[k] * src                        (LayerNorm folded into the projection, see below)
//   B_LN_RELU  B = relu(rstd_r * (src - mean_r * c1[k]) + c2[k])   (FFN hidden layer from the folded first GEMM)
//
// What bounds it: a chain of hand-overs inside one launch.  Cycles at 64 rows, K = 256 per CTA: tiles of 32 rows (from L2, converted, written)
// 2050, 16 MMAs and their hand-over 1800, reductions 1620 (an SM gives out 28 bytes a cycle).  So the k-blocks are converted side by side
// by groups of warps whose per-k constants wait in registers, and the MMAs are issued in one go.  One CTA per tile, which converted all 64 rows, took
// 3180 + 1900 + 1860 cycles; us per step of the 24-layer model, 49 / 56 / 64 / 72 / 80 / 96 / 112 / 128 rows: 911 / 940 / 970 / 1120 / 1176 /
// 1252 / 1335 / 1420 then, 867 / 888 / 917 / 1082 / 1132 / 1181 / 1268 / 1321 now.  (8 converting warps instead of 16: 873 / 885 / 904 / 1081 /
// 1137 / 1200 / 1333 / 1390.  Registers for two CTAs per SM: 947 / 990 / 1022 and 1174 to 1516, because blocks of the next projection then take the room
// of attention's.  Tried before the pairs: k-splits that meet in a cluster through distributed shared memory, which would leave complete sums
// and planes for the next projection: SM-to-SM reads ran at 10 to 20 bytes a cycle beside the other traffic.)
//
// LayerNorm folding: LN(x) W^T = rstd * ((gamma*x) W^T - mean * c1) + c2 with c1[o] = sum_k gamma_k W[o,k] and
// c2[o] = sum_k beta_k W[o,k] + b[o].  The GEMM therefore runs on gamma*x without knowing the row statistics;
// whoever consumes its output applies (mean, rstd).  The statistics themselves are a side job: a warp of its own
// computes mean and rstd of the rows assigned to its CTA and stores them for the
// consumer.  A second side job clears the fp32 rows a later split-K projection accumulates into.
//
// Two matrices in one launch: feature tiles blockIdx.x >= tiles_first belong to a second weight
// matrix over the same activation rows, with its own tensor map, gamma,
// bias and output buffer.  This is how one launch serves two projections that depend on the same earlier kernel.
//
// Waits are bounded.
#pragma once
#include "crosskv_gemm.cuh"

namespace aed {
namespace sg {

using namespace tc;

constexpr int kMaxKb = 4;             // k-blocks that a CTA holds at most
constexpr int kSgConvertWarps = 16, kSgMmaWarp = 16, kSgConvertThreads = kSgConvertWarps * 32;
constexpr int kSgThreads = 576;       // warps 0..15 activation tiles and epilogue, warp 16 MMAs, warp 17 side jobs
constexpr int kSgMaxRows = 128;       // rows per tile of a pair
constexpr int kSgSmem = 192 * 1024;   // of all tiles at most

enum BMode { B_PLAIN = 0, B_GAMMA = 1, B_LN_RELU = 2 };

struct StepGemmParams {
    int a_rows;                // output features M
    int k_blocks;              // K / 64
    int n_tile;                // rows per pair of CTAs (32..128, multiple of 32)
    int stages;                // k-blocks that a CTA holds at a time, 1..kMaxKb
    int share;                 // 1 << share groups of threads take turns with the k-blocks
    // activation source [rows, ld_src] fp32
    const float *src;
    int ld_src;
    const __nv_bfloat16 *gamma;    // B_GAMMA: [K]
    const float *c1, *c2;          // B_LN_RELU: [K] each
    const float2 *stats_in;        // B_LN_RELU: (mean, rstd) per row
    // epilogue
    float *out;
    int ldo;
    const __nv_bfloat16 *bias;     // added by k-split 0, may be null
    // second matrix (feature tiles tiles_first .. gridDim.x - 1); tiles_first == 0: none
    int tiles_first;
    // the kernel before this launch makes the row table and the row count: read after the dependency wait, and the next
    // kernel, which reads them ahead of its own, may start only then
    int after_rows;
    int a_rows2;
    const __nv_bfloat16 *gamma2;   // B_GAMMA
    float *out2;
    int ldo2;
    const float *bias2;            // fp32, added by k-split 0, may be null
    // side job 1: (mean, rstd) of the rows of stats_src [rows, stats_d]
    const float *stats_src;
    float2 *stats_out;
    int stats_d;
    float eps;
    // side job 2: clear zero_buf [rows, zero_cols]
    float *zero_buf;
    int zero_cols;
    // side job 3: pull a byte range that a later kernel streams (next layer's weights) into L2
    const void *prefetch_ptr, *prefetch2_ptr;      // (the second range: the output matrix, from the last layer)
    size_t prefetch_bytes, prefetch2_bytes;
    DecState *state;
};

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_bf16(float a, float b)
{
    __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&p);
}

// 8 values -> one 16-byte chunk of the high plane and one of the low plane
__device__ __forceinline__ void split_planes(const float (&y)[8], uint4 &hi, uint4 &lo)
{
    uint32_t h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        h[i] = pack_bf16(y[2 * i], y[2 * i + 1]);
        l[i] = pack_bf16(y[2 * i] - __uint_as_float(h[i] << 16), y[2 * i + 1] - __uint_as_float(h[i] & 0xFFFF0000u));
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// 4 floats added to 4 consecutive addresses with one reduction (16-byte aligned)
__device__ __forceinline__ void red_add_v4(float *addr, float4 v)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

__device__ __forceinline__ void red_add(float *addr, float v) { asm volatile("red.global.add.f32 [%0], %1;" ::"l"(addr), "f"(v) : "memory"); }

// ---- side jobs of a projection launch, run by warps of their own in every CTA, off the critical path ----------------------
// (Their loops are not unrolled, nor that of attention's prefetches: a step's kernels together are as large as what an SM holds of
// code, and 30 -> 21 KB for QKV of few rows, 42 -> 35 for the tcgen05 form and 25 -> 21 for attention were worth, at 8 / 16 / 24 / 64 / 128 rows, 424 / 511 /
// 614 / 916 / 1322 -> 418 / 500 / 607 / 881 / 1304 us per step of the 24-layer model.)
// w / n_w: this warp among all that do them in the launch.
// Static data (a later kernel's weights) into L2: no need to wait for the previous kernel.  4 KB pieces.
__device__ __forceinline__ void side_prefetch(const StepGemmParams &p, int w, int n_w, int lane)
{
    for (int range = 0; range < 2; ++range) {
        const char *base = static_cast<const char *>(range ? p.prefetch2_ptr : p.prefetch_ptr);
        if (!base) continue;
        const size_t pieces = (range ? p.prefetch2_bytes : p.prefetch_bytes) / 4096;
        // (a warp issues these one lane after the other: spread over the warps first)
        for (size_t i = static_cast<size_t>(lane) * n_w + w; i < pieces; i += static_cast<size_t>(n_w) * 32)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(base + i * 4096), "r"(4096) : "memory");
    }
}
// After the dependency wait: (mean, rstd) of the rows assigned to this warp, and clear the rows a later split-K projection
// accumulates into.  A launch ends with its last side job, so a row is read once by one warp, with all loads in flight, and kept in
// registers (rows of at most 1024 features; wider ones are read again for the deviations).  (Two warps per row that read it twice, a
// few loads at a time, were what QKV and FFN1 of a few rows ended with: 24 layers, 4 / 16 rows 478 / 533 -> 475 / 526 us a step.)
__device__ __forceinline__ void side_after_wait(const StepGemmParams &p, int n_rows, int w, int n_w, int lane)
{
    if (p.stats_src) {
        constexpr int kHeld = 8;
#pragma unroll 1
        for (int r = w; r < n_rows; r += n_w) {
            const float *const xr = p.stats_src + static_cast<size_t>(r) * p.stats_d + lane * 4;
            const int n = (p.stats_d + 127) / 128;    // (widths are multiples of 64)
            float4 v[kHeld];
            float s = 0.f, q = 0.f;
            auto load = [&](int i) { return i * 128 + lane * 4 < p.stats_d ? *reinterpret_cast<const float4 *>(xr + i * 128) : make_float4(0.f, 0.f, 0.f, 0.f); };
#pragma unroll
            for (int i = 0; i < kHeld; ++i) v[i] = load(i);
#pragma unroll
            for (int i = 0; i < kHeld; ++i) s += (v[i].x + v[i].y) + (v[i].z + v[i].w);
#pragma unroll 1
            for (int i = kHeld; i < n; ++i) { const float4 u = load(i); s += (u.x + u.y) + (u.z + u.w); }
            const float mean = warp_sum(s) / p.stats_d;
            auto spread = [&](int i, float4 u) {
                const float d0 = u.x - mean, d1 = u.y - mean, d2 = u.z - mean, d3 = u.w - mean;
                if (i * 128 + lane * 4 < p.stats_d) q += (d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3);
            };
#pragma unroll
            for (int i = 0; i < kHeld; ++i) spread(i, v[i]);
#pragma unroll 1
            for (int i = kHeld; i < n; ++i) spread(i, load(i));
            q = warp_sum(q);
            if (lane == 0) p.stats_out[r] = make_float2(mean, rsqrtf(q / p.stats_d + p.eps));
        }
    }
    if (p.zero_buf) {
        const size_t total4 = static_cast<size_t>(n_rows) * p.zero_cols / 4;
        float4 *z = reinterpret_cast<float4 *>(p.zero_buf);
#pragma unroll 1
        for (size_t idx = static_cast<size_t>(w) * 32 + lane; idx < total4; idx += static_cast<size_t>(n_w) * 32)
            z[idx] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// One arrival at a barrier of either block of the pair (shared::cluster address).  What it tells of are tiles that tensor cores read: every
// writer has put a proxy fence behind its writes (tiles_written), so the arrival itself, in its default form, need not be a release at
// cluster scope, which would wait for all that its thread has under way (64 / 128 rows 981 / 1392 us a step even with one such arrival per CTA, 917 / 1321 so).
__device__ __forceinline__ void arrive_cluster(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// this thread's generic-proxy writes of operand tiles -> tensor-core reads of either block
__device__ __forceinline__ void tiles_written() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// grid: x = 128-feature tiles (an even number of either matrix), y = k-splits, z = row tiles.  kNI: rows of a k-block per thread at most.
// Dynamic smem (from a 1024-byte boundary): p.stages weight tiles of 16 KB | as many activation tiles of n_tile x 128 bytes: the high
// plane of this block's half of the rows, then their low plane.
template <int MODE, int kNI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kSgThreads, 1)
step_gemm_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_w2, const __grid_constant__ StepGemmParams p)
{
    extern __shared__ uint8_t smem_dyn[];
    __shared__ __align__(8) uint64_t bar_w, bar_act, bar_done;      // (the first two: of the pair's first block)
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;

    AED_TRACE_RESERVE(tcur, p.state, (threadIdx.x == 32 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) ? 10u : 0u);
    AED_TRACE_PUT_NS(p.state, tcur, 40 + MODE);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = ckv::cluster_rank();
    const bool second_w = p.tiles_first > 0 && static_cast<int>(blockIdx.x) >= p.tiles_first;
    const CUtensorMap *const mw = second_w ? &map_w2 : &map_w;
    const int a0 = (second_w ? static_cast<int>(blockIdx.x) - p.tiles_first : static_cast<int>(blockIdx.x)) * kTileM;
    const int a_rows = second_w ? p.a_rows2 : p.a_rows;
    const int row0 = blockIdx.z * p.n_tile, half_tile = p.n_tile / 2;
    const int kb_begin = static_cast<int>(p.k_blocks * blockIdx.y / gridDim.y);
    const int kb_end = static_cast<int>(p.k_blocks * (blockIdx.y + 1) / gridDim.y);
    const int n_kb = kb_end - kb_begin, S = p.stages;
    uint8_t *const tiles = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~static_cast<uintptr_t>(1023));
    const int plane_bytes = half_tile * kBlockK * 2;
    uint8_t *const acts = tiles + S * kATileBytes;
    uint32_t tmem_cols = 32;
    while (tmem_cols < static_cast<uint32_t>(2 * p.n_tile)) tmem_cols <<= 1;

    if (threadIdx.x == kSgMmaWarp * 32) {
        mbar_init(&bar_w, 1);
        mbar_init(&bar_act, 2 * kSgConvertWarps);
        mbar_init(&bar_done, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kSgMmaWarp) {
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before_sync();
    __syncthreads();
    ckv::cluster_meet();                                  // the peer's barriers exist before anything reports to them
    tc_fence_after_sync();
    const uint32_t tmem_base = tmem_slot;
    if (!p.after_rows) pdl_launch_dependents();

    // Rounds of up to S k-blocks (one round unless the launch has few blocks for its K): tiles of both blocks written -> bar_act -> MMAs ->
    // bar_done -> barrier 3.  The MMAs of a round are issued in one go, by the pair's first block: a wait or a commit between them costs more
    // than the four MMAs of a k-block (16 MMAs of 128 x 64 x 16: 1160 cycles, with a wait and a commit per k-block 2290).
    if (warp == kSgMmaWarp) {
        const uint32_t bar_w0 = ckv::map_to_rank(&bar_w, 0);
        auto fetch = [&](int i0) {                        // weights of a round: independent of every earlier kernel
            if (elect_one()) {
                const int n = min(n_kb - i0, S);
                if (rank == 0) mbar_expect_tx(&bar_w, 2 * n * kATileBytes);
                for (int i = 0; i < n; ++i) ckv::tma_load_2d_pair(tiles + i * kATileBytes, mw, (kb_begin + i0 + i) * kBlockK, a0, bar_w0);
            }
            __syncwarp();
        };
        fetch(0);
        // M = 256 features, N = 2 n_tile: high planes and low planes of the first block's rows, then of the second's
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(2 * p.n_tile >> 3) << 17) | (static_cast<uint32_t>(2 * kTileM >> 4) << 24);
        const uint64_t dw0 = smem_desc_sw128(smem_u32(tiles)), da0 = smem_desc_sw128(smem_u32(acts));
        bool ok = true;
        uint32_t phase = 0;
        for (int i0 = 0; i0 < n_kb; i0 += S, phase ^= 1) {
            if (rank == 0) {
                if (ok) ok = mbar_wait(&bar_w, phase, &abort_flag);
                if (ok) ok = ckv::mbar_wait_cluster(&bar_act, phase, &abort_flag);
                if (ok) {
                    tc_fence_after_sync();
                    if (elect_one()) {
                        for (int i = 0; i < min(S, n_kb - i0); ++i) {
                            const uint64_t dw = dw0 + i * (kATileBytes >> 4), da = da0 + static_cast<uint64_t>(i * 2 * plane_bytes >> 4);
#pragma unroll
                            for (int k = 0; k < kBlockK / 16; ++k) ckv::mma_bf16_pair(tmem_base, dw + 2 * k, da + 2 * k, idesc, (i0 + i > 0 || k > 0) ? 1u : 0u);
                        }
                        ckv::mma_commit_pair(&bar_done);
                    }
                    __syncwarp();
                }
            }
            if (ok) ok = mbar_wait(&bar_done, phase, &abort_flag);
            if (ok && i0 + S < n_kb) fetch(i0 + S);
            if (!ok) {
                // gave up: copies in flight land within microseconds; leave them a millisecond
                const long long start = clock64();
                while (clock64() - start < 2000000ll) {}
            }
            // (one warp polls, the others sleep here)
            asm volatile("bar.sync 3, %0;" ::"n"(kSgConvertThreads + 32) : "memory");
        }
    } else if (warp > kSgMmaWarp) {
        // ---- side jobs, off the critical path --------------------------------------------------------------
        const int cta = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
        const int n_cta = gridDim.x * gridDim.y * gridDim.z;
        side_prefetch(p, cta, n_cta, lane);
        pdl_wait();
        side_after_wait(p, p.state->n_active, cta, n_cta, lane);
    } else {
        // A k-block is the work of 512 >> share threads: each has a 16-byte chunk c (8 consecutive k) of rows rbase, rbase + step, ...
        // of either plane.  The groups of threads take a k-block of the round each, and have its per-k constants (static) in registers
        // before the dependency wait.
        const int step = (kSgConvertThreads / 8) >> p.share, c = threadIdx.x & 7, rbase = (threadIdx.x >> 3) & (step - 1), group = threadIdx.x >> (9 - p.share);
        const __nv_bfloat16 *const gamma = second_w ? p.gamma2 : p.gamma;
        const uint32_t bar_act0 = ckv::map_to_rank(&bar_act, 0);
        float ka[8], kb[8];                           // gamma; or c1, c2
        auto constants = [&](int i) {
            const int k = (kb_begin + i) * kBlockK + c * 8;
            if (MODE == B_GAMMA) load_vec(gamma + k, aligned16(gamma), ka);
            if (MODE == B_LN_RELU) { load8(p.c1 + k, ka); load8(p.c2 + k, kb); }
        };
        if (group < n_kb) constants(group);
        const int quarter = warp & 3, a_idx = a0 + quarter * 32 + lane;
        float bias = 0.f;
        if (blockIdx.y == 0 && a_idx < a_rows) {
            if (second_w) bias = p.bias2 ? p.bias2[a_idx] : 0.f;
            else bias = p.bias ? to_f32(p.bias[a_idx]) : 0.f;
        }
        float *const out = second_w ? p.out2 : p.out;
        const int ldo = second_w ? p.ldo2 : p.ldo;
        int n_rows = p.after_rows ? 0 : p.state->n_active;
        AED_TRACE_PUT(p.state, tcur, 50);             // set up, weights requested
        pdl_wait();
        if (p.after_rows) { n_rows = p.state->n_active; pdl_launch_dependents(); }
        AED_TRACE_PUT_NS(p.state, tcur, 51);          // dependency resolved
        // ---- activation tiles: this block's half of the rows ----
        const int rows_here = min(p.n_tile, max(n_rows - row0, 0)), first = (rows_here + 1) / 2;      // first: rows of the pair's first block
        const int my0 = rank ? first : 0, mine = (rank ? rows_here - first : first) - rbase;
        const float *const src = p.src + static_cast<size_t>(row0 + my0 + rbase) * p.ld_src + kb_begin * kBlockK + c * 8;
        constexpr int kHeld = kNI < 4 ? kNI : 4;      // rows in flight
        for (int i0 = 0; i0 < n_kb; i0 += S) {
            for (int s = group; s < min(S, n_kb - i0); s += 1 << p.share) {
                const int i = i0 + s;
                float x[kHeld][8];
                float2 st[kHeld];
                auto load = [&](int j) {
                    if (j * step >= mine) return;
                    load8(src + static_cast<size_t>(j * step) * p.ld_src + i * kBlockK, x[j % kHeld]);
                    if (MODE == B_LN_RELU) st[j % kHeld] = p.stats_in[row0 + my0 + rbase + j * step];
                };
#pragma unroll
                for (int j = 0; j < kHeld; ++j) load(j);
                if (i != group) constants(i);
                uint8_t *const hi_tile = acts + s * 2 * plane_bytes, *const lo_tile = hi_tile + plane_bytes;
#pragma unroll
                for (int j = 0; j < kNI; ++j) {
                    if (j * step >= mine) break;      // (rows past the last: what the tile holds, in columns that nobody reads)
                    float (&y)[8] = x[j % kHeld];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        if (MODE == B_GAMMA) y[e] *= ka[e];
                        if (MODE == B_LN_RELU) y[e] = fmaxf(fmaf(st[j % kHeld].y, y[e] - st[j % kHeld].x * ka[e], kb[e]), 0.f);
                    }
                    uint4 hi, lo;
                    split_planes(y, hi, lo);
                    const int rl = rbase + j * step, off = rl * 128 + ((c ^ (rl & 7)) << 4);
                    *reinterpret_cast<uint4 *>(hi_tile + off) = hi;
                    *reinterpret_cast<uint4 *>(lo_tile + off) = lo;
                    if (j + kHeld < kNI) load(j + kHeld);
                }
            }
            tiles_written();
            __syncwarp();
            if (lane == 0) arrive_cluster(bar_act0);
            if (i0 == 0) AED_TRACE_PUT(p.state, tcur, 52);                 // activation tiles written
            asm volatile("bar.sync 3, %0;" ::"n"(kSgConvertThreads + 32) : "memory");
        }
        // ---- epilogue: reductions straight from the accumulator, 128 consecutive bytes per warp and row ----------------------
        // (An SM gives out about 28 bytes a cycle, as 4-byte reductions of whole warps or as 16-byte ones: 64 rows x 128 features 1220 and
        // 1230 cycles; a pass through shared memory for the latter costs another 800.)
        // Warps w, w + 4, ... reach the same accumulator lanes (lane quarter = warp & 3): they split the rows in 16s.
        const bool ok = *static_cast<volatile int *>(&abort_flag) == 0;
        tc_fence_after_sync();
        AED_TRACE_PUT(p.state, tcur, 53);             // accumulator complete
        if (ok) {
            const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
            for (int c0 = 16 * (warp >> 2); c0 < p.n_tile; c0 += kSgConvertWarps * 4) {
                const bool upper = c0 >= half_tile;      // rows of the pair's second block
                const int at = upper ? c0 - half_tile : c0, live = (upper ? rows_here - first : first) - at;
                if (live <= 0) continue;
                const uint32_t col = taddr + (upper ? p.n_tile : 0) + at;
                float *const dst = out + static_cast<size_t>(row0 + (upper ? first : 0) + at) * ldo + a_idx;
                float hi[16], lo[16];
                tmem_ld16x2(col, col + half_tile, hi, lo);
                if (a_idx < a_rows) {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (j < live) red_add(dst + static_cast<size_t>(j) * ldo, hi[j] + lo[j] + bias);
                }
            }
        }
        AED_TRACE_PUT(p.state, tcur, 54);
    }
    AED_TRACE_PUT_NS(p.state, tcur, 55);              // reductions issued
    tc_fence_before_sync();
    __syncthreads();
    ckv::cluster_meet();                               // neither block ends while the other may still report to it or read its tiles
    if (warp == kSgMmaWarp) {
        tc_fence_after_sync();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
    }
    if (threadIdx.x == 0 && abort_flag) atomicExch(&p.state->error, kErrTimeout);
}

// c1[o] = sum_k gamma[k] W[o,k];  c2[o] = sum_k beta[k] W[o,k] + bias[o]   (one warp per output feature)
__global__ void ln_fold_constants_kernel(const __nv_bfloat16 *__restrict__ w, const __nv_bfloat16 *__restrict__ gamma,
                                         const __nv_bfloat16 *__restrict__ beta, const __nv_bfloat16 *__restrict__ bias,
                                         int m, int k, float *__restrict__ c1, float *__restrict__ c2)
{
    const int o = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (o >= m) return;
    float s1 = 0.f, s2 = 0.f;
    for (int i = lane; i < k; i += 32) {
        const float wv = to_f32(w[static_cast<size_t>(o) * k + i]);
        s1 = fmaf(to_f32(gamma[i]), wv, s1);
        s2 = fmaf(to_f32(beta[i]), wv, s2);
    }
    s1 = warp_sum(s1);
    s2 = warp_sum(s2);
    if (lane == 0) { c1[o] = s1; c2[o] = s2 + (bias ? to_f32(bias[o]) : 0.f); }
}

// Two projections that meet without a nonlinearity between them, composed once at set-up:
//   C[o][i] = sum_k A[o][k] g[k] B[k][i]   (bf16, row-major [n, n]);   cb[o] = sum_k A[o][k] g[k] b[k]
// so that (g * (x + y B^T + b)) A^T = (g * x) A^T + y C^T + cb: the second projection no longer has to wait for the
// sum over all features of the first.  16 x 16 outputs per block, fp32 accumulation.
__global__ void compose_weights_kernel(const __nv_bfloat16 *__restrict__ a, const __nv_bfloat16 *__restrict__ g,
                                       const __nv_bfloat16 *__restrict__ b, int n, __nv_bfloat16 *__restrict__ c)
{
    __shared__ float sa[16][17], sb[16][17];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int o = blockIdx.y * 16 + ty, i = blockIdx.x * 16 + tx;
    float acc = 0.f;
    for (int k0 = 0; k0 < n; k0 += 16) {
        const int ka = k0 + tx, kb = k0 + ty;
        sa[ty][tx] = (o < n && ka < n) ? to_f32(a[static_cast<size_t>(o) * n + ka]) * to_f32(g[ka]) : 0.f;
        sb[ty][tx] = (kb < n && i < n) ? to_f32(b[static_cast<size_t>(kb) * n + i]) : 0.f;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 16; ++k) acc = fmaf(sa[ty][k], sb[k][tx], acc);
        __syncthreads();
    }
    if (o < n && i < n) c[static_cast<size_t>(o) * n + i] = __float2bfloat16_rn(acc);
}

__global__ void compose_bias_kernel(const __nv_bfloat16 *__restrict__ a, const __nv_bfloat16 *__restrict__ g,
                                    const __nv_bfloat16 *__restrict__ b, int n, float *__restrict__ cb)
{
    const int o = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (o >= n) return;
    float s = 0.f;
    if (b)
        for (int k = lane; k < n; k += 32) s = fmaf(to_f32(a[static_cast<size_t>(o) * n + k]) * to_f32(g[k]), to_f32(b[k]), s);
    s = warp_sum(s);
    if (lane == 0) cb[o] = s;
}

}  // namespace sg
}  // namespace aed

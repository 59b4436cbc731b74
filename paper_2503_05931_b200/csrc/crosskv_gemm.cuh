// Cross-attention K/V of every layer in one persistent tensor-core GEMM (sm_100a).
//
//   store[l][k|v][head][frame][64] = bf16( enc[frame, :] . w_kv_c[l][feature, :] + b_kv_c[l][feature] )
// (or rounded to the 8-bit format E4M3 instead of bf16 when the handle stores the cross-attention K/V in 8 bits)
//
// over the packed encoder frames (no padding rows).  Pairs of blocks, one block per SM, walk a list of output tiles
// (2 x 128 frames x 256 features, K = d_enc in 64-wide k-blocks).  Tile order: groups of as many frame tile pairs as
// there are block pairs outermost; inside a group the tiles are numbered (layer, feature tile) major, frame tile pair
// minor, and pair b takes the numbers b, b + pairs, ...  With a full group a pair therefore keeps its frames for every
// layer and feature tile: the frame tiles of a group stay in L2 while all layers' weights stream past them, and the
// weights are re-read once per group only.  With fewer frame tiles than pairs the same numbering spreads the
// (layer, feature tile) pairs over the idle ones.
//
// Why pairs: a block alone on 128 frames x 256 features takes 48 KB per k-block into its shared memory for 512 cycles
// of tensor core, and an SM takes in about 50 bytes a cycle, so the tensor cores sat at 0.54 of what cuBLAS measures.
// With tcgen05 cta_group::2 each block of the pair fetches its own 128 frames and half of the features (32 KB per
// k-block for the same 512 cycles); the tensor cores read the other half from the peer's shared memory.
//
// 75k frames, 4 layers (d 1024): 1371 us before, 956 us in pairs, 900 us since an elected lane issues (1.40 PFLOP/s, 0.86 of the
// measured cuBLAS rate); with four epilogue warps instead of eight (at 956) 1078 us: draining 256 columns then takes longer than
// accumulating them.
//
// Warp roles (16 warps): 0..5 producers, 6 issues the MMAs (in the pair's first block only), 7 idle, 8..15 epilogue.
//   * Six producer warps share the k-blocks round robin, each loading
//     both operands of its k-blocks into a ring stage of its own.  The copies of
//     both blocks report to the first block's barrier.
//   * The accumulator (128 lanes x 256 fp32 columns in either block) is double-buffered in tensor memory: while the
//     epilogue warps drain tile i (bias, bf16 pack, 32-byte stores straight into the per-head K/V rows), the MMA warp
//     already accumulates tile i + 1.
// Every wait is bounded; on expiry the block raises the sticky error word, lets its copies land, frees its tensor
// memory and returns.
#pragma once
#include "tc_gemm.cuh"

namespace aed {
namespace ckv {

using namespace tc;

constexpr int kTileN = 256;                       // features per tile = MMA N
constexpr int kStageBytes = 2 * kATileBytes;      // per block: 16 KB frames + 16 KB weights
constexpr int kStages = 6;
constexpr int kProducers = 6;                     // one stage each
constexpr int kMmaWarp = 6;
constexpr int kCkvThreads = 512;

// The frames of a launch: up to kMaxSegs runs of consecutive rows of the encoder tensor, each with a store row of its
// own (a packed batch is one run; utterances admitted into slots are one run each).  Frame tiles never straddle runs.
constexpr int kMaxSegs = 16;
struct CkvSegs {
    int n;
    int tile0[kMaxSegs + 1];          // first frame tile of every run, and the total
    int src0[kMaxSegs];               // row of the run's first frame in the encoder tensor
    int frames[kMaxSegs];
    int dst0[kMaxSegs];               // store row of the run's first frame
};

struct CkvParams {
    CkvSegs segs;
    int frame_capacity;
    int d_model, n_heads, d_enc;
    int n_layers;
    void *store;                      // layer 0; layers are layer_elems elements apart; bf16, or E4M3 bytes (template argument)
    size_t layer_elems;
    const __nv_bfloat16 *const *bias; // [n_layers] device pointers (entries may be null), or null
    DecState *state;
};

// ---- the pair -----------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// the address of a shared-memory object in block `rank` of this cluster
__device__ __forceinline__ uint32_t map_to_rank(const void *p, uint32_t rank)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    return a;
}
// Where the blocks of a pair meet: before the first report to a barrier of the peer's (behind fence.mbarrier_init, which makes the
// barriers visible) and before either ends.  Nothing else written before it is read behind it, so the arrival is relaxed: with release
// each thread waits there until the reductions and stores it has under way have been performed, at the end of every launch (24 layers, 160 /
// 200 / 256 / 512 rows 1611 / 1796 / 2021 / 2885 -> 1536 / 1722 / 1930 / 2821 us per step).
__device__ __forceinline__ void cluster_meet()
{
    asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
// copy into this block's shared memory; the bytes are reported to a barrier of either block (shared::cluster address)
__device__ __forceinline__ void tma_load_2d_pair(void *dst, const CUtensorMap *map, int c_inner, int c_outer, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(c_inner), "r"(c_outer), "r"(bar) : "memory");
}
// M = 256 (128 rows from either block), N = 256 (128 from either block); accumulator rows stay with their block
__device__ __forceinline__ void mma_bf16_pair(uint32_t tmem_d, uint64_t desc_a, uint64_t desc_b, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(desc_a), "l"(desc_b), "r"(idesc), "r"(accumulate) : "memory");
}
// arrives on the barrier at this offset in both blocks once the MMAs issued so far have completed
__device__ __forceinline__ void mma_commit_pair(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(smem_u32(bar)), "h"(static_cast<uint16_t>(3)) : "memory");
}
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t *bar, uint32_t parity, volatile int *abort_flag)
{
    return bounded_poll(
        [&] {
            uint32_t ok;
            asm volatile("{\n\t.reg .pred p;\n\t"
                         "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                         "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
            return ok != 0;
        },
        [] { return clock64(); }, kWaitCycles, abort_flag, WarpVote());
}

// The tiles of one block pair, in order (m_tiles: frame tile pairs; G, b: block pairs of the grid and this one).  Every warp role walks the same sequence.
struct TileWalk {
    int m_tiles, per_group, G, b;
    int group, gsize;
    long long id, total;
    __device__ TileWalk(int m_tiles_, int per_group_, int G_, int b_) : m_tiles(m_tiles_), per_group(per_group_), G(G_), b(b_)
    {
        group = 0;
        gsize = min(G, m_tiles);
        total = static_cast<long long>(per_group) * gsize;
        id = b;
        settle();
    }
    __device__ void settle()
    {
        while (gsize > 0 && id >= total) {          // next group
            ++group;
            gsize = min(G, m_tiles - group * G);
            if (gsize <= 0) { gsize = 0; break; }
            total = static_cast<long long>(per_group) * gsize;
            id = b;
        }
    }
    __device__ bool valid() const { return gsize > 0; }
    __device__ int lnt() const { return static_cast<int>(id / gsize); }                       // layer * n_tiles + feature tile
    __device__ int m_tile() const { return group * G + static_cast<int>(id % gsize); }
    __device__ void next() { id += G; settle(); }
};

// grid: persistent pairs of blocks.  map_w: one tensor map per layer over w_kv_c [2d, d_enc], boxes of 128 rows x 64.
template <bool kE4M3>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kCkvThreads, 1)
crosskv_gemm_kernel(const __grid_constant__ CUtensorMap map_enc, const CUtensorMap *__restrict__ map_w, const __grid_constant__ CkvParams p)
{
    extern __shared__ uint8_t smem_dyn[];
    __shared__ __align__(8) uint64_t bar_full[kStages];
    __shared__ __align__(8) uint64_t bar_empty[kStages];
    __shared__ __align__(8) uint64_t bar_acc_full[2];     // accumulator buffer complete (MMA -> epilogue)
    __shared__ __align__(8) uint64_t bar_acc_free[2];     // accumulator buffer drained (epilogue -> MMA)
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    uint8_t *tiles = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~static_cast<uintptr_t>(1023));
    const int k_blocks = p.d_enc / kBlockK;
    const int m_tiles = p.segs.tile0[p.segs.n], m_pairs = (m_tiles + 1) / 2;
    const int pairs = gridDim.x / 2, pair = blockIdx.x / 2;
    // run and tile inside the run of a frame tile
    auto locate = [&](int m_tile, int &seg, int &j) {
        seg = 0;
        while (seg + 1 < p.segs.n && m_tile >= p.segs.tile0[seg + 1]) ++seg;
        j = m_tile - p.segs.tile0[seg];
    };
    const int n_tiles = (2 * p.d_model + kTileN - 1) / kTileN;
    const int per_group = p.n_layers * n_tiles;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) { mbar_init(&bar_full[s], 1); mbar_init(&bar_empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&bar_acc_full[b], 1); mbar_init(&bar_acc_free[b], 16); }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before_sync();
    __syncthreads();
    cluster_meet();                                    // the peer's barriers exist before anything reports to them
    tc_fence_after_sync();
    const uint32_t tmem_base = tmem_slot;

    if (warp < kProducers) {
        {
            if (elect_one()) prefetch_tensormap(&map_enc);
            __syncwarp();
            const uint32_t full0 = map_to_rank(&bar_full[warp], 0);      // kStages == kProducers: this warp's stage
            uint8_t *const st = tiles + static_cast<size_t>(warp) * kStageBytes;
            long long it = 0;                           // k-block counter over all of this pair's tiles
            uint32_t fills = 0;                         // of this warp's stage
            bool ok = true;
            for (TileWalk w(m_pairs, per_group, pairs, pair); w.valid() && ok; w.next()) {
                const int layer = w.lnt() / n_tiles, nt = w.lnt() % n_tiles;
                int seg, j;
                locate(min(2 * w.m_tile() + static_cast<int>(rank), m_tiles - 1), seg, j);
                const int m0 = p.segs.src0[seg] + j * kTileM;          // rows past the run's end are loaded and never stored
                for (int kb = 0; kb < k_blocks; ++kb, ++it) {
                    if (static_cast<int>(it % kProducers) != warp) continue;
                    if (fills > 0 && !mbar_wait(&bar_empty[warp], (fills - 1) & 1, &abort_flag)) { ok = false; break; }
                    if (elect_one()) {
                        if (rank == 0) mbar_expect_tx(&bar_full[warp], 2 * kStageBytes);      // its own copies and the peer's
                        tma_load_2d_pair(st, &map_enc, kb * kBlockK, m0, full0);
                        tma_load_2d_pair(st + kATileBytes, map_w + layer, kb * kBlockK, nt * kTileN + static_cast<int>(rank) * (kTileN / 2), full0);
                    }
                    __syncwarp();
                    ++fills;
                }
            }
            // the last MMAs that read this stage report here: they must have done so before the block may end
            if (ok && fills > 0) ok = mbar_wait(&bar_empty[warp], (fills - 1) & 1, &abort_flag);
            if (!ok) {
                // gave up: copies in flight land within microseconds; leave them a millisecond
                const long long start = clock64();
                while (clock64() - start < 2000000ll) {}
            }
        }
    } else if (warp == kMmaWarp) {
        if (rank == 0) {
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(kTileN >> 3) << 17) |
                                   (static_cast<uint32_t>(2 * kTileM >> 4) << 24);
            int s = 0;
            uint32_t phase = 0;
            bool ok = true;
            long long t = 0;
            for (TileWalk w(m_pairs, per_group, pairs, pair); w.valid() && ok; w.next(), ++t) {
                const int buf = static_cast<int>(t & 1);
                // both blocks' epilogues must have drained this buffer (its previous use was tile t - 2)
                if (t >= 2) ok = mbar_wait_cluster(&bar_acc_free[buf], static_cast<uint32_t>((t >> 1) - 1) & 1, &abort_flag);
                if (!ok) break;
                tc_fence_after_sync();
                const uint32_t acc = tmem_base + static_cast<uint32_t>(buf * kTileN);
                for (int kb = 0; kb < k_blocks && ok; ++kb) {
                    ok = mbar_wait(&bar_full[s], phase, &abort_flag);
                    if (!ok) break;
                    tc_fence_after_sync();
                    const uint32_t sa = smem_u32(tiles + static_cast<size_t>(s) * kStageBytes);
                    const uint64_t da = smem_desc_sw128(sa), db = smem_desc_sw128(sa + kATileBytes);
                    if (elect_one()) {
#pragma unroll
                        for (int k = 0; k < kBlockK / 16; ++k) mma_bf16_pair(acc, da + 2 * k, db + 2 * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
                        mma_commit_pair(&bar_empty[s]);
                        if (kb == k_blocks - 1) mma_commit_pair(&bar_acc_full[buf]);
                    }
                    __syncwarp();
                    if (++s == kStages) { s = 0; phase ^= 1; }
                }
            }
        }
    } else if (warp >= 8) {
        // epilogue: warp w reads TMEM lanes 32 * (w & 3) .. + 31; this thread owns one frame of the block's tile
        const int quarter = warp & 3, half = (warp >> 2) & 1;
        const uint32_t acc_free0[2] = {map_to_rank(&bar_acc_free[0], 0), map_to_rank(&bar_acc_free[1], 0)};
        bool ok = true;
        long long t = 0;
        for (TileWalk w(m_pairs, per_group, pairs, pair); w.valid() && ok; w.next(), ++t) {
            const int layer = w.lnt() / n_tiles, nt = w.lnt() % n_tiles;
            const int m_tile = 2 * w.m_tile() + static_cast<int>(rank);
            int seg, j;
            locate(min(m_tile, m_tiles - 1), seg, j);
            const int frame_in_run = j * kTileM + quarter * 32 + lane;
            const bool frame_ok = m_tile < m_tiles && frame_in_run < p.segs.frames[seg];      // (an odd last tile has no partner)
            const int frame = p.segs.dst0[seg] + frame_in_run;
            const int buf = static_cast<int>(t & 1);
            ok = mbar_wait(&bar_acc_full[buf], static_cast<uint32_t>(t >> 1) & 1, &abort_flag);
            if (!ok) break;
            tc_fence_after_sync();
            const uint32_t taddr = tmem_base + static_cast<uint32_t>(buf * kTileN) + (static_cast<uint32_t>(quarter * 32) << 16);
            const size_t layer_off = static_cast<size_t>(layer) * p.layer_elems;
            const __nv_bfloat16 *bias = p.bias ? p.bias[layer] : nullptr;
            const bool bias_vec = (reinterpret_cast<uintptr_t>(bias) & 15) == 0;
            // two warps per lane quarter, 128 features each, one head (64 features) at a time
            int o = nt * kTileN + half * (kTileN / 2);
            int kv = o / p.d_model, h = (o - kv * p.d_model) / kHeadDim;
            for (int c0 = half * (kTileN / 2); c0 < (half + 1) * (kTileN / 2); c0 += kHeadDim, o += kHeadDim) {
                if (o >= 2 * p.d_model) break;                   // (uniform over the warp)
                const size_t elem = layer_off + ((static_cast<size_t>(kv) * p.n_heads + h) * p.frame_capacity + frame) * kHeadDim;
                if (++h == p.n_heads) { h = 0; ++kv; }
#pragma unroll
                for (int e = 0; e < kHeadDim; e += 16) {
                    float v[16];
                    tmem_ld16(taddr + c0 + e, v);
                    if (bias) {
                        if (bias_vec) {
#pragma unroll
                            for (int q = 0; q < 16; q += 8) {
                                float bv[8];
                                load8(bias + o + e + q, bv);
#pragma unroll
                                for (int i = 0; i < 8; ++i) v[q + i] += bv[i];
                            }
                        } else {
#pragma unroll
                            for (int i = 0; i < 16; ++i) v[i] += to_f32(bias[o + e + i]);
                        }
                    }
                    if (!frame_ok) continue;
                    uint32_t packed[8];
                    if (kE4M3) {
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            packed[i] = static_cast<uint32_t>(pack_e4m3x2(v[4 * i], v[4 * i + 1])) |
                                        (static_cast<uint32_t>(pack_e4m3x2(v[4 * i + 2], v[4 * i + 3])) << 16);
                        *reinterpret_cast<uint4 *>(static_cast<uint8_t *>(p.store) + elem + e) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
                    } else {
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            __nv_bfloat162 two = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
                            packed[i] = *reinterpret_cast<uint32_t *>(&two);
                        }
                        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                                     ::"l"(static_cast<__nv_bfloat16 *>(p.store) + elem + e), "r"(packed[0]), "r"(packed[1]), "r"(packed[2]),
                                     "r"(packed[3]), "r"(packed[4]), "r"(packed[5]), "r"(packed[6]), "r"(packed[7]) : "memory");
                    }
                }
            }
            // this warp is done with the buffer
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(acc_free0[buf]) : "memory");
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    cluster_meet();                                    // neither block ends while the other may still report to it
    if (warp == kMmaWarp) {
        tc_fence_after_sync();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
    }
    if (threadIdx.x == 0 && abort_flag) atomicExch(&p.state->error, kErrTimeout);
}

}  // namespace ckv
}  // namespace aed

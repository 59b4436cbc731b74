// fp32 steps of small models: a whole decoder step in one launch, by clusters that each take four rows through all layers.
//
// With eight launches per layer a step of a small fp32 model is launches in a row: about 2.8 us each, of which the
// arithmetic is a few hundred cycles.  Rows do not depend on one another, so a cluster of 16 blocks (of 8 where the step has more rows than
// clusters of 16 find room for) takes four of them from the embedding to the greedy choice by itself.  Its blocks share the output
// features of every projection and the (row, head) pairs of attention, and what a block computes it stores into the shared memory of those that need it
// (st.async, whose bytes the receiver's barrier counts): that costs 1000 to 1500 cycles a stage where a launch costs 2500 beside its work.
// Each cluster reads all weights of the step from L2.
//
// Stages of a layer:
//   0  LN1, [q | k | v] of a pair to the pair's block          1  self-attention, output to all
//   2  output projection + residual, rows to all               3  LN2, q of a pair to the pair's block
//   4  cross-attention, output to all                          5  output projection + residual, rows to all
//   6  LN3, hidden features to all                             7  FFN2 + residual, rows to all
// There is one buffer for each kind of data and four barriers that take turns.  Stages 2, 5 and 7 need something of every block, so no block is
// more than three stages ahead of another; and every sender of a stage has received, from the block that it overwrites something of, what that
// block sent after it last read it (stage 1 before 2 overwrites the rows that LN1 read, and so on).  A block that has no features in a
// projection (64-wide models) may see rows change while it normalises them: nobody uses what it normalises then.
//
// A warp owns eight output features of a wide projection (QKV, FFN1, vocabulary) or two of a narrow one, lanes along K, sums as in rows_kernel
// (f32_rows.cuh) but for packed multiply-adds.  Weights (64 registers a lane) and the keys and values of the first positions are requested before a
// stage's data are waited for.  The sums of the even and the odd k apart: logits against the fp64 checker, relative 2-norm, 20
// batches each with weights N(0, 0.02) and with attention projections four and eight times as large: 1.42e-7, 1.79e-7, 6.70e-7 with launches, 1.39e-7, 1.76e-7,
// 6.45e-7 here.
//
// us per step of the 2-layer model (d 256, 40 frames), 1 / 4 / 8 / 16 / 28 / 32 / 48 / 56 rows: 47.6 / 52.2 / 69.5 / 75.0 / 79.6 / 82.5 / 87.0 / 93.6 with
// launches, 38.0 / 40.0 / 40.6 / 39.0 / 39.2 / 51.1 / 51.7 / 51.7 here.  What bounds it: about 12,000 instructions in a row per warp and step, 75 KB of
// them, with two warps per scheduler.  On the way: cluster barriers and plain remote stores instead of counted ones 50 us (4 rows), 16 warps of half as many
// features 49 (twice the reads of the rows from shared memory), everything written out per stage 57, eight rows per cluster 65 (32 rows).
#pragma once
#include <type_traits>
#include "crosskv_gemm.cuh"
#include "f32_rows.cuh"

namespace aed {
namespace f32 {

constexpr int kClusterThreads = 256, kClusterWarps = kClusterThreads / 32;
constexpr int kClusterRows = 4, kClusterSizes[2] = {16, 8};
constexpr int kHeld = 16;                    // weight loads per lane requested ahead

struct ClusterLayer {
    const float *ln1_g, *ln1_b, *w_qkv, *b_qkv, *w_o, *b_o, *ln2_g, *ln2_b, *w_q_c, *b_q_c, *w_o_c, *b_o_c, *ln3_g, *ln3_b, *w_ff1, *b_ff1, *w_ff2, *b_ff2;
};

struct ClusterArgs {
    DecState *state;
    const ClusterLayer *layers;
    int n_layers, cluster_log, d, n_heads, d_ffn, vocab, max_dec_len, frame_capacity;
    float eps, scale;                        // scale: of the embedding
    const int4 *row_info;
    const int32_t *tokens;                   // by utterance
    const float *embed, *pe;
    const float *x;                          // the embedded rows, if the kernel before has made them; or null
    float *self_cache;
    const float *cross;
    size_t self_layer_elems, cross_layer_elems;
    const float *final_ln_g, *final_ln_b, *w_out, *b_out;
    float *logits_out;                       // [batch, vocab] by utterance or null
    unsigned long long *keys;                // packed argmax keys [rows]
};

// (row, head) pairs of a block
__host__ __device__ constexpr int cluster_slots(int rows, int n_heads, int cluster) { return (rows * n_heads + cluster - 1) / cluster; }
// Bytes of dynamic shared memory.
__host__ __device__ constexpr size_t cluster_smem(int d, int d_ffn, int n_heads, int cluster, int n_layers)
{
    return (static_cast<size_t>(kClusterRows) * (3 * d + d_ffn) + cluster_slots(kClusterRows, n_heads, cluster) * 3 * kHeadDim + 2 * kClusterWarps * kHeadDim + 2 * d) * 4 +
           n_layers * sizeof(ClusterLayer);
}
// What it is for: models whose K fits the weights that a lane holds, 256 for the wide projections and 1024 for the narrow ones.  (Every cluster reads
// all weights, 16 SMs of 60 bytes a cycle: a layer twice as wide would take longer than its launches.)
__host__ __device__ constexpr bool cluster_supports(int d, int d_ffn, int n_layers) { return d <= kHeld / 8 * 128 && d_ffn <= kHeld / 2 * 128 && n_layers <= 64; }

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// Stores into the shared memory of a block of the cluster that report their bytes to a barrier of that block.
__device__ __forceinline__ void send(uint32_t addr, float v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(addr), "f"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void send(uint32_t addr, float2 v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(addr), "f"(v.x), "f"(v.y), "r"(bar) : "memory");
}
__device__ __forceinline__ void send(uint32_t addr, float4 v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar) : "memory");
}

// Four floats as two pairs, for packed multiply-adds.
struct Quad { unsigned long long a, b; };
__device__ __forceinline__ void fma2(unsigned long long &acc, unsigned long long x, unsigned long long w) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(x), "l"(w)); }
__device__ __forceinline__ float pair_sum(unsigned long long v) { return __uint_as_float(static_cast<uint32_t>(v)) + __uint_as_float(static_cast<uint32_t>(v >> 32)); }
// A load that stays where it is written.  (__ldg may be moved to where its value is used, behind a wait.)
__device__ __forceinline__ Quad load_weights(const float *at, bool yes)
{
    Quad v;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\tmov.b64 %0, 0;\n\tmov.b64 %1, 0;\n\t@p ld.global.nc.v2.b64 {%0, %1}, [%2];\n\t}"
                 : "=&l"(v.a), "=&l"(v.b) : "l"(at), "r"(static_cast<int>(yes)) : "memory");
    return v;
}
__device__ __forceinline__ float load_weight(const float *at, bool yes)
{
    float v;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\tmov.b32 %0, 0f00000000;\n\t@p ld.global.nc.f32 %0, [%1];\n\t}"
                 : "=&f"(v) : "l"(at), "r"(static_cast<int>(yes)) : "memory");
    return v;
}

// grid: 16 or 8 blocks (1 << p.cluster_log) per R rows.
__global__ void __launch_bounds__(kClusterThreads, 1)
cluster_step_kernel(const __grid_constant__ ClusterArgs p)
{
    constexpr int R = kClusterRows;
    extern __shared__ __align__(16) float sm[];
    __shared__ int4 s_row[R];
    __shared__ float s_max[kClusterWarps], s_sum[kClusterWarps];
    __shared__ unsigned long long s_key[R];
    __shared__ __align__(8) uint64_t bars[4];
    __shared__ int abort_flag;
    const int d = p.d, F = p.d_ffn, H = p.n_heads, CL = p.cluster_log, C = 1 << CL, slots = cluster_slots(R, H, C);
    float *const xs = sm, *const ns = xs + R * d, *const as = ns + R * d, *const hs = as + R * d;         // residual, normalised, attention rows [R][d]; hidden [R][F]
    float *const qs = hs + R * F, *const red = qs + slots * 3 * kHeadDim, *const outs = red + kClusterWarps * kHeadDim, *const lnp = outs + kClusterWarps * kHeadDim;
    ClusterLayer *const layers = reinterpret_cast<ClusterLayer *>(lnp + 2 * d);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
    const int rank = static_cast<int>(ckv::cluster_rank()), row0 = (static_cast<int>(blockIdx.x) >> CL) * R;

    // ---- exchanges -------------------------------------------------------------------------------------------------
    // What a stage sends to a block reports to its bars[stage % 4].
    int stage = 0;
    auto put = [&](auto *at, int dst, auto v) { send(ckv::map_to_rank(at, dst), v, ckv::map_to_rank(&bars[stage & 3], dst)); };
    auto receive = [&](int bytes) {
        uint64_t *const bar = &bars[stage & 3];
        if (tid == 0) tc::mbar_expect_tx(bar, bytes);
        ckv::mbar_wait_cluster(bar, stage >> 2 & 1, &abort_flag);
        ++stage;
    };

    // ---- projections -----------------------------------------------------------------------------------------------
    // FPW features of a warp at a time and all of K (kHeld / FPW * 128 at most: see cluster_supports), rows in fours: the sums of a four are reduced over the lanes, which leaves the one of feature f and row r in the
    // lanes from (f * 4 + r) * 8 / FPW on.
    Quad w[kHeld];
    float bias_first;
    auto range = [&](int M, int fpw, int &begin, int &end) {      // this block's features
        const int per = (((M + C - 1) >> CL) + fpw - 1) / fpw * fpw;
        begin = rank * per;
        end = min(M, begin + per);
    };
    auto load_window = [&](auto fpw_c, const float *W, int K, int f0, int end) {
        constexpr int FPW = decltype(fpw_c)::value, kAhead = kHeld / FPW;
        const float *const at = W + static_cast<size_t>(f0) * K + lane * 4;
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            const bool in = i * 128 + lane * 4 < K;
#pragma unroll
            for (int f = 0; f < FPW; ++f) w[f * kAhead + i] = load_weights(at + f * K + i * 128, in && f0 + f < end);
        }
    };
    auto load_bias = [&](auto fpw_c, const float *bias, int f0, int end) {
        const int f = f0 + lane * decltype(fpw_c)::value / 32;
        return load_weight(bias + f, bias && f < end);
    };
    // the first weights of a projection, requested ahead of its input
    auto request = [&](auto fpw_c, const float *W, const float *bias, int M, int K) {
        int begin, end;
        range(M, decltype(fpw_c)::value, begin, end);
        const int f0 = begin + warp * decltype(fpw_c)::value;
        load_window(fpw_c, W, K, f0, end);
        bias_first = load_bias(fpw_c, bias, f0, end);
    };
    // sink(f0, rows from, this lane's sum): all lanes of the warp call it
    auto project = [&](auto fpw_c, const float *in, const float *W, const float *bias, int M, int K, auto sink) {
        constexpr int FPW = decltype(fpw_c)::value, kAhead = kHeld / FPW, N = FPW * 4;
        int begin, end;
        range(M, FPW, begin, end);
#pragma unroll 1
        for (int f0 = begin + warp * FPW; f0 < end; f0 += kClusterWarps * FPW) {
            unsigned long long acc[R / 4][N];                 // (sums of the even and of the odd k)
#pragma unroll
            for (int i = 0; i < R / 4 * N; ++i) acc[i / N][i % N] = 0ull;
#pragma unroll
            for (int i = 0; i < kAhead; ++i) {
                if (i * 128 >= K) break;
                const int k = i * 128 + lane * 4;
                ulonglong2 x[R];
#pragma unroll
                for (int r = 0; r < R; ++r) x[r] = k < K ? *reinterpret_cast<const ulonglong2 *>(in + r * K + k) : make_ulonglong2(0ull, 0ull);
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int f = 0; f < FPW; ++f) {
                        fma2(acc[r / 4][f * 4 + r % 4], x[r].x, w[f * kAhead + i].a);
                        fma2(acc[r / 4][f * 4 + r % 4], x[r].y, w[f * kAhead + i].b);
                    }
            }
            const float b = bias_first;
            const int next = f0 + kClusterWarps * FPW;
            if (next < end) {
                load_window(fpw_c, W, K, next, end);
                bias_first = load_bias(fpw_c, bias, next, end);
            }
#pragma unroll
            for (int h = 0; h < R / 4; ++h) {
                float sums[N];
#pragma unroll
                for (int i = 0; i < N; ++i) sums[i] = pair_sum(acc[h][i]);
                sink(f0, h * 4, reduce_transposed<N>(sums, lane) + b);
            }
        }
    };
    const std::integral_constant<int, 2> narrow;
    const std::integral_constant<int, 8> wide;

    // ---- LayerNorm ------------------------------------------------------------------------------------------------------
    auto request_ln = [&](const float *g, const float *b) {
#pragma unroll 1
        for (int i = tid; i < d; i += kClusterThreads) {
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(tc::smem_u32(lnp + i)), "l"(g + i) : "memory");
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(tc::smem_u32(lnp + d + i)), "l"(b + i) : "memory");
        }
    };
    const float inv_d = 1.f / d;
    auto normalise = [&] {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
#pragma unroll 1
        for (int r = warp; r < R; r += kClusterWarps) {
            const float *const x = xs + r * d;
            float s = 0.f, q = 0.f;
#pragma unroll 2
            for (int k = lane * 4; k < d; k += 128) {
                const float4 v = *reinterpret_cast<const float4 *>(x + k);
                s += (v.x + v.y) + (v.z + v.w);
            }
            const float mean = warp_sum(s) * inv_d;
#pragma unroll 2
            for (int k = lane * 4; k < d; k += 128) {
                const float4 v = *reinterpret_cast<const float4 *>(x + k);
                const float d0 = v.x - mean, d1 = v.y - mean, d2 = v.z - mean, d3 = v.w - mean;
                q += (d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3);
            }
            const float2 st = make_float2(mean, rsqrtf(warp_sum(q) * inv_d + p.eps));
#pragma unroll 2
            for (int k = lane * 4; k < d; k += 128)
                *reinterpret_cast<float4 *>(ns + r * d + k) = normalize(*reinterpret_cast<const float4 *>(x + k), st, *reinterpret_cast<const float4 *>(lnp + k),
                                                                        *reinterpret_cast<const float4 *>(lnp + d + k));
        }
        __syncthreads();
    };

    const int h_inv = 65536 / H + 1;                          // pair / H = pair * h_inv >> 16 (pairs are few)
    // ---- attention -------------------------------------------------------------------------------------------------------
    // Pair (row, head) = slot * C + rank.  `groups` pairs at a time with `nw` warps each; a warp takes 8 positions at a time, two per lane.
    int groups = 1;
    while (groups < min(slots, kClusterWarps)) groups <<= 1;
    const int nw = kClusterWarps / groups, group = warp / nw, wi = warp % nw, dg = lane & 7, pg = lane >> 3;
    constexpr int kPos = 2, kStep = kPos * 4;
    RawLane<float> rk[kPos], rv[kPos];
    struct Pair { bool live; int slot, row, head, len; const float *k, *v; };
    auto pair_of = [&](bool cross, int l, int slot) {
        Pair a{};
        const int pair = slot * C + rank;
        a.slot = slot; a.row = pair * h_inv >> 16; a.head = pair - a.row * H;
        const int4 ri = slot < slots && a.row < R ? s_row[a.row] : make_int4(-1, 0, 0, 0);
        a.live = ri.x >= 0;
        if (!a.live) return a;
        if (cross) {
            a.len = ri.z;
            a.k = p.cross + l * p.cross_layer_elems + (static_cast<size_t>(a.head) * p.frame_capacity + ri.w) * kHeadDim + dg * 8;
            a.v = a.k + static_cast<size_t>(H) * p.frame_capacity * kHeadDim;
        } else {
            a.len = ri.y + 1;
            a.k = p.self_cache + l * p.self_layer_elems + (static_cast<size_t>(ri.x) * 2 * H + a.head) * p.max_dec_len * kHeadDim + dg * 8;
            a.v = a.k + static_cast<size_t>(H) * p.max_dec_len * kHeadDim;
        }
        return a;
    };
    auto load_positions = [&](const Pair &a, bool cross, int p0) {
#pragma unroll
        for (int i = 0; i < kPos; ++i) {
            const int pos = p0 + i * 4 + pg;
            if (a.live && pos < (cross ? a.len : a.len - 1)) { rk[i].load(a.k + static_cast<size_t>(pos) * kHeadDim); rv[i].load(a.v + static_cast<size_t>(pos) * kHeadDim); }
            else { rk[i].zero(); rv[i].zero(); }
        }
    };
    auto attend = [&](bool cross, int l) {
#pragma unroll 1
        for (int s0 = 0; s0 < slots; s0 += groups) {
            const Pair a = pair_of(cross, l, s0 + group);
            if (s0 > 0) load_positions(a, cross, wi * kStep);
            float m = -INFINITY, sum = 0.f, acc[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[j] = 0.f;
            if (a.live) {
                const float *const q = qs + a.slot * 3 * kHeadDim + dg * 8;
                float qv[8];
                load_n<8>(q, qv);
#pragma unroll
                for (int j = 0; j < 8; ++j) qv[j] *= 0.125f * kScoreUnit;               // 1 / sqrt(64)
                if (!cross && wi == 0 && pg == 0) {          // the new position into the cache; nobody reads it there in this step
                    RawLane<float> n;
                    n.load(q + kHeadDim); n.store(const_cast<float *>(a.k) + static_cast<size_t>(a.len - 1) * kHeadDim);
                    n.load(q + 2 * kHeadDim); n.store(const_cast<float *>(a.v) + static_cast<size_t>(a.len - 1) * kHeadDim);
                }
#pragma unroll 1
                for (int p0 = wi * kStep; p0 < a.len; p0 += nw * kStep) {
                    if (p0 != wi * kStep) load_positions(a, cross, p0);
                    float s[kPos], cmax = -INFINITY;
#pragma unroll
                    for (int i = 0; i < kPos; ++i) {
                        const int pos = p0 + i * 4 + pg;
                        if (!cross && pos == a.len - 1) { rk[i].load(q + kHeadDim); rv[i].load(q + 2 * kHeadDim); }
                        float kf[8], dot = 0.f;
                        rk[i].get(kf);
#pragma unroll
                        for (int j = 0; j < 8; ++j) dot = fmaf(qv[j], kf[j], dot);
#pragma unroll
                        for (int o = 1; o < 8; o <<= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
                        s[i] = pos < a.len ? dot : -INFINITY;
                        cmax = fmaxf(cmax, s[i]);
                    }
                    cmax = fmaxf(cmax, __shfl_xor_sync(0xffffffffu, cmax, 8));
                    cmax = fmaxf(cmax, __shfl_xor_sync(0xffffffffu, cmax, 16));
                    const float m_new = fmaxf(m, cmax), corr = softmax_weight<float>(m - m_new);
                    sum *= corr;
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc[j] *= corr;
#pragma unroll
                    for (int i = 0; i < kPos; ++i) {
                        const float pr = softmax_weight<float>(s[i] - m_new);
                        float vf[8];
                        rv[i].get(vf);
                        sum += pr;
#pragma unroll
                        for (int j = 0; j < 8; ++j) acc[j] = fmaf(pr, vf[j], acc[j]);
                    }
                    m = m_new;
                }
            }
            if (lane == 0) s_max[warp] = m;
            __syncthreads();
            float big = s_max[group * nw + (lane & (nw - 1))];
#pragma unroll 1
            for (int o = nw >> 1; o > 0; o >>= 1) big = fmaxf(big, __shfl_xor_sync(0xffffffffu, big, o));
            const float wgt = m == -INFINITY ? 0.f : softmax_weight<float>(m - big);
#pragma unroll
            for (int o = 8; o < 32; o <<= 1) {
                sum += __shfl_xor_sync(0xffffffffu, sum, o);
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
            }
            if (lane == 0) s_sum[warp] = sum * wgt;
            if (pg == 0) {
#pragma unroll
                for (int j = 0; j < 8; ++j) red[warp * kHeadDim + dg * 8 + j] = acc[j] * wgt;
            }
            __syncthreads();
#pragma unroll 1
            for (int i = tid; i < groups * kHeadDim; i += kClusterThreads) {
                const int g = i / kHeadDim, e = i % kHeadDim;
                float total = 0.f, o = 0.f;
#pragma unroll 8
                for (int j = 0; j < nw; ++j) { total += s_sum[g * nw + j]; o += red[(g * nw + j) * kHeadDim + e]; }
                outs[i] = o / total;
            }
            __syncthreads();
#pragma unroll 1
            for (int i = tid; i < groups * 16 * C; i += kClusterThreads) {
                const int g = i >> (4 + CL), dst = (i >> 4) & (C - 1), c = i & 15;
                const int pair = (s0 + g) * C + rank, row = pair * h_inv >> 16, head = pair - row * H;
                if (s0 + g >= slots || row >= R || s_row[row].x < 0) continue;
                put(as + row * d + head * kHeadDim + c * 4, dst, *reinterpret_cast<const float4 *>(outs + g * kHeadDim + c * 4));
            }
        }
    };
    auto to_pair = [&](int kind, int r, int c, float y) {      // component c of q, k or v (kind) of row r: to the block of its pair
        const int pair = r * H + c / kHeadDim;
        put(qs + ((pair >> CL) * 3 + kind) * kHeadDim + c % kHeadDim, pair & (C - 1), y);
    };

    // ---- the step ----------------------------------------------------------------------------------------------------------
    // One copy of everything in the code, gone through six times per layer and once at the end.
    for (int i = tid; i < p.n_layers * static_cast<int>(sizeof(ClusterLayer) / 8); i += kClusterThreads)
        reinterpret_cast<unsigned long long *>(layers)[i] = reinterpret_cast<const unsigned long long *>(p.layers)[i];
    if (tid == 0) {
        for (int i = 0; i < 4; ++i) tc::mbar_init(&bars[i], 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    enum { QKV, O, QC, OC, FF1, FF2, VOCAB };
    int phase = QKV, l = 0, M = 3 * d, K = d;
    const float *W = layers->w_qkv, *bias = layers->b_qkv;
    request(wide, W, bias, M, K);
    request_ln(layers->ln1_g, layers->ln1_b);
    sg::pdl_wait();
    const int n_rows = p.state->n_active;
    sg::pdl_launch_dependents();                              // (the row table is there: see StepGemmParams)
    if (row0 >= n_rows) return;                               // (all blocks of the cluster)
    if (tid < R) {
        s_row[tid] = row0 + tid < n_rows ? p.row_info[row0 + tid] : make_int4(-1, 0, 0, 0);
        s_key[tid] = 0ull;
    }
#pragma unroll 1
    for (int i = tid; i < R * d; i += kClusterThreads) as[i] = 0.f;
    __syncthreads();
#pragma unroll 1
    for (int i = tid; i < R * d; i += kClusterThreads) {
        const int r = i / d, c = i - r * d;
        const int4 ri = s_row[r];
        float v = 0.f;
        if (ri.x >= 0) {
            if (p.x) v = p.x[static_cast<size_t>(row0 + r) * d + c];
            else {
                const int tok = min(max(p.tokens[ri.x], 0), p.vocab - 1);
                v = p.embed[static_cast<size_t>(tok) * d + c] * p.scale + p.pe[static_cast<size_t>(ri.y) * d + c];
            }
        }
        xs[i] = v;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    cluster_arrive();                                         // every block of the cluster has started, cleared its rows and made its barriers
    cluster_wait();
    const int mine = (R * H - rank + C - 1) >> CL;            // this block's pairs, those of missing rows included
    const int attended = min(n_rows - row0, R) * d * 4;       // bytes of the attention rows
#pragma unroll 1
    for (;;) {
        const ClusterLayer &L = layers[min(l, p.n_layers - 1)];
        const bool many = phase == QKV || phase == FF1 || phase == VOCAB, cross = phase == QC;
        if (many || cross) {
            normalise();
            const bool last = l == p.n_layers - 1;
            if (phase != VOCAB)
                request_ln(phase == QKV ? L.ln2_g : cross ? L.ln3_g : last ? p.final_ln_g : (&L)[1].ln1_g,
                           phase == QKV ? L.ln2_b : cross ? L.ln3_b : last ? p.final_ln_b : (&L)[1].ln1_b);
        }
        if (many)
            project(wide, ns, W, bias, M, K, [&](int f0, int r0, float y) {
                const int f = f0 + (lane >> 2), r = r0 + (lane & 3);
                if (phase == QKV) {
                    const int kind = (f >= d) + (f >= 2 * d);
                    if (f < M) to_pair(kind, r, f - kind * d, y);
                } else if (phase == FF1) {                    // (whole eights of features) 16 bytes of a row to a block at a time
                    hs[r * F + f] = fmaxf(y, 0.f);
                    __syncwarp();
                    float *const at = hs + (r0 + (lane & 3)) * F + f0 + (lane >> 2 & 1) * 4;
                    const float4 v = *reinterpret_cast<const float4 *>(at);
#pragma unroll 4
                    for (int dst = lane >> 3; dst < C; dst += 4) put(at, dst, v);
                } else {
                    const int u = s_row[r].x;
                    unsigned long long key = 0ull;
                    if (f < M && u >= 0) {
                        if (p.logits_out) p.logits_out[static_cast<size_t>(u) * p.vocab + f] = y;
                        key = argmax_key(y, static_cast<uint32_t>(f));
                    }
#pragma unroll
                    for (int o = 4; o < 32; o <<= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
                    if (lane < 4 && key) atomicMax(&s_key[r], key);
                }
            });
        else
            project(narrow, cross ? ns : phase == FF2 ? hs : as, W, bias, M, K, [&](int f0, int r0, float y) {
                const int f = f0 + (lane >> 4), r = r0 + (lane >> 2 & 3);
                if (cross) {
                    if ((lane & 3) == 0) to_pair(0, r, f, y);
                } else {                                      // residual rows: two features of a row to a block at a time
                    const float v = xs[r * d + f] + y, other = __shfl_xor_sync(0xffffffffu, v, 16);
                    const float2 both = lane < 16 ? make_float2(v, other) : make_float2(other, v);
#pragma unroll 2
                    for (int dst = (lane & 3) + (lane >> 4) * 4; dst < C; dst += 8) put(xs + r * d + f0, dst, both);
                }
            });
        if (phase == VOCAB) break;
        const int at_layer = l, bytes = phase == QKV ? mine * 3 * kHeadDim * 4 : cross ? mine * kHeadDim * 4 : R * (phase == FF1 ? F : d) * 4;
        const bool attention = phase == QKV || cross;
        if (attention) load_positions(pair_of(cross, l, group), cross, wi * kStep);
        // what comes next
        if (phase == FF2) phase = ++l < p.n_layers ? QKV : VOCAB;
        else ++phase;
        const ClusterLayer &N = layers[min(l, p.n_layers - 1)];
        K = d;
        M = d;
        switch (phase) {
        case QKV: W = N.w_qkv; bias = N.b_qkv; M = 3 * d; break;
        case O: W = N.w_o; bias = N.b_o; break;
        case QC: W = N.w_q_c; bias = N.b_q_c; break;
        case OC: W = N.w_o_c; bias = N.b_o_c; break;
        case FF1: W = N.w_ff1; bias = N.b_ff1; M = F; break;
        case FF2: W = N.w_ff2; bias = N.b_ff2; K = F; break;
        default: W = p.w_out; bias = p.b_out; M = p.vocab;
        }
        if (phase == QKV || phase == FF1 || phase == VOCAB) request(wide, W, bias, M, K);
        else request(narrow, W, bias, M, K);
        receive(bytes);
        if (attention) {
            attend(cross, at_layer);
            receive(attended);
        }
        if (phase == VOCAB) asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");      // this block sends nothing more
    }
    __syncthreads();
    if (tid < R && row0 + tid < n_rows && s_key[tid] != 0ull) atomicMax(p.keys + row0 + tid, s_key[tid]);
    if (tid == 0 && abort_flag) atomicExch(&p.state->error, tc::kErrTimeout);
    cluster_wait();                                           // (a block that has given up a wait may be ahead of what is sent to it)
}

}  // namespace f32
}  // namespace aed

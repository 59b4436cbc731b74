// fp32 projections (fp32 configuration: FMA only, no TF32) of a step's rows or of encoder frames, with the LayerNorm of the
// input rows and the epilogue fused.
//
//   out[r, o] = sum_k A'[r, k] * W[o, k] + bias[o],   A' = LayerNorm(A) or A
//
// Steps of few rows (rows_kernel): a projection is bound by latency, not by arithmetic: one warp
// per one or two output features and RT rows, lanes along K.  A warp's weights (16 bytes per lane and 128 k) are requested
// before the programmatic-dependency wait; the rows are staged through shared memory (normalised on the way); the RT x FPW
// sums of the lanes are reduced by halving, one value per lane in the end.  The former 64-row x 32-feature tiles left most
// of a 4-row tile idle and walked K in steps of 32 with a memory latency each.  Decode step of the 2-layer fp32 model at 4
// rows: 316 us before (27 launches), 52 us now (18 launches of about 2.8 us, which is what a link of the chain costs).
#pragma once
#include "step_gemm.cuh"

namespace aed {
namespace f32 {

enum Epilogue { EPI_STORE = 0, EPI_RELU = 1, EPI_RESID = 2, EPI_LOGITS = 3, EPI_CROSSKV = 4 };

constexpr int kTileK = 1024;                 // columns of the rows staged at a time
constexpr int kWarps = 8;

struct RowsArgs {
    int after_rows;
    const DecState *state;
    int rows_fixed;                          // >= 0: number of rows; < 0: read it from the decode state
    const float *a;                          // [rows, K]
    const float *ln_g, *ln_b;                // LayerNorm of the rows (null: none)
    float eps;
    const float *w, *bias;                   // [M, K], [M] or null
    int M, K;
    float *out;                              // STORE, RELU, RESID: [rows, ldo]; CROSSKV: this layer's store [2][H][frame_capacity][64]
    int ldo;
    float *logits_out;                       // LOGITS: [batch, M] by utterance or null
    unsigned long long *keys;                // LOGITS: packed argmax keys [rows]
    const int32_t *active_list;
    int d_model, n_heads, frame_capacity, frame0;      // CROSSKV
};

__host__ __device__ constexpr int rows_smem(int rt, int k) { return rt * (k < kTileK ? k : kTileK) * 4; }

// Sums of N (a power of two, at most 32) values over the warp: lane l ends up with the sum of value l >> (5 - log2 N).
template <int N>
__device__ __forceinline__ float reduce_transposed(float (&v)[N], int lane)
{
    int o = 16;
#pragma unroll
    for (int n = N; n > 1; n >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int j = 0; j < n / 2; ++j) {
            const float give = up ? v[j] : v[j + n / 2], keep = up ? v[j + n / 2] : v[j];
            v[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    float s = v[0];
    for (; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// (mean, rstd) of a row by one warp: two passes, the second reads what the first brought into L1
__device__ __forceinline__ float2 row_stats(const float *a, int K, float eps, int lane)
{
    float s = 0.f, q = 0.f;
    for (int k = lane * 4; k < K; k += 128) {
        const float4 v = *reinterpret_cast<const float4 *>(a + k);
        s += (v.x + v.y) + (v.z + v.w);
    }
    const float mean = warp_sum(s) / K;
    for (int k = lane * 4; k < K; k += 128) {
        const float4 v = *reinterpret_cast<const float4 *>(a + k);
        const float d0 = v.x - mean, d1 = v.y - mean, d2 = v.z - mean, d3 = v.w - mean;
        q += (d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3);
    }
    return make_float2(mean, rsqrtf(warp_sum(q) / K + eps));
}
template <bool kLnVec> __device__ __forceinline__ float4 load_ln(const float *v)
{
    return kLnVec ? __ldg(reinterpret_cast<const float4 *>(v)) : make_float4(__ldg(v), __ldg(v + 1), __ldg(v + 2), __ldg(v + 3));
}
__device__ __forceinline__ float4 normalize(float4 v, float2 st, float4 g, float4 b)
{
    return make_float4(fmaf(g.x * (v.x - st.x), st.y, b.x), fmaf(g.y * (v.y - st.x), st.y, b.y), fmaf(g.z * (v.z - st.x), st.y, b.z),
                       fmaf(g.w * (v.w - st.x), st.y, b.w));
}
// the result y of row r and output feature o (but for the key of the greedy choice)
template <int EPI> __device__ __forceinline__ void store(const RowsArgs &p, int r, int o, float y)
{
    if (EPI == EPI_STORE) p.out[static_cast<size_t>(r) * p.ldo + o] = y;
    else if (EPI == EPI_RELU) p.out[static_cast<size_t>(r) * p.ldo + o] = fmaxf(y, 0.f);
    else if (EPI == EPI_RESID) p.out[static_cast<size_t>(r) * p.ldo + o] += y;
    else if (EPI == EPI_LOGITS) {
        if (p.logits_out) p.logits_out[static_cast<size_t>(p.active_list[r]) * p.M + o] = y;
    } else {
        const int kv = o / p.d_model, c = o % p.d_model, h = c / kHeadDim, e = c % kHeadDim;
        p.out[((static_cast<size_t>(kv) * p.n_heads + h) * p.frame_capacity + p.frame0 + r) * kHeadDim + e] = y;
    }
}

// grid: x = blocks of blockDim / 32 * FPW output features, y = tiles of RT rows.
// kLnVec: the LayerNorm vectors are read 16 bytes at a time, otherwise one value (the caller may have put them at any element).
// A form of its own and not a test in the loop: that took 54 us instead of 52 per step of 4 rows of the 2-layer model.
template <int EPI, int RT, int FPW, bool kLnVec>
__global__ void __launch_bounds__(kWarps * 32)
rows_kernel(const RowsArgs p)
{
    constexpr int N = RT * FPW, kAhead = 8 / FPW;          // weight loads per lane and feature requested ahead
    extern __shared__ __align__(16) float s_rows[];        // [RT][columns of the tile]
    __shared__ float2 s_stat[RT];
    __shared__ unsigned long long s_key[RT];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;
    const int f0 = (blockIdx.x * n_warps + warp) * FPW, row0 = blockIdx.y * RT;
    int n_rows = p.rows_fixed >= 0 ? p.rows_fixed : p.after_rows ? 0 : p.state->n_active;
    if (!p.after_rows) sg::pdl_launch_dependents();
    const int K = p.K;
    float4 w[FPW][kAhead];
    auto load_w = [&](int f, int k) {
        return (f0 + f < p.M && k < K) ? __ldg(reinterpret_cast<const float4 *>(p.w + static_cast<size_t>(f0 + f) * K + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
#pragma unroll
    for (int f = 0; f < FPW; ++f)
#pragma unroll
        for (int i = 0; i < kAhead; ++i) w[f][i] = load_w(f, i * 128 + lane * 4);
    sg::pdl_wait();
    if (p.after_rows) { n_rows = p.state->n_active; sg::pdl_launch_dependents(); }      // (see StepGemmParams)
    if (row0 >= n_rows) return;
    if (EPI == EPI_LOGITS && threadIdx.x < RT) s_key[threadIdx.x] = 0ull;
    if (p.ln_g) {
        for (int r = warp; r < RT; r += n_warps) {
            const float2 st = row_stats(p.a + static_cast<size_t>(min(row0 + r, n_rows - 1)) * K, K, p.eps, lane);
            if (lane == 0) s_stat[r] = st;
        }
        __syncthreads();
    }
    float acc[N];
#pragma unroll
    for (int i = 0; i < N; ++i) acc[i] = 0.f;
    for (int k0 = 0; k0 < K; k0 += kTileK) {
        const int kt = min(K - k0, kTileK), ld = min(K, kTileK);
        if (k0 > 0) __syncthreads();
        for (int i = threadIdx.x; i < RT * (kt / 4); i += blockDim.x) {
            const int r = i / (kt / 4), k = (i % (kt / 4)) * 4;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (row0 + r < n_rows) {
                v = *reinterpret_cast<const float4 *>(p.a + static_cast<size_t>(row0 + r) * K + k0 + k);
                if (p.ln_g) v = normalize(v, s_stat[r], load_ln<kLnVec>(p.ln_g + k0 + k), load_ln<kLnVec>(p.ln_b + k0 + k));
            }
            *reinterpret_cast<float4 *>(s_rows + r * ld + k) = v;
        }
        __syncthreads();
        for (int i0 = 0; i0 * 128 < kt; i0 += kAhead) {
#pragma unroll
            for (int i = 0; i < kAhead; ++i) {
                const int k = (i0 + i) * 128 + lane * 4;
                if (k < kt) {
#pragma unroll
                    for (int r = 0; r < RT; ++r) {
                        const float4 x = *reinterpret_cast<const float4 *>(s_rows + r * ld + k);
#pragma unroll
                        for (int f = 0; f < FPW; ++f)
                            acc[f * RT + r] = fmaf(x.w, w[f][i].w, fmaf(x.z, w[f][i].z, fmaf(x.y, w[f][i].y, fmaf(x.x, w[f][i].x, acc[f * RT + r]))));
                    }
                }
            }
            // (whole tiles are multiples of kAhead * 128 columns, so the next weights follow on)
            const int next = k0 + (i0 + kAhead) * 128;
            if (next < K) {
#pragma unroll
                for (int f = 0; f < FPW; ++f)
#pragma unroll
                    for (int i = 0; i < kAhead; ++i) w[f][i] = load_w(f, next + i * 128 + lane * 4);
            }
        }
    }
    const float sum = reduce_transposed<N>(acc, lane);
    const int idx = lane * N / 32, r = row0 + idx % RT, o = f0 + idx / RT;
    const bool mine = lane % (32 / N) == 0 && r < n_rows && o < p.M;
    if (mine) {
        const float y = sum + (p.bias ? p.bias[o] : 0.f);
        store<EPI>(p, r, o, y);
        if (EPI == EPI_LOGITS) atomicMax(&s_key[idx % RT], argmax_key(y, static_cast<uint32_t>(o)));
    }
    if (EPI == EPI_LOGITS) {
        __syncthreads();
        if (threadIdx.x < RT && row0 + static_cast<int>(threadIdx.x) < n_rows && s_key[threadIdx.x] != 0ull) atomicMax(p.keys + row0 + threadIdx.x, s_key[threadIdx.x]);
    }
}

// The same for many rows: tiles of 64 rows x 64 features, 256 threads with 4 x 4 sums each, K in slices of 32 through two
// buffers of shared memory.  The kernel above reads its weights from L2 once per 8 rows and is bound by that, at about 15
// TFLOP/s; this one is bound by FMA issue (a quarter of the slots go to shared-memory loads, a tenth to the sums of sums), at
// 30 TFLOP/s: cross-attention keys and values of 32000 frames, 4 layers, d 1024 in 17.2 ms against 35.9, d 256 and 2 layers
// 0.64 against 2.04; 512 rows of a step of the 4-layer model 4.7 against 6.1 ms.  A tile takes about 0.05 us per k whether there
// is one or two on every SM, so it needs enough of them: see use_tiles.
// Sums are taken in four steps (8 products, 4 of those, 4 of those, the rest), so that they round like the lanes' sums of the
// kernel above (logits against the fp64 checker 1.45e-7 with either kernel; in one chain 3.6e-7, in slices of 32 1.74e-7).
// Grid: row tile * feature tiles + feature tile, in x alone, so that any number of rows fits.
constexpr int kTile = 64, kSlice = 32, kShort = 8, kTileThreads = 256, kTilePitch = kSlice + 4;

// Where the two kernels take the same time: 96 tiles' worth of outputs, whatever K is (M x rows in thousands: 338 to 384 with
// K 1024 and 4096, 262 to 369 with 512, 256 to 300 with 256), but for tiles that would be half empty (16384 features: 24 rows
// 75 us against 97, 32 rows 95 against 97, 48 rows 137 against 97).
inline bool use_tiles(int M, int rows) { return rows > kTile / 2 && static_cast<long long>(M) * rows >= 96ll * kTile * kTile; }

template <int EPI, bool kLnVec>
__global__ void __launch_bounds__(kTileThreads, 2)
tile_kernel(const RowsArgs p)
{
    __shared__ __align__(16) float s_a[2][kTile * kTilePitch], s_w[2][kTile * kTilePitch];
    __shared__ float2 s_stat[kTile];
    __shared__ unsigned long long s_key[kTile];
    const int f_tiles = (p.M + kTile - 1) / kTile, K = p.K;
    const int row0 = static_cast<int>(blockIdx.x / f_tiles) * kTile, f0 = static_cast<int>(blockIdx.x % f_tiles) * kTile;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    sg::pdl_wait();
    sg::pdl_launch_dependents();
    const int n_rows = p.rows_fixed >= 0 ? p.rows_fixed : p.state->n_active;
    if (row0 >= n_rows) return;
    if (EPI == EPI_LOGITS && threadIdx.x < kTile) s_key[threadIdx.x] = 0ull;
    if (p.ln_g) {
        for (int r = warp; r < kTile; r += kTileThreads / 32) {
            const float2 st = row_stats(p.a + static_cast<size_t>(min(row0 + r, n_rows - 1)) * K, K, p.eps, lane);
            if (lane == 0) s_stat[r] = st;
        }
        __syncthreads();
    }
    // a slice: rows (features) threadIdx.x / 8 and 32 more, 4 values at 4 * (threadIdx.x % 8)
    const int lr = threadIdx.x >> 3, lk = (threadIdx.x & 7) * 4;
    float4 va[2];
    auto fetch = [&](int buf, int k0) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int r = row0 + lr + 32 * i, f = f0 + lr + 32 * i;
            va[i] = r < n_rows ? *reinterpret_cast<const float4 *>(p.a + static_cast<size_t>(r) * K + k0 + lk) : make_float4(0.f, 0.f, 0.f, 0.f);
            // (0 bytes of the source: zeros)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(tc::smem_u32(&s_w[buf][(lr + 32 * i) * kTilePitch + lk])),
                         "l"(p.w + static_cast<size_t>(min(f, p.M - 1)) * K + k0 + lk), "r"(f < p.M ? 16 : 0) : "memory");
        }
    };
    auto put = [&](int buf, int k0) {
        float4 g, b;
        if (p.ln_g) { g = load_ln<kLnVec>(p.ln_g + k0 + lk); b = load_ln<kLnVec>(p.ln_b + k0 + lk); }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            if (p.ln_g) va[i] = normalize(va[i], s_stat[lr + 32 * i], g, b);
            *reinterpret_cast<float4 *>(&s_a[buf][(lr + 32 * i) * kTilePitch + lk]) = va[i];
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    };
    // this thread's sums: rows tr + 16 i, features tf + 16 j (a warp reads 4 rows and 8 features of a slice, each in banks of its own)
    const int tr = (warp >> 1) * 4 + (lane >> 3), tf = (warp & 1) * 8 + (lane & 7);
    float acc[4][4], group[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    fetch(0, 0);
    put(0, 0);
    for (int k0 = 0, buf = 0, n = 0; k0 < K; k0 += kSlice, buf ^= 1, ++n) {
        __syncthreads();
        const bool more = k0 + kSlice < K;
        if (more) fetch(buf ^ 1, k0 + kSlice);
        float slice[4][4];
#pragma unroll
        for (int k = 0; k < kSlice; k += kShort) {
            float part[4][4];
#pragma unroll
            for (int k4 = 0; k4 < kShort; k4 += 4) {
                float4 a[4], w[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    a[i] = *reinterpret_cast<const float4 *>(&s_a[buf][(tr + 16 * i) * kTilePitch + k + k4]);
                    w[i] = *reinterpret_cast<const float4 *>(&s_w[buf][(tf + 16 * i) * kTilePitch + k + k4]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        part[i][j] = fmaf(a[i].w, w[j].w, fmaf(a[i].z, w[j].z, fmaf(a[i].y, w[j].y, k4 == 0 ? a[i].x * w[j].x : fmaf(a[i].x, w[j].x, part[i][j]))));
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) slice[i][j] = k == 0 ? part[i][j] : slice[i][j] + part[i][j];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) group[i][j] = n % 4 == 0 ? slice[i][j] : group[i][j] + slice[i][j];
        if (n % 4 == 3 || !more) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] += group[i][j];
        }
        if (more) put(buf ^ 1, k0 + kSlice);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = row0 + tr + 16 * i;
        unsigned long long key = 0ull;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int o = f0 + tf + 16 * j;
            if (r >= n_rows || o >= p.M) continue;
            const float y = acc[i][j] + (p.bias ? p.bias[o] : 0.f);
            store<EPI>(p, r, o, y);
            if (EPI == EPI_LOGITS) key = max(key, argmax_key(y, static_cast<uint32_t>(o)));
        }
        if (EPI == EPI_LOGITS && key != 0ull) atomicMax(&s_key[tr + 16 * i], key);
    }
    if (EPI == EPI_LOGITS) {
        __syncthreads();
        if (threadIdx.x < kTile && s_key[threadIdx.x] != 0ull) atomicMax(p.keys + row0 + threadIdx.x, s_key[threadIdx.x]);
    }
}

}  // namespace f32
}  // namespace aed

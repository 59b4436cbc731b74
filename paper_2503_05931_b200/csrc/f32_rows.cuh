// fp32 projections (fp32 configuration: FMA only, no TF32) of a step's rows or of encoder frames, with the LayerNorm of the
// input rows and the epilogue fused.
//
//   out[r, o] = sum_k A'[r, k] * W[o, k] + bias[o],   A' = LayerNorm(A) or A
//
// The configuration is small and its steps have few rows, so a projection is bound by latency, not by arithmetic: one warp
// per one or two output features and RT rows, lanes along K.  A warp's weights (16 bytes per lane and 128 k) are requested
// before the programmatic-dependency wait; the rows are staged through shared memory (normalised on the way); the RT x FPW
// sums of the lanes are reduced by halving, one value per lane in the end.  The former 64-row x 32-feature tiles left most
// of a 4-row tile idle and walked K in steps of 32 with a memory latency each.  Decode step of the 2-layer fp32 model at 4
// rows: 316 us before (27 launches), 56 us now (20 launches of about 2.8 us, which is what a link of the chain costs).
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
        // two passes over the row; the second reads what the first brought into L1
        for (int r = warp; r < RT; r += n_warps) {
            const float *a = p.a + static_cast<size_t>(min(row0 + r, n_rows - 1)) * K;
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
            q = warp_sum(q);
            if (lane == 0) s_stat[r] = make_float2(mean, rsqrtf(q / K + p.eps));
        }
        __syncthreads();
    }
    auto load_ln = [](const float *v) {
        return kLnVec ? __ldg(reinterpret_cast<const float4 *>(v)) : make_float4(__ldg(v), __ldg(v + 1), __ldg(v + 2), __ldg(v + 3));
    };
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
                if (p.ln_g) {
                    const float2 st = s_stat[r];
                    const float4 g = load_ln(p.ln_g + k0 + k), b = load_ln(p.ln_b + k0 + k);
                    v.x = fmaf(g.x * (v.x - st.x), st.y, b.x); v.y = fmaf(g.y * (v.y - st.x), st.y, b.y);
                    v.z = fmaf(g.z * (v.z - st.x), st.y, b.z); v.w = fmaf(g.w * (v.w - st.x), st.y, b.w);
                }
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
        if (EPI == EPI_STORE) p.out[static_cast<size_t>(r) * p.ldo + o] = y;
        else if (EPI == EPI_RELU) p.out[static_cast<size_t>(r) * p.ldo + o] = fmaxf(y, 0.f);
        else if (EPI == EPI_RESID) p.out[static_cast<size_t>(r) * p.ldo + o] += y;
        else if (EPI == EPI_LOGITS) {
            if (p.logits_out) p.logits_out[static_cast<size_t>(p.active_list[r]) * p.M + o] = y;
            atomicMax(&s_key[idx % RT], argmax_key(y, static_cast<uint32_t>(o)));
        } else {
            const int kv = o / p.d_model, c = o % p.d_model, h = c / kHeadDim, e = c % kHeadDim;
            p.out[((static_cast<size_t>(kv) * p.n_heads + h) * p.frame_capacity + p.frame0 + r) * kHeadDim + e] = y;
        }
    }
    if (EPI == EPI_LOGITS) {
        __syncthreads();
        if (threadIdx.x < RT && row0 + static_cast<int>(threadIdx.x) < n_rows && s_key[threadIdx.x] != 0ull) atomicMax(p.keys + row0 + threadIdx.x, s_key[threadIdx.x]);
    }
}

}  // namespace f32
}  // namespace aed

// Per-step kernels of the AED decoder: row bookkeeping, embedding, attention over ragged caches (single pass; split over
// chunks for the fp32 step with its scratch in the library image), activation planes, argmax finalisation.
#pragma once
#include "common.cuh"

namespace aed {

// ------------------------------------------------------------------------------------------------------------
// Row bookkeeping: compaction of the utterances that take part in the next step, in a fixed visiting order.
//   active_list[r] = utterance id of compact row r;  state->n_active = number of rows.
// An utterance takes part if it is not retired, the caller's mask (if any) selects it, and its self-attention
// cache still has room; a selected utterance with a full cache raises the sticky error instead of overflowing.
// ------------------------------------------------------------------------------------------------------------
// It also fills the row table: row_info[r] = (utterance, t_u, encoder length, encoder offset) for every compact
// row, and utterance -1 for the slots past the last row, so that a kernel needs one 16-byte load per row.
// The batch size is read from the decode state, not passed by value: a captured step graph outlives the batch it
// was recorded for and is replayed for later batches of other sizes.
//
// The greedy loop runs this kernel at the end of every step, with the bookkeeping of the step that ends (kFinish): decode
// the argmax keys, record the token and feed it back, advance t_u, retire finished utterances, and then the rows of the
// next step.  Steps of at most kRowsInside rows find their embedded rows there as well.  These are chains of dependent
// loads of a few hundred cycles each, so what matters is the number of launches in a row: one here, where the end of a
// step, the compaction and the embedding were three, with the boundary between two graphs in the middle.  (4-layer
// model, per step of 1 / 16 rows: 97 / 115 us with three launches, 96 / 116 with this one, 93 / 113 with its loads ahead of the
// wait, 91 / 110 with several steps per graph.)
// Kernels read the row count and the row table ahead of their dependency wait; the one right after this kernel does not,
// and lets its own successor start only after its wait.
constexpr int kRowsInside = 8;       // one block embeds these in less than the 2.8 us of another launch

template <typename T>
struct StepRowsArgs {
    DecState *state;
    const uint8_t *mask;                      // by utterance, or null
    const int32_t *tokens;                    // by utterance: the token that goes into the next step
    int32_t *t_u, *retired, *active_list;
    int max_dec_len;
    const int32_t *enc_len, *enc_off, *order;
    int4 *row_info;
    int row_slots;
    // embedding of up to kRowsInside rows
    const T *embed;
    const float *pe;
    int d, vocab;
    float scale;
    float *x, *zero_buf, *zero_buf2;          // rows that the first projection accumulates into, cleared if not null
    int zero_cols, zero_cols2;
    // kFinish
    unsigned long long *keys;
    int32_t *cur_tok;
    const int32_t *max_len;
    int eos_id;
    volatile int32_t *retired_host;           // with an end-of-sequence id: how many have retired, for the host; or null
    // !kFinish: where the greedy steps to come leave their results, or this step of the caller's loop does
    int32_t *tokens_out, *out_lens;
    float *step_logits;
    int32_t *step_next;
};

// One block of 1024 threads, one utterance per thread and pass.  Everything but the argmax keys is known before the
// dependency wait (only this kernel changes the bookkeeping of greedy steps, and kernels of another kind in between are
// separated by full dependencies): rows of the step that ends, lengths, positions are loaded and computed ahead of it.
// By then the weights of a step have pushed those arrays out of L2, so each is a miss of about 1 us.
template <typename T, bool kFinish>
__global__ void __launch_bounds__(1024) step_rows_kernel(const __grid_constant__ StepRowsArgs<T> a)
{
    AED_TRACE_BEGIN(a.state, 1);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ int counts_old[32], counts_new[32];
    __shared__ int4 first[kRowsInside];       // (utterance, t_u, token) of the first rows
    DecState *const state = a.state;
    const int batch = state->batch, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t *const tokens_out = kFinish ? state->tokens_out : a.tokens_out, *const out_lens = kFinish ? state->out_lens : a.out_lens;
    int u, t, enc_len, enc_off, max_len;
    bool live;                                // takes part unless masked: not retired (and then within its cache)
    auto load = [&](int i) {
        // utterances are visited in the given order (longest encoder output first), so compact rows come out
        // sorted by encoder length: the attention blocks of the longest rows are scheduled first
        live = false;
        u = t = enc_len = enc_off = max_len = 0;
        if (i < batch) {
            u = a.order[i];
            t = a.t_u[u];
            live = a.retired[u] == 0;
            enc_len = a.enc_len[u]; enc_off = a.enc_off[u];
            if (kFinish) max_len = a.max_len[u];
        }
    };
    // rank of this thread among those of the block that satisfy the predicate, and their number (two barriers)
    auto rank = [&](bool yes, int *counts, int &total) {
        const unsigned ballot = __ballot_sync(0xffffffffu, yes);
        if (lane == 0) counts[warp] = __popc(ballot);
        __syncthreads();
        const int count = counts[lane];                   // (32 warps)
        total = static_cast<int>(__reduce_add_sync(0xffffffffu, count));
        return static_cast<int>(__reduce_add_sync(0xffffffffu, lane < warp ? count : 0)) + __popc(ballot & ((1u << lane) - 1u));
    };
    load(threadIdx.x);
    int base_old = 0, base = 0, total = 0, row = 0;
    if (kFinish) {
        row = rank(live && t < a.max_dec_len, counts_old, total);
        if (live && row < kRowsInside)        // the position rows that the next step probably adds
            for (int i = 0; i < a.d; i += 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.pe + (size_t)min(t + 1, a.max_dec_len - 1) * a.d + i));
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!kFinish && threadIdx.x == 0) {
        state->tokens_out = tokens_out; state->out_lens = out_lens;
        state->step_tokens = a.tokens; state->step_logits = a.step_logits; state->step_next = a.step_next;
    }
    for (int start = 0; start < batch; start += blockDim.x) {
        if (start > 0) {
            load(start + threadIdx.x);
            __syncthreads();                  // counts_old, counts_new of the previous pass have been read
            if (kFinish) row = rank(live && t < a.max_dec_len, counts_old, total);
        }
        int tok = 0;
        if (kFinish) {
            row += base_old;
            base_old += total;
            if (live && t < a.max_dec_len) {
                tok = argmax_key_index(a.keys[row]);
                a.keys[row] = 0ull;
                tokens_out[(size_t)u * a.max_dec_len + t] = tok;
                a.t_u[u] = ++t;
                a.cur_tok[u] = tok;
                if (t >= max_len || (a.eos_id >= 0 && tok == a.eos_id)) {
                    live = false;
                    a.retired[u] = 1;
                    out_lens[u] = t;
                    atomicAdd(&state->n_retired, 1);          // the host polls this to stop issuing steps once every utterance is done
                }
            }
        }
        bool take = live && (kFinish || a.mask == nullptr || a.mask[u] != 0);
        if (take && t >= a.max_dec_len) { take = false; atomicExch(&state->error, 1); }
        const int slot = base + rank(take, counts_new, total);
        base += total;
        if (take) {
            a.active_list[slot] = u;
            a.row_info[slot] = make_int4(u, t, enc_len, enc_off);
            if (slot < kRowsInside) first[slot] = make_int4(u, t, min(max(kFinish ? tok : a.tokens[u], 0), a.vocab - 1), 0);
        }
    }
    __syncthreads();
    const int n_rows = base;
    if (threadIdx.x == 0) {
        state->n_active = n_rows;
        if (kFinish && a.retired_host) {
            *a.retired_host = state->n_retired;       // pinned host memory; the host looks at it behind an event
            __threadfence_system();
        }
    }
    for (int r = n_rows + threadIdx.x; r < a.row_slots; r += blockDim.x) a.row_info[r] = make_int4(-1, 0, 0, 0);
    if (n_rows > kRowsInside) return;
    for (int i = threadIdx.x; i < a.d; i += blockDim.x) {
        float e[kRowsInside], pe[kRowsInside];               // (table rows come from DRAM: all of them requested at once)
#pragma unroll
        for (int r = 0; r < kRowsInside; ++r)
            if (r < n_rows) { e[r] = to_f32(a.embed[(size_t)first[r].z * a.d + i]); pe[r] = a.pe[(size_t)first[r].y * a.d + i]; }
#pragma unroll
        for (int r = 0; r < kRowsInside; ++r)
            if (r < n_rows) a.x[(size_t)r * a.d + i] = e[r] * a.scale + pe[r];
    }
    if (a.zero_buf)
        for (int i = threadIdx.x; i < n_rows * a.zero_cols; i += blockDim.x) a.zero_buf[i] = 0.f;
    if (a.zero_buf2)
        for (int i = threadIdx.x; i < n_rows * a.zero_cols2; i += blockDim.x) a.zero_buf2[i] = 0.f;
}

// A new batch: clear the state and the bookkeeping arrays behind it, and note the batch size.  One block.
__global__ void begin_batch_kernel(int4 *region, int n16, DecState *state, int batch)
{
    for (int i = threadIdx.x; i < n16; i += blockDim.x) region[i] = make_int4(0, 0, 0, 0);
    __syncthreads();
    if (threadIdx.x == 0) state->batch = batch;
}

// Start of a greedy decode: the start token into every utterance, empty results.
__global__ void begin_greedy_kernel(int32_t *__restrict__ cur_tok, int bos, int batch, int32_t *__restrict__ tokens_out, size_t n_tokens,
                                    int32_t *__restrict__ out_lens)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n_tokens) tokens_out[i] = -1;
    if (i < (size_t)batch) { cur_tok[i] = bos; out_lens[i] = 0; }
}

// Sinusoidal position table PE[t][2i] = sin(t / 10000^(2i/d)), PE[t][2i+1] = cos(same), evaluated in double.
__global__ void fill_pe_kernel(float *pe, int max_len, int d)
{
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= max_len * d) return;
    int t = idx / d, i = idx % d;
    double angle = static_cast<double>(t) / pow(10000.0, (2.0 * (i / 2)) / static_cast<double>(d));
    pe[idx] = static_cast<float>((i & 1) ? cos(angle) : sin(angle));
}

// x[r] = E[token of utterance] * sqrt(d) + PE[t_u]
template <typename T>
__global__ void embed_kernel(const DecState *state, const int32_t *active_list,
                             const int32_t *tokens, const int32_t *t_u,
                             const T *__restrict__ embed, const float *__restrict__ pe, int d, int vocab, float scale,
                             float *__restrict__ x, float *__restrict__ zero_buf = nullptr, int zero_cols = 0,
                             float *__restrict__ zero_buf2 = nullptr, int zero_cols2 = 0)
{
    AED_TRACE_BEGIN(state, 2);
    // may be launched with programmatic stream serialization, right behind the row compaction
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    int r = blockIdx.x;
    if (r >= state->n_active) return;
    int u = active_list[r];
    int tok = (tokens ? tokens : state->step_tokens)[u];
    tok = min(max(tok, 0), vocab - 1);
    int t = t_u[u];
    for (int i = threadIdx.x; i < d; i += blockDim.x)
        x[(size_t)r * d + i] = to_f32(embed[(size_t)tok * d + i]) * scale + pe[(size_t)t * d + i];
    for (int i = threadIdx.x; i < zero_cols; i += blockDim.x) zero_buf[(size_t)r * zero_cols + i] = 0.f;
    for (int i = threadIdx.x; i < zero_cols2; i += blockDim.x) zero_buf2[(size_t)r * zero_cols2 + i] = 0.f;
}

// ------------------------------------------------------------------------------------------------------------
// Flash-decoding attention over ragged caches.  One warp per (row, head, chunk of 64 positions): lanes are
// 4 position groups x 8 dimension groups, each lane holds 8 of the 64 head dimensions (one 128-bit load of a
// bf16 key or value row segment).  Scores are reduced over the 8 dimension lanes with shuffles, softmax is
// kept online per position group and merged over the 4 groups at the end.  Each work item writes
// (running max, running sum, 64 un-normalised accumulators); the combine kernel merges the chunks of a row.
//   SELF : keys/values of utterance u, head h at  cache[((u*2 + kv)*H + h)*max_len*64],  length t_u + 1
//   CROSS: keys/values at store[(kv*H + h)*capacity*64 + enc_off[u]*64],                 length enc_len[u]
// ------------------------------------------------------------------------------------------------------------
// With kAppend (self-attention after a split-K projection) q, k and v of the new position sit side by side in
// one fp32 row [q | k | v] of `q`; the warp whose chunk holds position t_u first stores k and v into the cache.
template <typename CT, bool kCross, bool kAppend = false>
__global__ void __launch_bounds__(128)
attn_partial_kernel(const DecState *state, const int32_t *__restrict__ active_list, const float *__restrict__ q,
                    int ldq, CT *__restrict__ cache, int n_heads, int seq_capacity,
                    const int32_t *__restrict__ t_u, const int32_t *__restrict__ enc_off,
                    const int32_t *__restrict__ enc_len, int max_chunks, float scale, float *__restrict__ partials)
{
    const int rh = blockIdx.x;
    const int r = rh / n_heads, h = rh % n_heads;
    if (r >= state->n_active) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int chunk = blockIdx.y * 4 + warp;
    const int u = active_list[r];
    const int len = kCross ? enc_len[u] : t_u[u] + 1;
    const int p0 = chunk * kAttnChunk;
    if (chunk >= max_chunks || p0 >= len) return;
    const int p1 = min(len, p0 + kAttnChunk);
    const CT *kbase, *vbase;
    if (kCross) {
        kbase = cache + ((size_t)(0 * n_heads + h) * seq_capacity + enc_off[u]) * kHeadDim;
        vbase = cache + ((size_t)(1 * n_heads + h) * seq_capacity + enc_off[u]) * kHeadDim;
    } else {
        kbase = cache + (((size_t)u * 2 + 0) * n_heads + h) * (size_t)seq_capacity * kHeadDim;
        vbase = cache + (((size_t)u * 2 + 1) * n_heads + h) * (size_t)seq_capacity * kHeadDim;
    }
    const int dg = lane & 7, pg = lane >> 3;
    if (kAppend && !kCross && len - 1 >= p0 && len - 1 < p1) {
        if (lane < 16) {
            const int kv = lane >> 3, d_model = n_heads * kHeadDim;
            float nv[8];
            load8(q + (size_t)r * ldq + (1 + kv) * d_model + h * kHeadDim + dg * 8, nv);
            CT *dst = const_cast<CT *>(kv ? vbase : kbase) + (size_t)(len - 1) * kHeadDim + dg * 8;
#pragma unroll
            for (int i = 0; i < 8; ++i) dst[i] = from_f32<CT>(nv[i]);
        }
        __syncwarp();
    }
    float qv[8];
    load8(q + (size_t)r * ldq + h * kHeadDim + dg * 8, qv);
#pragma unroll
    for (int i = 0; i < 8; ++i) qv[i] *= scale;

    float m = -INFINITY, l = 0.f, acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = 0.f;
    for (int p = p0 + pg; p < p0 + kAttnChunk; p += 4) {   // uniform trip count: shuffles need all lanes
        const bool ok = p < p1;
        float kv[8], s = 0.f;
        if (ok) {
            load8(kbase + (size_t)p * kHeadDim + dg * 8, kv);
#pragma unroll
            for (int i = 0; i < 8; ++i) s = fmaf(qv[i], kv[i], s);
        }
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        s += __shfl_xor_sync(0xffffffffu, s, 4);
        if (ok) {
            float vv[8];
            load8(vbase + (size_t)p * kHeadDim + dg * 8, vv);
            float m_new = fmaxf(m, s);
            float corr = expf(m - m_new), pr = expf(s - m_new);
            l = l * corr + pr;
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] = fmaf(pr, vv[i], acc[i] * corr);
            m = m_new;
        }
    }
    // merge the 4 position groups (lanes differing in bits 3 and 4)
#pragma unroll
    for (int off = 8; off < 32; off <<= 1) {
        float m_o = __shfl_xor_sync(0xffffffffu, m, off);
        float l_o = __shfl_xor_sync(0xffffffffu, l, off);
        float m_new = fmaxf(m, m_o);
        float c_self = (m == -INFINITY) ? 0.f : expf(m - m_new);
        float c_oth = (m_o == -INFINITY) ? 0.f : expf(m_o - m_new);
        l = l * c_self + l_o * c_oth;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float a_o = __shfl_xor_sync(0xffffffffu, acc[i], off);
            acc[i] = acc[i] * c_self + a_o * c_oth;
        }
        m = m_new;
    }
    float *dst = partials + ((size_t)rh * max_chunks + chunk) * kPartialStride;
    if (lane == 0) { dst[0] = m; dst[1] = l; }
    if (pg == 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) dst[2 + dg * 8 + i] = acc[i];
    }
}


// ------------------------------------------------------------------------------------------------------------
// Single-pass attention for one (row, head) per block: no scratch, no second kernel.  Warp w takes the
// 16-position chunks w, w + n_warps, ...; within a chunk every lane issues its 4 key and 4 value loads (128 bits
// each) together, so one memory latency covers the chunk, then reduces the scores with shuffles.
// Warps keep a running (max, sum, accumulator) and are merged through shared memory at the end.
// Lanes: 8 dimension groups (8 head dimensions each) x 4 position groups.
//   kAppend (self-attention): q row is [q | k | v]; k and v of the new position are stored first.
//   Output: fp32 [row, d] (out) and/or bf16 high/low planes (out_hi/out_lo), whichever pointers are non-null.
// ------------------------------------------------------------------------------------------------------------
template <typename CT> struct RawLane;
template <> struct RawLane<__nv_bfloat16> {
    uint4 v;
    __device__ __forceinline__ void load(const __nv_bfloat16 *p) { v = *reinterpret_cast<const uint4 *>(p); }
    __device__ __forceinline__ void zero() { v = make_uint4(0u, 0u, 0u, 0u); }
    __device__ __forceinline__ void set(const float (&f)[8])          // rounds to bf16, as the cache stores it
    {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            __nv_bfloat162 pr = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
            w[i] = *reinterpret_cast<uint32_t *>(&pr);
        }
        v = make_uint4(w[0], w[1], w[2], w[3]);
    }
    __device__ __forceinline__ void store(__nv_bfloat16 *p) const { *reinterpret_cast<uint4 *>(p) = v; }
    __device__ __forceinline__ void get(float (&f)[8]) const
    {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) { f[2 * i] = __uint_as_float(w[i] << 16); f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u); }
    }
};
template <> struct RawLane<fp8e4m3> {
    uint2 v;                                                                   // 8 bytes = 8 values
    __device__ __forceinline__ void load(const fp8e4m3 *p) { v = *reinterpret_cast<const uint2 *>(p); }
    __device__ __forceinline__ void zero() { v = make_uint2(0u, 0u); }
    __device__ __forceinline__ void set(const float (&f)[8])
    {
        v.x = static_cast<uint32_t>(pack_e4m3x2(f[0], f[1])) | (static_cast<uint32_t>(pack_e4m3x2(f[2], f[3])) << 16);
        v.y = static_cast<uint32_t>(pack_e4m3x2(f[4], f[5])) | (static_cast<uint32_t>(pack_e4m3x2(f[6], f[7])) << 16);
    }
    __device__ __forceinline__ void store(fp8e4m3 *p) const { *reinterpret_cast<uint2 *>(p) = v; }
    __device__ __forceinline__ void get(float (&f)[8]) const
    {
        const float2 a = unpack_e4m3x2(static_cast<uint16_t>(v.x & 0xFFFFu)), b = unpack_e4m3x2(static_cast<uint16_t>(v.x >> 16));
        const float2 c = unpack_e4m3x2(static_cast<uint16_t>(v.y & 0xFFFFu)), d = unpack_e4m3x2(static_cast<uint16_t>(v.y >> 16));
        f[0] = a.x; f[1] = a.y; f[2] = b.x; f[3] = b.y; f[4] = c.x; f[5] = c.y; f[6] = d.x; f[7] = d.y;
    }
};
template <> struct RawLane<float> {
    float4 a, b;
    __device__ __forceinline__ void load(const float *p) { a = *reinterpret_cast<const float4 *>(p); b = *reinterpret_cast<const float4 *>(p + 4); }
    __device__ __forceinline__ void zero() { a = make_float4(0.f, 0.f, 0.f, 0.f); b = a; }
    __device__ __forceinline__ void set(const float (&f)[8]) { a = make_float4(f[0], f[1], f[2], f[3]); b = make_float4(f[4], f[5], f[6], f[7]); }
    __device__ __forceinline__ void store(float *p) const { *reinterpret_cast<float4 *>(p) = a; *reinterpret_cast<float4 *>(p + 4) = b; }
    __device__ __forceinline__ void get(float (&f)[8]) const
    { f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w; }
};

// Head dimensions per lane.  8 for every storage type: with single-byte keys and values, 16 per lane (one 16-byte load
// per row and lane, 32 positions per warp and pass) was measured slower at 512 rows (693 against 654 ms per pass of
// the 24-layer batch-512 workload): the kernel is bound by how many loads its resident warps keep in flight, not by
// bytes per load, and the wider lanes cost a resident block per SM.
template <typename CT> struct LaneWidth { static constexpr int kE = 8; };
// positions per warp and iteration: 4 passes over the 32 / (64 / kE) position groups of a warp
template <typename CT> constexpr int fused_chunk() { return 4 * (32 / (kHeadDim / LaneWidth<CT>::kE)); }
constexpr int kFusedMaxWarps = 8;

// Softmax weights of the single-pass attention kernels: scores are in units of ln 2, so a weight is 2^x.  bf16 configuration:
// the hardware approximation (relative error about 2^-22, results below the smallest normal number are 0).  fp32: exp2f, as
// fp32 as everything else there, down to the smallest weights (per step of the 2-layer model at 1 / 4 / 16 / 64 rows 45.8 /
// 52.3 / 74.7 / 95.1 us, with the approximation 45.3 / 51.6 / 74.5 / 93.6, with expf 46.4 / 52.8 / 74.8 / 97.2).
constexpr float kScoreUnit = 1.4426950408889634f;
template <typename CT> __device__ __forceinline__ float softmax_weight(float x)
{
    if constexpr (sizeof(CT) == 4) return exp2f(x);
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <int N> __device__ __forceinline__ void load_n(const float *p, float (&v)[N])
{
#pragma unroll
    for (int i = 0; i < N; i += 4) {
        const float4 a = *reinterpret_cast<const float4 *>(p + i);
        v[i] = a.x; v[i + 1] = a.y; v[i + 2] = a.z; v[i + 3] = a.w;
    }
}

// Sums of a warp's four position groups (lanes dg + 8 pg) of 8 head dimensions each: a lane keeps dimensions 2 pg and 2 pg + 1 of its 8 (6 shuffles
// instead of 16).
__device__ __forceinline__ float2 sum_position_groups(const float (&acc)[8], int pg)
{
    float a4[4], o2[2];
    const bool up = pg & 2, up1 = pg & 1;
#pragma unroll
    for (int j = 0; j < 4; ++j) a4[j] = (up ? acc[4 + j] : acc[j]) + __shfl_xor_sync(0xffffffffu, up ? acc[j] : acc[4 + j], 16);
#pragma unroll
    for (int j = 0; j < 2; ++j) o2[j] = (up1 ? a4[2 + j] : a4[j]) + __shfl_xor_sync(0xffffffffu, up1 ? a4[j] : a4[2 + j], 8);
    return make_float2(o2[0], o2[1]);
}

// kPipe: the loads of a warp's next chunk are issued before the current chunk is reduced (twice the K/V registers,
// so only two blocks per SM: for grids that fit anyway).
// kRowStats: the block computes (mean, rstd) of its row of stats_x itself instead of reading ln_stats.
template <typename CT, bool kCross, bool kAppend, bool kPipe = false, bool kRowStats = false>
__global__ void __launch_bounds__(kFusedMaxWarps * 32, sizeof(CT) == 4 ? 1 : ((kAppend || kPipe) ? 2 : (LaneWidth<CT>::kE > 8 ? 3 : 4)))      // self-attention holds the new key/value as well; wider lanes and fp32 need more registers
attn_fused_kernel(const DecState *state, const int4 *row_info, const float *q, int ldq,
                  CT *__restrict__ cache, int n_heads, int seq_capacity, float scale,
                  float *__restrict__ out, __nv_bfloat16 *__restrict__ out_hi, __nv_bfloat16 *__restrict__ out_lo, int ldo,
                  const float2 *ln_stats, const float *__restrict__ ln_c1, const float *__restrict__ ln_c2,
                  const float *stats_x = nullptr, float ln_eps = 0.f)
{
    // (What earlier kernels of the step write is not __restrict__: this kernel is resident before they have finished, and loads
    // through the read-only path may return what their lines held then.)
    // stats_x: rows [*, heads * 64] whose (mean, rstd) this block computes itself instead of reading ln_stats (the
    // kernel before this one completed those rows, so nobody could have computed the statistics earlier).
    // Launched with programmatic stream serialization.  Before the dependency wait only data that no kernel of
    // this step writes is touched: the row table (written by the step's first kernel, which ran to completion
    // before any programmatic launch of the step) and, for cross-attention, the encoder K/V store.
    __shared__ float sm_m[kFusedMaxWarps], sm_l[kFusedMaxWarps];
    __shared__ __align__(8) float sm_acc[kFusedMaxWarps][kHeadDim];
    __shared__ float2 sm_red[kFusedMaxWarps];
    const int rh = blockIdx.x;
    const int r = rh / n_heads, h = rh % n_heads;
    const int4 ri = row_info[r];                       // (utterance, t_u, encoder length, encoder offset)
    // The next kernel may start at once where that is a few-row projection, so that its weights are on their way while this
    // one still waits (24 layers, 4 / 8 / 24 rows: 499 / 513 / 681 -> 473 / 486 / 661 us per step).  It starts when every block has
    // called it or ended, so the blocks of padding rows, which end only after the wait, call it as well (1 / 2 / 7 / 9 / 12 rows in
    // grids of 4 / 4 / 8 / 16 / 16: 455 / 470 / 506 / 523 / 533 -> 442 / 449 / 492 / 503 / 515).  Not the cross-attention of
    // steps with more than 128 rows, which read their statistics (no kRowStats): blocks of the next kernel would take room from
    // its own later ones (200 / 512 rows 2130 / 3488 -> 2224 / 3650).  Nor fp32, whose projections hold their weights in
    // registers (2 layers, 4 / 8 rows: 54 / 70 us per step against 59 / 75).
    constexpr bool kEarly = sizeof(CT) < 4 && (!kCross || kRowStats);
    if (kEarly) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (ri.x < 0) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;
    const int u = ri.x;
    const int len = kCross ? ri.z : ri.y + 1;
    const CT *kbase, *vbase;
    if (kCross) {
        kbase = cache + ((size_t)(0 * n_heads + h) * seq_capacity + ri.w) * kHeadDim;
        vbase = cache + ((size_t)(1 * n_heads + h) * seq_capacity + ri.w) * kHeadDim;
    } else {
        kbase = cache + (((size_t)u * 2 + 0) * n_heads + h) * (size_t)seq_capacity * kHeadDim;
        vbase = cache + (((size_t)u * 2 + 1) * n_heads + h) * (size_t)seq_capacity * kHeadDim;
    }
    // Positions that earlier steps (or the precompute) wrote are static for this kernel; the position appended
    // by this step (self-attention only) is taken from the projection output after the dependency wait.
    const int len_static = (kAppend && !kCross) ? len - 1 : len;
    constexpr int kE = LaneWidth<CT>::kE, kDG = kHeadDim / kE, kPG = 32 / kDG, kChunk = 4 * kPG;
    const int dg = lane % kDG, pg = lane / kDG;      // lanes: kDG groups of kE head dimensions x kPG positions
    RawLane<CT> rk[4], rv[4];
    // Self-attention without an append of its own (prefill pass): the cache positions it reads are written by the
    // kernel before it, so nothing is loaded ahead of the dependency wait.
    if (!kCross && !kAppend) asm volatile("griddepcontrol.wait;" ::: "memory");
    {
        // This warp's first chunk starts streaming while the kernel that produces the query is still running.
        const int p0 = warp * kChunk;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int p = p0 + i * kPG + pg;
            if (p < len_static) {
                rk[i].load(kbase + (size_t)p * kHeadDim + dg * kE);
                rv[i].load(vbase + (size_t)p * kHeadDim + dg * kE);
            } else { rk[i].zero(); rv[i].zero(); }
        }
        // later chunks of this warp: pull them into L2 now (one 128-byte row per lane group)
        if (dg == 0) {
#pragma unroll 1
            for (int q0 = p0 + n_warps * kChunk; q0 < len_static; q0 += n_warps * kChunk) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int p = q0 + i * kPG + pg;
                    if (p < len_static) {
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(kbase + (size_t)p * kHeadDim));
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(vbase + (size_t)p * kHeadDim));
                    }
                }
            }
        }
    }
    // The LayerNorm-fold constants of this block's columns are static as well (read once per step and layer, so
    // they come from DRAM): requested here, before the dependency wait.
    const int new_chunk = (len - 1) / kChunk;
    const bool owns_new = kAppend && !kCross && warp == new_chunk % n_warps;
    const int d_model = n_heads * kHeadDim;
    const int qcol = h * kHeadDim + dg * kE;
    float qc1[kE], qc2[kE], kc1[kE], kc2[kE], vc1[kE], vc2[kE];
    const bool fold = ln_stats != nullptr || kRowStats;
    if (fold) {
        load_n<kE>(ln_c1 + qcol, qc1); load_n<kE>(ln_c2 + qcol, qc2);
        if (owns_new) {
            load_n<kE>(ln_c1 + d_model + qcol, kc1); load_n<kE>(ln_c2 + d_model + qcol, kc2);
            load_n<kE>(ln_c1 + 2 * d_model + qcol, vc1); load_n<kE>(ln_c2 + 2 * d_model + qcol, vc2);
        }
    }
    AED_TRACE_RESERVE(tcur, state, (threadIdx.x == 0 && blockIdx.x == 0) ? 6u : 0u);
    AED_TRACE_PUT_NS(state, tcur, 8 + (kCross ? 1 : 0));      // resident, first chunk requested
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!kEarly) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    AED_TRACE_PUT(state, tcur, 3);                          // dependency resolved
    // Everything this block needs from earlier kernels is requested in one round: statistics, query, and (in the
    // warp that owns the new position) the new key and value.  When the projection ran on gamma*x, its raw output
    // y becomes rstd*(y - mean*c1) + c2 here.
    float2 st = make_float2(0.f, 1.f);
    float qv[kE], kn[kE], vn[kE];
    if (ln_stats) st = ln_stats[r];
    load_n<kE>(q + (size_t)r * ldq + qcol, qv);
    if (owns_new) {
        load_n<kE>(q + (size_t)r * ldq + d_model + qcol, kn);
        load_n<kE>(q + (size_t)r * ldq + 2 * d_model + qcol, vn);
    }
    if (kRowStats) {
        // mean and rstd of row r in one pass over deviations from the row's first element (a row whose mean is far
        // from zero loses nothing to cancellation that way): var = (S2 - S1^2 / n) / n, mean = x0 + S1 / n
        const float *xr = stats_x + (size_t)r * d_model;
        const float x0 = xr[0];
        float s1 = 0.f, s2 = 0.f;
        for (int idx = threadIdx.x * 4; idx < d_model; idx += blockDim.x * 4) {
            const float4 v = *reinterpret_cast<const float4 *>(xr + idx);
            const float d0 = v.x - x0, d1 = v.y - x0, d2 = v.z - x0, d3 = v.w - x0;
            s1 += (d0 + d1) + (d2 + d3);
            s2 += (d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3);
        }
        s1 = warp_sum(s1);
        s2 = warp_sum(s2);
        if (lane == 0) sm_red[warp] = make_float2(s1, s2);
        __syncthreads();
        float t1 = 0.f, t2 = 0.f;
#pragma unroll
        for (int w = 0; w < kFusedMaxWarps; ++w)
            if (w < n_warps) { t1 += sm_red[w].x; t2 += sm_red[w].y; }
        const float inv_n = 1.f / d_model;
        const float var = fmaxf((t2 - t1 * t1 * inv_n) * inv_n, 0.f);
        st = make_float2(x0 + t1 * inv_n, rsqrtf(var + ln_eps));
    }
    if (fold) {
#pragma unroll
        for (int i = 0; i < kE; ++i) qv[i] = fmaf(st.y, qv[i] - st.x * qc1[i], qc2[i]);
    }
#pragma unroll
    for (int i = 0; i < kE; ++i) qv[i] *= scale * kScoreUnit;
    RawLane<CT> new_k, new_v;
    if (owns_new) {
        if (fold) {
#pragma unroll
            for (int i = 0; i < kE; ++i) {
                kn[i] = fmaf(st.y, kn[i] - st.x * kc1[i], kc2[i]);
                vn[i] = fmaf(st.y, vn[i] - st.x * vc1[i], vc2[i]);
            }
        }
        new_k.set(kn);
        new_v.set(vn);
        if (pg == 0) {      // append to the cache; no other block reads this position during the kernel
            new_k.store(const_cast<CT *>(kbase) + (size_t)(len - 1) * kHeadDim + dg * kE);
            new_v.store(const_cast<CT *>(vbase) + (size_t)(len - 1) * kHeadDim + dg * kE);
        }
    }

    AED_TRACE_PUT(state, tcur, 4);                          // query ready (statistics, fold)
    float m = -INFINITY, l = 0.f, acc[kE];
#pragma unroll
    for (int i = 0; i < kE; ++i) acc[i] = 0.f;
    bool loaded = true;
    RawLane<CT> nk[4], nv[4];
    for (int p0 = warp * kChunk; p0 < len; p0 += n_warps * kChunk) {
        if (kPipe) {
            const int pn = p0 + n_warps * kChunk;
            if (pn < len) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int p = pn + i * kPG + pg;
                    if (p < len_static) {
                        nk[i].load(kbase + (size_t)p * kHeadDim + dg * kE);
                        nv[i].load(vbase + (size_t)p * kHeadDim + dg * kE);
                    } else { nk[i].zero(); nv[i].zero(); }
                }
            }
        } else if (!loaded) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {          // keys and values of the chunk are requested together
                const int p = p0 + i * kPG + pg;
                if (p < len_static) {
                    rk[i].load(kbase + (size_t)p * kHeadDim + dg * kE);
                    rv[i].load(vbase + (size_t)p * kHeadDim + dg * kE);
                } else { rk[i].zero(); rv[i].zero(); }
            }
        }
        loaded = false;
        if (owns_new && p0 == new_chunk * kChunk) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (p0 + i * kPG + pg == len - 1) { rk[i] = new_k; rv[i] = new_v; }
        }
        float s[4], cmax = -INFINITY;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float kf[kE], d = 0.f;
            rk[i].get(kf);
#pragma unroll
            for (int j = 0; j < kE; ++j) d = fmaf(qv[j], kf[j], d);
#pragma unroll
            for (int o = 1; o < kDG; o <<= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
            s[i] = (p0 + i * kPG + pg < len) ? d : -INFINITY;
            cmax = fmaxf(cmax, s[i]);
        }
#pragma unroll
        for (int o = kDG; o < 32; o <<= 1) cmax = fmaxf(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));     // chunk max, uniform over the warp, finite
        const float m_new = fmaxf(m, cmax);
        const float corr = softmax_weight<CT>(m - m_new);
        l *= corr;
#pragma unroll
        for (int j = 0; j < kE; ++j) acc[j] *= corr;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float pr = softmax_weight<CT>(s[i] - m_new);      // 0 for positions past the end
            float vf[kE];
            rv[i].get(vf);
            l += pr;
#pragma unroll
            for (int j = 0; j < kE; ++j) acc[j] = fmaf(pr, vf[j], acc[j]);
        }
        m = m_new;
        if (kPipe) {
#pragma unroll
            for (int i = 0; i < 4; ++i) { rk[i] = nk[i]; rv[i] = nv[i]; }
        }
    }
    AED_TRACE_PUT(state, tcur, 5);                          // all chunks of this warp reduced
    // sum the position groups (they share m)
    static_assert(kE == 8 && kPG == 4, "as sum_position_groups has it");
    l += __shfl_xor_sync(0xffffffffu, l, 8);
    l += __shfl_xor_sync(0xffffffffu, l, 16);
    if (lane == 0) { sm_m[warp] = m; sm_l[warp] = l; }
    *reinterpret_cast<float2 *>(&sm_acc[warp][dg * 8 + pg * 2]) = sum_position_groups(acc, pg);
    __syncthreads();
    if (threadIdx.x < kHeadDim) {
        // Unrolled, so that all warps' results are loaded at once (24 layers, 8 / 64 rows, with the same above: 8 / 7 us a step).  fp32,
        // whose weights take many instructions, is left alone (2 layers, 1 row: 45.7 us a step, unrolled 46.6).
        float lsum = 0.f, a = 0.f;
        if constexpr (sizeof(CT) < 4) {
            float mw[kFusedMaxWarps], big = -INFINITY;
#pragma unroll
            for (int w = 0; w < kFusedMaxWarps; ++w) {
                mw[w] = w < n_warps ? sm_m[w] : -INFINITY;
                big = fmaxf(big, mw[w]);
            }
#pragma unroll
            for (int w = 0; w < kFusedMaxWarps; ++w) {
                if (w >= n_warps) continue;
                const float wgt = (mw[w] == -INFINITY) ? 0.f : softmax_weight<CT>(mw[w] - big);
                lsum = fmaf(sm_l[w], wgt, lsum);
                a = fmaf(sm_acc[w][threadIdx.x], wgt, a);
            }
        } else {
            float big = -INFINITY;
            for (int w = 0; w < n_warps; ++w) big = fmaxf(big, sm_m[w]);
            for (int w = 0; w < n_warps; ++w) {
                const float wgt = (sm_m[w] == -INFINITY) ? 0.f : softmax_weight<CT>(sm_m[w] - big);
                lsum = fmaf(sm_l[w], wgt, lsum);
                a = fmaf(sm_acc[w][threadIdx.x], wgt, a);
            }
        }
        const float o = a / lsum;
        const size_t off = (size_t)r * ldo + h * kHeadDim + threadIdx.x;
        if (out) out[off] = o;
        if (out_hi) {
            const __nv_bfloat16 hi = __float2bfloat16_rn(o);
            out_hi[off] = hi;
            out_lo[off] = __float2bfloat16_rn(o - __bfloat162float(hi));
        }
    }
    AED_TRACE_PUT_NS(state, tcur, 7);                       // output written
}

// Self-attention of many rows: one warp per (row, head), 8 pairs per block, no shared memory and no merge of warps.
// Short caches make this a matter of latency (the dependency wait, then one round of loads and a chain of shuffles), so
// what counts is how many pairs an SM holds at once: 24 warps of at most 85 registers.  A pair's later chunks are loaded
// one after the other; 24 x 4 KB in flight per SM are enough for long caches (512 rows, positions 221 to 240: 483 MB in 93.5 us
// by events, 5.2 TB/s; 129 rows 4.1).  What it gained per step stands at its launch.  The next kernel starts after the wait
// here, unlike behind attn_fused_kernel: steps of 65 to 128 rows (16 heads) have early starts behind cross-attention only.
template <typename CT, bool kAppend>
__global__ void __launch_bounds__(256, 3)
self_attn_warp_kernel(const DecState *state, const int4 *row_info, const float *q, int ldq,
                      CT *__restrict__ cache, int n_heads, int seq_capacity, float scale, float *__restrict__ out,
                      __nv_bfloat16 *__restrict__ out_hi, __nv_bfloat16 *__restrict__ out_lo, int ldo,
                      const float2 *ln_stats, const float *__restrict__ ln_c1, const float *__restrict__ ln_c2, int row_heads)
{
    constexpr int kE = LaneWidth<CT>::kE, kDG = kHeadDim / kE, kPG = 32 / kDG, kChunk = 4 * kPG;
    const int lane = threadIdx.x & 31, rh = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int r = rh / n_heads, h = rh - r * n_heads;
    const int4 ri = rh < row_heads ? row_info[r] : make_int4(-1, 0, 0, 0);
    const int len = ri.y + 1, len_static = kAppend ? len - 1 : len;
    const int dg = lane % kDG, pg = lane / kDG, qcol = h * kHeadDim + dg * kE, d_model = n_heads * kHeadDim;
    CT *const kbase = cache + ((size_t)max(ri.x, 0) * 2 * n_heads + h) * (size_t)seq_capacity * kHeadDim + dg * kE;
    CT *const vbase = kbase + (size_t)n_heads * seq_capacity * kHeadDim;
    RawLane<CT> rk[4], rv[4];
    auto load_chunk = [&](int p0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int p = p0 + i * kPG + pg;
            if (p < len_static) { rk[i].load(kbase + (size_t)p * kHeadDim); rv[i].load(vbase + (size_t)p * kHeadDim); }
            else { rk[i].zero(); rv[i].zero(); }
        }
    };
    if (kAppend && ri.x >= 0) load_chunk(0);            // positions of earlier steps: before the dependency wait
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (ri.x < 0) return;
    if (!kAppend) load_chunk(0);
    const float2 st = ln_stats[r];
    const float *const qr = q + (size_t)r * ldq + qcol;
    float qv[kE];
    RawLane<CT> new_k, new_v;
    {
        float y[3][kE], c1[kE], c2[kE];
#pragma unroll
        for (int j = 0; j < (kAppend ? 3 : 1); ++j) load_n<kE>(qr + j * d_model, y[j]);
#pragma unroll
        for (int j = 0; j < (kAppend ? 3 : 1); ++j) {
            load_n<kE>(ln_c1 + j * d_model + qcol, c1);
            load_n<kE>(ln_c2 + j * d_model + qcol, c2);
#pragma unroll
            for (int i = 0; i < kE; ++i) y[j][i] = fmaf(st.y, y[j][i] - st.x * c1[i], c2[i]);
        }
#pragma unroll
        for (int i = 0; i < kE; ++i) qv[i] = y[0][i] * (scale * kScoreUnit);
        if (kAppend) {
            new_k.set(y[1]);
            new_v.set(y[2]);
            if (pg == 0) {
                new_k.store(kbase + (size_t)(len - 1) * kHeadDim);
                new_v.store(vbase + (size_t)(len - 1) * kHeadDim);
            }
        }
    }
    float m = -INFINITY, l = 0.f, acc[kE];
#pragma unroll
    for (int i = 0; i < kE; ++i) acc[i] = 0.f;
    for (int p0 = 0; p0 < len; p0 += kChunk) {
        if (p0) load_chunk(p0);
        float s[4], cmax = -INFINITY;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int p = p0 + i * kPG + pg;
            if (kAppend && p == len - 1) { rk[i] = new_k; rv[i] = new_v; }
            float kf[kE], d = 0.f;
            rk[i].get(kf);
#pragma unroll
            for (int j = 0; j < kE; ++j) d = fmaf(qv[j], kf[j], d);
#pragma unroll
            for (int o = 1; o < kDG; o <<= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
            s[i] = p < len ? d : -INFINITY;
            cmax = fmaxf(cmax, s[i]);
        }
#pragma unroll
        for (int o = kDG; o < 32; o <<= 1) cmax = fmaxf(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));
        const float m_new = fmaxf(m, cmax), corr = softmax_weight<CT>(m - m_new);
        l *= corr;
#pragma unroll
        for (int j = 0; j < kE; ++j) acc[j] *= corr;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float pr = softmax_weight<CT>(s[i] - m_new);
            float vf[kE];
            rv[i].get(vf);
            l += pr;
#pragma unroll
            for (int j = 0; j < kE; ++j) acc[j] = fmaf(pr, vf[j], acc[j]);
        }
        m = m_new;
    }
    // sum the position groups: every lane keeps 2 of its 8 dimensions, so the groups write one row together
    static_assert(kE == 8 && kPG == 4, "as sum_position_groups has it");
    l += __shfl_xor_sync(0xffffffffu, l, kDG);
    l += __shfl_xor_sync(0xffffffffu, l, 2 * kDG);
    float2 o2 = sum_position_groups(acc, pg);
    const float inv = 1.f / l;
    o2.x *= inv; o2.y *= inv;
    const size_t off = (size_t)r * ldo + qcol + pg * 2;
    if (out) *reinterpret_cast<float2 *>(out + off) = o2;
    if (out_hi) {
        const __nv_bfloat162 hi = __floats2bfloat162_rn(o2.x, o2.y);
        *reinterpret_cast<__nv_bfloat162 *>(out_hi + off) = hi;
        *reinterpret_cast<__nv_bfloat162 *>(out_lo + off) = __floats2bfloat162_rn(o2.x - __bfloat162float(hi.x), o2.y - __bfloat162float(hi.y));
    }
}

// Merge the chunk partials of each (row, head): one warp per pair, 2 head dimensions per lane.
template <bool kCross>
__global__ void __launch_bounds__(128)
attn_combine_kernel(const DecState *state, const int32_t *__restrict__ active_list, const float *__restrict__ partials,
                    int n_heads, const int32_t *__restrict__ t_u, const int32_t *__restrict__ enc_len, int max_chunks,
                    float *__restrict__ out, int ldo)
{
    const int rh = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int r = rh / n_heads, h = rh % n_heads;
    if (r >= state->n_active) return;
    const int u = active_list[r];
    const int len = kCross ? enc_len[u] : t_u[u] + 1;
    const int n_chunks = (len + kAttnChunk - 1) / kAttnChunk;
    const float *src = partials + (size_t)rh * max_chunks * kPartialStride;
    float m = -INFINITY;
    for (int c = 0; c < n_chunks; ++c) m = fmaxf(m, src[(size_t)c * kPartialStride]);
    float l = 0.f, a0 = 0.f, a1 = 0.f;
    for (int c = 0; c < n_chunks; ++c) {
        const float *p = src + (size_t)c * kPartialStride;
        float w = expf(p[0] - m);
        l = fmaf(p[1], w, l);
        a0 = fmaf(p[2 + lane * 2], w, a0);
        a1 = fmaf(p[3 + lane * 2], w, a1);
    }
    float inv = 1.f / l;
    float2 o = make_float2(a0 * inv, a1 * inv);
    *reinterpret_cast<float2 *>(out + (size_t)r * ldo + h * kHeadDim + lane * 2) = o;
}

// A block's row of d values (a multiple of 64, at most 8 per thread), 4 consecutive ones per thread and piece: (mean, rstd) with one
// barrier per sum.  sums: two floats per warp.
constexpr int kRowPieces = 2;
__device__ __forceinline__ float2 block_row_stats(const float4 (&v)[kRowPieces], int d, float eps, float (*sums)[32])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    auto total = [&](float x, float *red) {
        x = warp_sum(x);
        if (lane == 0) red[warp] = x;
        __syncthreads();
        return warp_sum(lane < n_warps ? red[lane] : 0.f);
    };
    float s = 0.f, q = 0.f;
#pragma unroll
    for (int i = 0; i < kRowPieces; ++i) s += (v[i].x + v[i].y) + (v[i].z + v[i].w);
    const float mean = total(s, sums[0]) / d;
#pragma unroll
    for (int i = 0; i < kRowPieces; ++i) {
        const float d0 = v[i].x - mean, d1 = v[i].y - mean, d2 = v[i].z - mean, d3 = v[i].w - mean;
        if (static_cast<int>(threadIdx.x + i * blockDim.x) * 4 < d) q += (d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3);
    }
    return make_float2(mean, rsqrtf(total(q, sums[1]) / d + eps));
}
// four values -> the planes
__device__ __forceinline__ void store_planes(__nv_bfloat16 *hi, __nv_bfloat16 *lo, const float (&y)[4])
{
    uint32_t h[2], l[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(y[2 * j], y[2 * j + 1]);
        const __nv_bfloat162 b = __floats2bfloat162_rn(y[2 * j] - __bfloat162float(a.x), y[2 * j + 1] - __bfloat162float(a.y));
        h[j] = *reinterpret_cast<const uint32_t *>(&a);
        l[j] = *reinterpret_cast<const uint32_t *>(&b);
    }
    *reinterpret_cast<uint2 *>(hi) = make_uint2(h[0], h[1]);
    *reinterpret_cast<uint2 *>(lo) = make_uint2(l[0], l[1]);
}

// LayerNorm whose result is written as bf16 high and low planes [row, d].  One block per row.
__global__ void layernorm_planes_kernel(const DecState *state, const float *x, const __nv_bfloat16 *__restrict__ g, const __nv_bfloat16 *__restrict__ b, int d,
                                        float eps, __nv_bfloat16 *__restrict__ out_hi, __nv_bfloat16 *__restrict__ out_lo)
{
    AED_TRACE_BEGIN(state, 4);
    __shared__ float sums[2][32];
    // gain and bias are static and come from DRAM: ahead of the wait (programmatic stream serialization; nothing of the previous kernel is)
    float4 v[kRowPieces];
    float gk[kRowPieces][4], bk[kRowPieces][4];
#pragma unroll
    for (int i = 0; i < kRowPieces; ++i) {
        const int k = static_cast<int>(threadIdx.x + i * blockDim.x) * 4;
#pragma unroll
        for (int j = 0; j < 4; ++j) { gk[i][j] = k < d ? to_f32(g[k + j]) : 0.f; bk[i][j] = k < d ? to_f32(b[k + j]) : 0.f; }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int r = blockIdx.x;
    if (r >= state->n_active) return;
#pragma unroll
    for (int i = 0; i < kRowPieces; ++i) {
        const int k = static_cast<int>(threadIdx.x + i * blockDim.x) * 4;
        v[i] = k < d ? *reinterpret_cast<const float4 *>(x + (size_t)r * d + k) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const float2 st = block_row_stats(v, d, eps, sums);
#pragma unroll
    for (int i = 0; i < kRowPieces; ++i) {
        const int k = static_cast<int>(threadIdx.x + i * blockDim.x) * 4;
        if (k >= d) continue;
        const float y[4] = {gk[i][0] * (v[i].x - st.x) * st.y + bk[i][0], gk[i][1] * (v[i].y - st.x) * st.y + bk[i][1],
                            gk[i][2] * (v[i].z - st.x) * st.y + bk[i][2], gk[i][3] * (v[i].w - st.x) * st.y + bk[i][3]};
        store_planes(out_hi + (size_t)r * d + k, out_lo + (size_t)r * d + k, y);
    }
}

// ------------------------------------------------------------------------------------------------------------
// Activation planes for steps with many rows.  There the projections fetch their activation operand ready-made
// (bf16 high plane + bf16 low plane = value - high) instead of converting it in every feature tile.
// Both kernels start with a programmatic-dependency wait and may be launched ahead of their predecessor's end.
// ------------------------------------------------------------------------------------------------------------
// planes of gamma * x, the LayerNorm statistics (mean, rstd) of every row, and the clearing of the fp32 rows a later
// split-K projection accumulates into (zero_cols columns of zero_buf, if any).  One block per row.  (A warp per row, without
// barriers, was slower: 200 rows 1980 us per step of the 24-layer model against 1850.)
__global__ void gamma_planes_kernel(const DecState *state, const float *x, const __nv_bfloat16 *__restrict__ g, int d, float eps, float2 *__restrict__ stats_out,
                                    __nv_bfloat16 *__restrict__ out_hi, __nv_bfloat16 *__restrict__ out_lo, float *__restrict__ zero_buf, int zero_cols)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ float sums[2][32];
    float4 v[kRowPieces];
    float gk[kRowPieces][4];                              // (static, and from DRAM: ahead of the wait)
#pragma unroll
    for (int i = 0; i < kRowPieces; ++i) {
        const int k = static_cast<int>(threadIdx.x + i * blockDim.x) * 4;
#pragma unroll
        for (int j = 0; j < 4; ++j) gk[i][j] = k < d ? to_f32(g[k + j]) : 0.f;
    }
    const int r = blockIdx.x;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (r >= state->n_active) return;
#pragma unroll
    for (int i = 0; i < kRowPieces; ++i) {
        const int k = static_cast<int>(threadIdx.x + i * blockDim.x) * 4;
        v[i] = k < d ? *reinterpret_cast<const float4 *>(x + (size_t)r * d + k) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (zero_buf) {
        float4 *const z = reinterpret_cast<float4 *>(zero_buf + (size_t)r * zero_cols);
        for (int i = threadIdx.x; i < zero_cols / 4; i += blockDim.x) z[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int i = 0; i < kRowPieces; ++i) {
        const int k = static_cast<int>(threadIdx.x + i * blockDim.x) * 4;
        if (k >= d) continue;
        const float y[4] = {gk[i][0] * v[i].x, gk[i][1] * v[i].y, gk[i][2] * v[i].z, gk[i][3] * v[i].w};
        store_planes(out_hi + (size_t)r * d + k, out_lo + (size_t)r * d + k, y);
    }
    const float2 st = block_row_stats(v, d, eps, sums);
    if (threadIdx.x == 0) stats_out[r] = st;
}

// ------------------------------------------------------------------------------------------------------------
// Prompt prefill: several positions of every utterance in one pass.  A compact row is an (utterance, position)
// pair; a chunk covers `chunk` consecutive positions of every utterance of the batch.  Rows are ordered position
// major with the chunk's last position first (row = (chunk - 1 - j) * batch + i), so that the rows of the last
// position, the only ones whose logits matter, are rows 0 .. batch - 1.
// ------------------------------------------------------------------------------------------------------------
__global__ void build_prefill_rows_kernel(DecState *state, int chunk, int j0, int prompt_len, const int32_t *__restrict__ prompt,
                                          const int32_t *__restrict__ t_u, const int32_t *__restrict__ enc_len,
                                          const int32_t *__restrict__ enc_off, const int32_t *__restrict__ order,
                                          int32_t *__restrict__ active_list, int4 *__restrict__ row_info,
                                          int32_t *__restrict__ row_tok, int row_slots)
{
    const int batch = state->batch, rows = batch * chunk;
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < row_slots; r += gridDim.x * blockDim.x) {
        if (r < rows) {
            const int u = order[r % batch], j = chunk - 1 - r / batch;
            active_list[r] = u;
            row_info[r] = make_int4(u, t_u[u] + j, enc_len[u], enc_off[u]);
            row_tok[r] = prompt[(size_t)u * prompt_len + j0 + j];
        } else {
            row_info[r] = make_int4(-1, 0, 0, 0);
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) state->n_active = rows;
}

// x[r] = E[token of the row] * sqrt(d) + PE[position of the row]
template <typename T>
__global__ void embed_rows_kernel(const DecState *state, const int4 *__restrict__ row_info, const int32_t *__restrict__ row_tok,
                                  const T *__restrict__ embed, const float *__restrict__ pe, int d, int vocab, float scale,
                                  float *__restrict__ x, float *__restrict__ zero_buf, int zero_cols,
                                  float *__restrict__ zero_buf2 = nullptr, int zero_cols2 = 0)
{
    const int r = blockIdx.x;
    if (r >= state->n_active) return;
    const int tok = min(max(row_tok[r], 0), vocab - 1), t = row_info[r].y;
    for (int i = threadIdx.x; i < d; i += blockDim.x)
        x[(size_t)r * d + i] = to_f32(embed[(size_t)tok * d + i]) * scale + pe[(size_t)t * d + i];
    for (int i = threadIdx.x; i < zero_cols; i += blockDim.x) zero_buf[(size_t)r * zero_cols + i] = 0.f;
    for (int i = threadIdx.x; i < zero_cols2; i += blockDim.x) zero_buf2[(size_t)r * zero_cols2 + i] = 0.f;
}

// Keys and values of every row into the self-attention cache (raw projection output with the LayerNorm fold applied,
// rounded as the cache stores it), before any row attends: in a prefill pass a row reads positions that other rows of
// the same pass append.  grid: rows; a thread takes 8 components at a time.  (With a block of 64 threads per row and head, one component each,
// 333 rows took 7.7 us a launch on its own.)
template <typename CT>
__global__ void __launch_bounds__(256)
append_kv_kernel(const DecState *state, const int4 *row_info, const float *qkv, int ldq, CT *__restrict__ cache, int n_heads, int seq_capacity,
                 const float2 *ln_stats, const float *__restrict__ ln_c1, const float *__restrict__ ln_c2)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int r = blockIdx.x, d_model = n_heads * kHeadDim;
    const int4 ri = row_info[r];
    if (ri.x < 0) return;
    const float2 st = ln_stats[r];
    for (int i = threadIdx.x * 8; i < 2 * d_model; i += blockDim.x * 8) {
        const int kv = i >= d_model, c = i - kv * d_model, col = d_model + i;
        float y[8], c1[8], c2[8];
        load8(qkv + (size_t)r * ldq + col, y);
        load8(ln_c1 + col, c1);
        load8(ln_c2 + col, c2);
#pragma unroll
        for (int e = 0; e < 8; ++e) y[e] = fmaf(st.y, y[e] - st.x * c1[e], c2[e]);
        RawLane<CT> out;
        out.set(y);
        out.store(cache + ((((size_t)ri.x * 2 + kv) * n_heads + c / kHeadDim) * (size_t)seq_capacity + ri.y) * kHeadDim + c % kHeadDim);
    }
}

// Cross-attention of a prefill pass of many rows: a block takes kPrompt positions of one utterance and head, which read the same keys and
// values, so that a chunk of them is loaded and unpacked once for all.  Otherwise as attn_fused_kernel with statistics from ln_stats and planes for output: warps take 16
// positions of the store at a time, one pass, merged through shared memory.  What bounds it is instructions (dot products and their shuffles, weights) at four
// warps per scheduler of 128 registers; with 8 warps per block, as a row alone has them, most have one chunk or none and the block is start and
// merge (37 x 9 positions at 110 frames 2306 us a prefill of 24 layers instead of 2155).  Where it is used, and what it gained, stands at its launch.
// grid: x = utterances * heads, y = groups of kPrompt positions; up to kFusedMaxWarps warps.  Position j of utterance i is row j * batch + i.
constexpr int kPrompt = 4;
template <typename CT>
__global__ void __launch_bounds__(256, 2)
prompt_cross_kernel(const int4 *row_info, const float *q, int ldq, const CT *__restrict__ cache, int n_heads, int seq_capacity, float scale,
                    __nv_bfloat16 *__restrict__ out_hi, __nv_bfloat16 *__restrict__ out_lo, int ldo, const float2 *ln_stats, const float *__restrict__ ln_c1,
                    const float *__restrict__ ln_c2, int batch, int chunk)
{
    constexpr int kWarps = kFusedMaxWarps;
    const int n_warps = blockDim.x >> 5, step = n_warps * 16;
    __shared__ float sm_m[kPrompt][kWarps], sm_l[kPrompt][kWarps];
    __shared__ __align__(8) float sm_acc[kPrompt][kWarps][kHeadDim];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, dg = lane & 7, pg = lane >> 3;
    const int utt = blockIdx.x / n_heads, h = blockIdx.x - utt * n_heads, j0 = blockIdx.y * kPrompt, n = min(chunk - j0, kPrompt);
    const int4 ri = row_info[utt];                     // (of its first row; the others have the same encoder output)
    const int len = ri.z, qcol = h * kHeadDim + dg * 8;
    const CT *const kbase = cache + ((size_t)h * seq_capacity + ri.w) * kHeadDim + dg * 8;
    const CT *const vbase = kbase + (size_t)n_heads * seq_capacity * kHeadDim;
    RawLane<CT> rk[4], rv[4];
    auto load_chunk = [&](int p0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int p = p0 + i * 4 + pg;
            if (p < len) { rk[i].load(kbase + (size_t)p * kHeadDim); rv[i].load(vbase + (size_t)p * kHeadDim); }
            else { rk[i].zero(); rv[i].zero(); }
        }
    };
    load_chunk(warp * 16);                             // static: before the dependency wait
    float c1[8], c2[8];
    load_n<8>(ln_c1 + qcol, c1);
    load_n<8>(ln_c2 + qcol, c2);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    float qv[kPrompt][8], acc[kPrompt][8], m[kPrompt], l[kPrompt];
#pragma unroll
    for (int j = 0; j < kPrompt; ++j) {
        const size_t r = (size_t)(j0 + min(j, n - 1)) * batch + utt;
        const float2 st = ln_stats[r];
        load_n<8>(q + r * ldq + qcol, qv[j]);
#pragma unroll
        for (int e = 0; e < 8; ++e) { qv[j][e] = fmaf(st.y, qv[j][e] - st.x * c1[e], c2[e]) * (scale * kScoreUnit); acc[j][e] = 0.f; }
        m[j] = -INFINITY;
        l[j] = 0.f;
    }
#pragma unroll 1
    for (int p0 = warp * 16; p0 < len; p0 += step) {
        if (p0 != warp * 16) load_chunk(p0);
        float s[kPrompt][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float kf[8];
            rk[i].get(kf);
            const bool in = p0 + i * 4 + pg < len;
#pragma unroll
            for (int j = 0; j < kPrompt; ++j) {
                float d = 0.f;
#pragma unroll
                for (int e = 0; e < 8; ++e) d = fmaf(qv[j][e], kf[e], d);
#pragma unroll
                for (int o = 1; o < 8; o <<= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
                s[j][i] = in ? d : -INFINITY;
            }
        }
#pragma unroll
        for (int j = 0; j < kPrompt; ++j) {
            float top = fmaxf(fmaxf(s[j][0], s[j][1]), fmaxf(s[j][2], s[j][3]));
            top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, 8));
            top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, 16));
            const float m_new = fmaxf(m[j], top), corr = softmax_weight<CT>(m[j] - m_new);
            m[j] = m_new;
            l[j] *= corr;
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[j][e] *= corr;
#pragma unroll
            for (int i = 0; i < 4; ++i) { s[j][i] = softmax_weight<CT>(s[j][i] - m_new); l[j] += s[j][i]; }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float vf[8];
            rv[i].get(vf);
#pragma unroll
            for (int j = 0; j < kPrompt; ++j)
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[j][e] = fmaf(s[j][i], vf[e], acc[j][e]);
        }
    }
#pragma unroll
    for (int j = 0; j < kPrompt; ++j) {
        l[j] += __shfl_xor_sync(0xffffffffu, l[j], 8);      // the position groups of the warp (they share m)
        l[j] += __shfl_xor_sync(0xffffffffu, l[j], 16);
        if (lane == 0) { sm_m[j][warp] = m[j]; sm_l[j][warp] = l[j]; }
        *reinterpret_cast<float2 *>(&sm_acc[j][warp][dg * 8 + pg * 2]) = sum_position_groups(acc[j], pg);
    }
    __syncthreads();
#pragma unroll 1
    for (int i = threadIdx.x; i < n * kHeadDim; i += blockDim.x) {
        const int j = i / kHeadDim, e = i % kHeadDim;
        float mw[kWarps], big = -INFINITY, sum = 0.f, o = 0.f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) { mw[w] = w < n_warps ? sm_m[j][w] : -INFINITY; big = fmaxf(big, mw[w]); }
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            if (w >= n_warps) break;
            const float wgt = mw[w] == -INFINITY ? 0.f : softmax_weight<CT>(mw[w] - big);
            sum = fmaf(sm_l[j][w], wgt, sum);
            o = fmaf(sm_acc[j][w][e], wgt, o);
        }
        o /= sum;
        const size_t at = ((size_t)(j0 + j) * batch + utt) * ldo + h * kHeadDim + e;
        const __nv_bfloat16 hi = __float2bfloat16_rn(o);
        out_hi[at] = hi;
        out_lo[at] = __float2bfloat16_rn(o - __bfloat162float(hi));
    }
}

// End of a prefill chunk: every utterance has `chunk` more positions cached; after the last chunk the argmax of the
// last prompt position (rows 0 .. batch - 1) is handed out and becomes the utterance's current token.
__global__ void prefill_finish_kernel(DecState *state, const int32_t *__restrict__ active_list,
                                      unsigned long long *__restrict__ keys, int32_t *__restrict__ t_u, int chunk, int last,
                                      int32_t *__restrict__ next_out, int32_t *__restrict__ cur_tok)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= state->batch) return;
    const int u = active_list[r];
    t_u[u] += chunk;
    if (last) {
        const int32_t tok = argmax_key_index(keys[r]);
        keys[r] = 0ull;
        cur_tok[u] = tok;
        if (next_out) next_out[u] = tok;
    }
}

// End of a step of the caller's own loop: decode the argmax keys, hand the choice out by utterance id, advance t_u.
__global__ void finish_step_kernel(DecState *state, const int32_t *__restrict__ active_list,
                                   unsigned long long *__restrict__ keys, int32_t *__restrict__ t_u,
                                   int32_t *next_out /* by utterance, nullable */, int from_state)
{
    AED_TRACE_BEGIN(state, 6);
    asm volatile("griddepcontrol.wait;" ::: "memory");       // launched with programmatic stream serialization
    if (from_state) next_out = state->step_next;
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= state->n_active) return;
    const int u = active_list[r];
    const int32_t tok = argmax_key_index(keys[r]);
    keys[r] = 0ull;
    t_u[u] += 1;
    if (next_out) next_out[u] = tok;
}

// New utterances take over slots: position 0, start token, their encoder range and forced length.  One thread each.
constexpr int kMaxAdmit = 16;
struct AdmitBatch {
    int n;
    int slot[kMaxAdmit], n_frames[kMaxAdmit], frame0[kMaxAdmit], forced_len[kMaxAdmit];
};
__global__ void admit_slots_kernel(AdmitBatch b, int bos, int32_t *__restrict__ enc_len, int32_t *__restrict__ enc_off,
                                   int32_t *__restrict__ t_u, int32_t *__restrict__ retired, int32_t *__restrict__ cur_tok,
                                   int32_t *__restrict__ max_len, int32_t *__restrict__ out_lens)
{
    const int i = threadIdx.x;
    if (blockIdx.x != 0 || i >= b.n) return;
    const int slot = b.slot[i];
    enc_len[slot] = b.n_frames[i];
    enc_off[slot] = b.frame0[i];
    t_u[slot] = 0;
    cur_tok[slot] = bos;
    max_len[slot] = b.forced_len[i];
    if (out_lens) out_lens[slot] = 0;
    retired[slot] = 0;
}

__global__ void fill_i32_kernel(int32_t *p, int32_t v, size_t n)
{
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = v;
}

}  // namespace aed

// Host side of the AED decoder library: handle, workspace layout, launch sequences, C ABI.
#include "../../include/aed_dec.h"

#include <algorithm>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <tuple>
#include <new>
#include <string>
#include <vector>

#include "common.cuh"
#include "step_kernels.cuh"
#include "tc_gemm.cuh"
#include "step_gemm.cuh"
#include "step_gemv.cuh"
#include "vocab_gemv.cuh"
#include "crosskv_gemm.cuh"
#include "plane_gemm.cuh"
#include "f32_rows.cuh"
#include "f32_cluster.cuh"
#include "step_graphs.h"
#include "stream_schedule.h"

using namespace aed;

namespace {

thread_local std::string g_create_error;

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Row counts are rounded up to 16, 32, ..., 256 and then to multiples of 256, so that few graphs cover a decode.
int rows_bucket(int rows)
{
    int b = 16;
    while (b < rows && b < 256) b <<= 1;
    if (b < rows) b = (rows + 255) / 256 * 256;
    return b;
}

// Row count a step graph is captured for.  Kernels whose grids follow the row count (attention: one block per row and
// head) pay for every row of the grid, also for those beyond the device-side count, whose blocks only find out that
// they have nothing to do, and take a slot of an SM until they have; the projections of few rows multiply tiles of four.  Every
// key is a graph to record, so: multiples of 4 up to 48 rows, of 8 up to 64, of 16 up to 256, of 32 beyond.  (Multiples of 8 from 8 on: 12 / 20 /
// 28 / 36 rows 499 / 593 / 669 / 773 us per step of the 24-layer model instead of 481 / 591 / 663 / 732.)  Never above rows_bucket(rows).
int rows_key(int rows)
{
    const int g = rows <= kFewRows ? 4 : rows <= 64 ? 8 : rows <= 256 ? 16 : 32;
    return (rows + g - 1) / g * g;
}

struct LayerWeights {
    const void *ln1_g, *ln1_b, *w_qkv, *b_qkv, *w_o, *b_o;
    const void *ln2_g, *ln2_b, *w_q_c, *b_q_c, *w_kv_c, *b_kv_c, *w_o_c, *b_o_c;
    const void *ln3_g, *ln3_b, *w_ff1, *b_ff1, *w_ff2, *b_ff2;
};

// Byte offsets of every region of the caller's workspace.
struct Layout {
    size_t self_cache, cross_store, x, act, qkv, hid, partials, pe, keys, state;
    size_t t_u, retired, active_list, cur_tok, enc_off, enc_len, max_len, row_info, row_tok, len_order, total;
    size_t self_layer_elems, cross_layer_elems;
    int max_chunks;
    // bf16 mode: activation planes (high, low) that feed the tensor-core projections
    size_t actd_hi, actd_lo, actf_hi, actf_lo;
    size_t fold_c, ln_stats, qc;          // LayerNorm-fold constants per layer, row statistics (3 sets)
    size_t slot_tokens, slot_lens;        // aed_dec_decode_stream: token rows and lengths of the slots
    size_t fold_out;                      // c1 | c2 of the vocabulary projection with the final LayerNorm folded in
    size_t comp_w, comp_b;                // per layer: Wqc diag(gamma2) Wo as bf16 [d, d], and Wqc (gamma2 * bo) as fp32 [d]
    size_t f32_layers;                    // fp32: pointers of every layer's weights
    size_t ckv_maps, ckv_bias;            // per-layer tensor maps and bias pointers of the cross-K/V weights
    size_t fold_layer_floats;
    int rows_cap;
};

bool config_supported(const aed_dec_config_t &c, std::string *why)
{
    auto fail = [&](const char *m) { if (why) *why = m; return false; };
    if (c.n_layers < 1 || c.d_model < 1 || c.n_heads < 1 || c.d_ffn < 1 || c.vocab < 2 || c.d_enc < 1)
        return fail("model dimensions must be positive (vocab >= 2)");
    if (c.dtype != AED_DTYPE_F32 && c.dtype != AED_DTYPE_BF16) return fail("dtype must be AED_DTYPE_F32 or AED_DTYPE_BF16");
    if (c.max_batch < 1 || c.max_total_enc_frames < 1 || c.max_enc_len < 1 || c.max_dec_len < 1)
        return fail("capacities must be positive");
    if (c.max_enc_len > c.max_total_enc_frames) return fail("max_enc_len exceeds max_total_enc_frames");
    if (!(c.ln_eps > 0.f)) return fail("ln_eps must be positive");
    if (c.cross_kv_format != AED_CROSS_KV_DTYPE && c.cross_kv_format != AED_CROSS_KV_E4M3)
        return fail("cross_kv_format must be AED_CROSS_KV_DTYPE or AED_CROSS_KV_E4M3");
    return true;
}

bool shape_supported(const aed_dec_config_t &c, std::string *why)
{
    auto fail = [&](const char *m) { if (why) *why = m; return false; };
    if (c.d_model % c.n_heads != 0 || c.d_model / c.n_heads != kHeadDim) return fail("head_dim must be 64");
    if (c.d_model % 64 || c.d_ffn % 64 || c.d_enc % 64) return fail("d_model, d_ffn and d_enc must be multiples of 64");
    if (c.d_model > 8192) return fail("d_model above 8192 is not supported");
    if (c.cross_kv_format == AED_CROSS_KV_E4M3 && c.dtype != AED_DTYPE_BF16)
        return fail("the 8-bit cross-attention K/V store needs the bf16 configuration");
    return true;
}

Layout make_layout(const aed_dec_config_t &c)
{
    Layout L{};
    const size_t e = c.dtype == AED_DTYPE_BF16 ? 2 : 4;
    const size_t B = c.max_batch, d = c.d_model, F = c.d_ffn;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t at = off; off = align_up(off + bytes, 256); return at; };
    L.self_layer_elems = B * 2 * d * (size_t)c.max_dec_len;
    L.cross_layer_elems = 2 * d * (size_t)c.max_total_enc_frames;
    L.self_cache = take(L.self_layer_elems * c.n_layers * e);
    L.cross_store = take(L.cross_layer_elems * c.n_layers * (c.cross_kv_format == AED_CROSS_KV_E4M3 ? 1 : e));
    L.x = take(B * d * 4);
    L.act = take(B * (d > F ? d : F) * 4);
    L.qkv = take(B * 3 * d * 4);
    L.hid = take(B * F * 4);
    int longest = c.max_enc_len > c.max_dec_len ? c.max_enc_len : c.max_dec_len;
    L.max_chunks = (longest + kAttnChunk - 1) / kAttnChunk;
    L.partials = take(B * c.n_heads * (size_t)L.max_chunks * kPartialStride * 4);
    L.pe = take((size_t)c.max_dec_len * d * 4);
    L.keys = take(B * 8);
    L.state = take(sizeof(DecState));
#ifdef AED_TRACE
    take(sizeof(TraceBuf));       // must directly follow the state (see trace_begin)
#endif
    L.t_u = take(B * 4);
    L.retired = take(B * 4);
    L.active_list = take(B * 4);
    L.cur_tok = take(B * 4);
    L.enc_off = take((B + 1) * 4);
    L.enc_len = take(B * 4);
    L.len_order = take(B * 4);                                     // utterances by decreasing encoder length (offsets, lengths and order: one copy)
    L.max_len = take(B * 4);
    L.row_info = take((size_t)rows_bucket(c.max_batch) * 16);      // grids are sized for the bucket
    L.row_tok = take((size_t)rows_bucket(c.max_batch) * 4);        // prefill: the token of every (utterance, position) row
    L.rows_cap = (int)align_up(B, 16);
    L.slot_tokens = take(B * (size_t)c.max_dec_len * 4);
    L.slot_lens = take(B * 4);
    if (c.dtype == AED_DTYPE_BF16) {
        L.actd_hi = take((size_t)L.rows_cap * d * 2);
        L.actd_lo = take((size_t)L.rows_cap * d * 2);
        L.actf_hi = take((size_t)L.rows_cap * F * 2);        // FFN hidden layer as planes (steps with many rows)
        L.actf_lo = take((size_t)L.rows_cap * F * 2);
        L.fold_layer_floats = 2 * (3 * d + d + F);       // c1 | c2 for qkv, then for cross-q, then for ffn1
        L.fold_c = take(L.fold_layer_floats * c.n_layers * 4);
        L.ln_stats = take((size_t)3 * rows_bucket(c.max_batch) * 8);
        L.qc = take(B * d * 4);
        L.ckv_maps = take((size_t)c.n_layers * sizeof(CUtensorMap));
        L.ckv_bias = take((size_t)c.n_layers * sizeof(void *));
        L.fold_out = take((size_t)2 * c.vocab * 4);
        L.comp_w = take((size_t)c.n_layers * d * d * 2);
        L.comp_b = take((size_t)c.n_layers * d * 4);
    } else {
        L.f32_layers = take((size_t)c.n_layers * sizeof(f32::ClusterLayer));
    }
    L.total = off;
    return L;
}

}  // namespace

struct aed_dec {
    aed_dec_config_t cfg;
    Layout lay;
    cudaStream_t stream;
    char *ws;
    // borrowed weights
    const void *embed, *final_ln_g, *final_ln_b, *w_out, *b_out;
    std::vector<LayerWeights> layers;
    // host view of the current batch
    int batch = 0;
    bool have_batch = false;
    bool fresh_batch = false;       // no step issued since the precompute
    int steps_issued = 0;           // steps of any kind since the precompute: upper bound on any t_u
    int full_steps = 0;             // steps without a mask: lower bound on t_u of every utterance not retired
    EncoderFrames frames;           // of the whole batch
    std::vector<int32_t> enc_len, enc_off;
    // continuous batching: the batch is a set of slots that utterances enter and leave one by one
    bool slot_mode = false;
    bool rows_ready = false;        // slots: the row table of the next step is in place ...
    const void *rows_tokens = nullptr, *rows_lens = nullptr;      // ... and these are the results' places it noted
    std::vector<int32_t> slot_t, slot_max;      // steps issued since the slot's utterance entered (-1: empty), its forced length
    std::string err;
    int64_t launches = 0;
    // optional per-kernel-family timing (CUDA events around every launch)
    bool profiling = false;
    std::vector<cudaEvent_t> prof_events;          // pool, two per recorded launch
    std::vector<int> prof_family;                  // family of each recorded launch
    size_t prof_used = 0;
    // bf16 mode: TMA descriptors of the weight matrices and of the activation planes (one per MMA N in 16..256)
    struct TcLayerMaps { CUtensorMap qkv, o, qc, oc, ff1, ff2, o_qc; };      // o_qc: the composite Wqc diag(gamma2) Wo
    std::vector<TcLayerMaps> tc_layers;
    CUtensorMap tc_w_out;
    CUtensorMap tc_actd[16][2], tc_actf[16][2];   // [N/16 - 1][plane]: activation planes [rows, d] and [rows, F]
    bool use_tc = false;
    int sm_count = 148;
    int tc_target_ctas = 128;
    bool tc_target_fixed = false;         // set from the environment: use tc_target_ctas at every row count
    bool use_pdl = true;
    bool attn_pipe = true;
    bool use_gemv = true;           // steps of few rows: projections by warp-level MMAs (step_gemv.cuh)
    int gemv_rows = kFewRows;       // ... up to this many rows
    bool use_vocab_gemv = false;    // ... and the vocabulary projection of at most 16 rows (vocab_gemv.cuh)
    int planes_rows = 128;                // steps with more rows make their activation planes once per projection input
    std::vector<f32::ClusterLayer> f32_table;
    int f32_clusters[2] = {0, 0};   // fp32 steps of small models in one launch (f32_cluster.cuh): how many clusters of 16 and of 8 blocks find room
    // steps are replayed as one captured CUDA graph per key; the output buffers stand in the device-side state
    typedef std::tuple<int, int, int, bool> GraphKey;       // (row count, chunks of self-attention positions, steps (0: one of the caller's loop), short_cross)
    typedef StepGraphs<GraphKey, cudaGraphExec_t> Graphs;
    Graphs graphs;
    bool short_cross = false;       // of the launches to come: many rows with short encoder outputs (see few_cross_warps)
    cudaStream_t capture_stream = nullptr;
    bool use_graphs = true;
    bool from_state = false;        // while such a step is recorded: its kernels find the caller's pointers in the device-side state
    // set only while aed_dec_step_static_scratch runs: attention partials go here instead of the workspace
    float *partials_override = nullptr;
    // with an end-of-sequence id: the retired count in pinned host memory, written by every greedy step
    static constexpr int kProbeSlots = 16;
    int32_t *retired_host = nullptr;
    cudaEvent_t probe_event[kProbeSlots] = {};

    template <typename T> T *at(size_t off) const { return reinterpret_cast<T *>(ws + off); }
    DecState *state() const { return at<DecState>(lay.state); }
};

namespace {

aed_status_t fail(aed_dec *d, aed_status_t code, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    if (d) d->err = buf; else g_create_error = buf;
    return code;
}

#define AED_CUDA(dec, expr)                                                                              \
    do {                                                                                                 \
        cudaError_t e__ = (expr);                                                                        \
        if (e__ != cudaSuccess) return fail(dec, AED_ERR_CUDA, "%s: %s", #expr, cudaGetErrorString(e__)); \
    } while (0)

#define AED_LAUNCHED(dec)                                                                                      \
    do {                                                                                                       \
        (dec)->launches++;                                                                                     \
        cudaError_t e__ = cudaGetLastError();                                                                  \
        if (e__ != cudaSuccess) return fail(dec, AED_ERR_CUDA, "kernel launch failed at %s:%d: %s", __FILE__, \
                                            __LINE__, cudaGetErrorString(e__));                               \
    } while (0)

enum KernelFamily { KF_BOOKKEEPING = 0, KF_EMBED, KF_LAYERNORM, KF_GEMM_QKV, KF_ATTN_SELF, KF_ATTN_COMBINE, KF_GEMM_O,
                    KF_GEMM_QC, KF_ATTN_CROSS, KF_GEMM_OC, KF_GEMM_FF1, KF_GEMM_FF2, KF_GEMM_VOCAB, KF_PRECOMPUTE,
                    KF_STEP, KF_COUNT };
const char *const kFamilyNames[KF_COUNT] = {"bookkeeping", "embed", "layernorm", "gemm_qkv", "attn_self", "attn_combine",
                                            "gemm_o", "gemm_qc", "attn_cross", "gemm_oc", "gemm_ff1", "gemm_ff2",
                                            "gemm_vocab", "precompute_cross_kv", "step"};
// A call site runs different kernels at different row counts; the profile keeps the call site and says which kernel ran it:
// family + KF_COUNT * variant, reported as "gemm_qkv@gemv", "attn_self@warp".
enum { KV_NONE = 0, KV_GEMV, KV_GEMV_STAGED, KV_PLANE, KV_GAMMA, KV_WARP, KV_F32_ROWS, KV_F32_TILE, KV_COUNT };
const char *const kVariantSuffix[KV_COUNT] = {"", "@gemv", "@gemv_staged", "@plane", "@gamma", "@warp", "@f32_rows", "@f32_tile"};

// Records an event before and after the launches issued while it is alive (profiling mode only).
struct ProfScope {
    aed_dec *dec;
    bool on;
    ProfScope(aed_dec *d, int family) : dec(d), on(d->profiling)
    {
        if (!on) return;
        if (dec->prof_used + 2 > dec->prof_events.size()) {
            for (int i = 0; i < 2; ++i) {
                cudaEvent_t e;
                if (cudaEventCreate(&e) != cudaSuccess) { on = false; return; }
                dec->prof_events.push_back(e);
            }
        }
        dec->prof_family.push_back(family);
        cudaEventRecord(dec->prof_events[dec->prof_used], dec->stream);
    }
    ~ProfScope()
    {
        if (!on) return;
        cudaEventRecord(dec->prof_events[dec->prof_used + 1], dec->stream);
        dec->prof_used += 2;
    }
};

// ---- typed launch sequences ------------------------------------------------------------------------------

template <typename T, bool kCross, bool kAppend = false>
aed_status_t launch_attention(aed_dec *dec, int rows_ub, int len_ub, const float *q, int ldq, const T *cache,
                              int seq_capacity, float *out)
{
    const auto &c = dec->cfg;
    const int H = c.n_heads;
    int chunks_ub = (len_ub + kAttnChunk - 1) / kAttnChunk;
    if (chunks_ub > dec->lay.max_chunks) chunks_ub = dec->lay.max_chunks;
    dim3 grid(rows_ub * H, (chunks_ub + 3) / 4);
    float *partials = dec->partials_override ? dec->partials_override : dec->at<float>(dec->lay.partials);
    {
    ProfScope ps(dec, kCross ? KF_ATTN_CROSS : KF_ATTN_SELF);
    attn_partial_kernel<T, kCross, kAppend><<<grid, 128, 0, dec->stream>>>(
        dec->state(), dec->at<int32_t>(dec->lay.active_list), q, ldq, const_cast<T *>(cache), H, seq_capacity,
        dec->at<int32_t>(dec->lay.t_u), dec->at<int32_t>(dec->lay.enc_off), dec->at<int32_t>(dec->lay.enc_len),
        dec->lay.max_chunks, 1.0f / sqrtf((float)kHeadDim), partials);
    AED_LAUNCHED(dec);
    }
    ProfScope ps(dec, KF_ATTN_COMBINE);
    attn_combine_kernel<kCross><<<(rows_ub * H + 3) / 4, 128, 0, dec->stream>>>(
            dec->state(), dec->at<int32_t>(dec->lay.active_list), partials, H, dec->at<int32_t>(dec->lay.t_u),
        dec->at<int32_t>(dec->lay.enc_len), dec->lay.max_chunks, out, c.d_model);
    AED_LAUNCHED(dec);
    return AED_OK;
}

// Attention in one kernel per call (no scratch): one block per (row, head), one warp per 16 positions, at most 8.
// The kernel starts with a programmatic-dependency wait, so it may be launched ahead of its predecessor's end.
template <typename T, bool kCross, bool kAppend>
aed_status_t launch_attention_fused(aed_dec *dec, int rows_ub, int len_ub, const float *q, int ldq, const T *cache,
                                    int seq_capacity, float *out, __nv_bfloat16 *out_hi, __nv_bfloat16 *out_lo,
                                    const float2 *ln_stats = nullptr, const float *ln_c1 = nullptr,
                                    const float *ln_c2 = nullptr, bool pdl = false, const float *stats_x = nullptr)
{
    // self-attention of many rows: see below
    const bool by_warp = !kCross && sizeof(T) == 2 && rows_ub * dec->cfg.n_heads > 1024;
    ProfScope ps(dec, (kCross ? KF_ATTN_CROSS : KF_ATTN_SELF) + KF_COUNT * (by_warp ? KV_WARP : KV_NONE));
    int warps = (len_ub + fused_chunk<T>() - 1) / fused_chunk<T>();
    if (warps < 2) warps = 2;                    // at least 64 threads: the merge uses one thread per head dimension
    if (warps > kFusedMaxWarps) warps = kFusedMaxWarps;
    if (kCross && dec->short_cross) warps = std::min(warps, 4);
    // Self-attention, bf16: 2 blocks of 8 warps per SM, so with more pairs than that a block has fewer warps, which take another chunk of
    // positions each, and the grid still fits.  With at most 128 positions the smaller merge is worth it a little earlier.
    // (24 layers, us per step with 8 / 4 / 2 warps: positions 100 to 120 at 8 / 16 / 48 rows 495 / 513 / 558, 572 / 550 / 586, 943 / 905 / 882;
    // 200 to 220 at 16 / 24 / 64 rows 585 / 588 / 656, 745 / 707 / 775, 1188 / 1136 / 1118; 24 to 56 at 24 / 32 / 64 rows, where 4 is the
    // most, 644 / 655, 738 / 721, 958 / 926.)
    if (!kCross && sizeof(T) == 2) {
        const int pairs = rows_ub * dec->cfg.n_heads, fit = len_ub <= 128 ? 200 : 2 * dec->sm_count;
        if (pairs > fit) warps = std::min(warps, 4);
        if (pairs > 2 * fit) warps = std::min(warps, 2);
    }
    // Attention starts early (programmatic launch) and holds each warp's first chunk in registers; rows longer than
    // 8 x 16 positions loop and find their later chunks prefetched in L2.
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(rows_ub * dec->cfg.n_heads);
    cfg.blockDim = dim3(warps * 32);
    cfg.stream = dec->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // Few blocks with long rows (late steps): the software-pipelined variant, two blocks per SM hold the whole grid.
    const bool pipe = kCross && !kAppend && rows_ub * dec->cfg.n_heads <= 2 * dec->sm_count && dec->attn_pipe;
    auto kernel = pipe ? attn_fused_kernel<T, kCross, kAppend, kCross && !kAppend> : attn_fused_kernel<T, kCross, kAppend, false>;
    if constexpr (kCross && !kAppend) {
        if (stats_x) kernel = pipe ? attn_fused_kernel<T, true, false, true, true> : attn_fused_kernel<T, true, false, false, true>;
    }
    if constexpr (!kCross && sizeof(T) == 2) {
        // One warp per (row, head) once there are more than about 7 of them per SM: a block of its own per pair spends
        // its time starting, merging and ending.  With fewer the pairs need several warps each to have enough loads in
        // flight (24-layer model, 16 heads, per step at up to 8 / 239 positions, a block per pair -> a warp per pair:
        // 64 rows 1051 / 1225 -> 1040 / 1382 us, 80 rows 1450 / 1635 -> 1394 / 1646, 128 rows 1778 / 2042 ->
        // 1666 / 1948, 512 rows 4022 / 5127 -> 3513 / 4452).
        if (by_warp) {
            cfg.gridDim = dim3((rows_ub * dec->cfg.n_heads + 7) / 8);
            cfg.blockDim = dim3(256);
            cudaError_t e = cudaLaunchKernelEx(&cfg, self_attn_warp_kernel<T, kAppend>, (const DecState *)dec->state(),
                                               (const int4 *)dec->at<int4>(dec->lay.row_info), q, ldq, const_cast<T *>(cache),
                                               dec->cfg.n_heads, seq_capacity, 1.0f / sqrtf((float)kHeadDim), out, out_hi, out_lo,
                                               dec->cfg.d_model, ln_stats, ln_c1, ln_c2, rows_ub * dec->cfg.n_heads);
            if (e != cudaSuccess) return fail(dec, AED_ERR_CUDA, "attention launch: %s", cudaGetErrorString(e));
            AED_LAUNCHED(dec);
            return AED_OK;
        }
    }
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, (const DecState *)dec->state(),
                                       (const int4 *)dec->at<int4>(dec->lay.row_info), q, ldq, const_cast<T *>(cache),
                                       dec->cfg.n_heads, seq_capacity, 1.0f / sqrtf((float)kHeadDim), out, out_hi, out_lo,
                                       dec->cfg.d_model, ln_stats, ln_c1, ln_c2, stats_x, dec->cfg.ln_eps);
    if (e != cudaSuccess) return fail(dec, AED_ERR_CUDA, "attention launch: %s", cudaGetErrorString(e));
    AED_LAUNCHED(dec);
    return AED_OK;
}

// The rule is in launch_shapes.h.
bool few_cross_warps(const aed_dec *dec, int rows_ub, const EncoderFrames &frames)
{
    return dec->use_tc && few_cross_warps((long long)rows_ub * dec->cfg.n_heads, dec->sm_count, frames, dec->cfg.cross_kv_format == AED_CROSS_KV_E4M3);
}

// A launch that may start before its predecessor in the stream has ended (programmatic stream serialization): the
// kernel itself waits (griddepcontrol.wait) before it touches what the predecessor wrote.  full: an ordinary dependency.
aed_status_t launch_pdl_impl(aed_dec *dec, const void *kernel, dim3 grid, dim3 block, size_t smem, void **args, bool full = false)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = dec->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = dec->use_pdl && !full ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelExC(&cfg, kernel, args);
    if (e != cudaSuccess) return fail(dec, AED_ERR_CUDA, "kernel launch: %s", cudaGetErrorString(e));
    AED_LAUNCHED(dec);
    return AED_OK;
}

#define AED_TRY(expr)                        \
    do {                                     \
        aed_status_t s__ = (expr);           \
        if (s__ != AED_OK) return s__;       \
    } while (0)

// fp32 projection of at most rows_ub rows (f32_rows.cuh).  Up to 4 rows one feature per warp and 4-row tiles, up to 16 rows
// 8-row tiles: as many warps as features, because a launch is bound by its latency.  Beyond, two features per warp halve the
// shared-memory reads per FMA.  Small outputs take 4 warps per block, so that they still spread over 64 SMs and more.  Many rows
// go to tiles of 64 x 64 (use_tiles says from where on); grid.y of the others stays below 25,000.
template <int EPI>
aed_status_t launch_f32(aed_dec *dec, int family, int rows_ub, f32::RowsArgs p, bool after_rows = false)
{
    const bool tiles = f32::use_tiles(p.M, rows_ub);
    ProfScope ps(dec, family + KF_COUNT * (tiles ? KV_F32_TILE : KV_F32_ROWS));
    const int warps = p.M <= 512 ? 4 : f32::kWarps;
    p.state = dec->state();
    p.eps = dec->cfg.ln_eps;
    p.after_rows = after_rows;
    void *args[] = {&p};
    const bool vec = aligned16(p.ln_g) && aligned16(p.ln_b);          // (or no LayerNorm)
    const void *kernel = rows_ub <= 4    ? (vec ? (const void *)f32::rows_kernel<EPI, 4, 1, true> : (const void *)f32::rows_kernel<EPI, 4, 1, false>)
                         : rows_ub <= 16 ? (vec ? (const void *)f32::rows_kernel<EPI, 8, 1, true> : (const void *)f32::rows_kernel<EPI, 8, 1, false>)
                                         : (vec ? (const void *)f32::rows_kernel<EPI, 8, 2, true> : (const void *)f32::rows_kernel<EPI, 8, 2, false>);
    if (tiles) {
        const dim3 grid(((p.M + f32::kTile - 1) / f32::kTile) * ((rows_ub + f32::kTile - 1) / f32::kTile));
        return launch_pdl_impl(dec, vec ? (const void *)f32::tile_kernel<EPI, true> : (const void *)f32::tile_kernel<EPI, false>, grid,
                               dim3(f32::kTileThreads), 0, args);
    }
    const int rt = rows_ub <= 4 ? 4 : 8, fpw = rows_ub <= 16 ? 1 : 2;
    const dim3 grid((p.M + warps * fpw - 1) / (warps * fpw), (rows_ub + rt - 1) / rt);
    return launch_pdl_impl(dec, kernel, grid, dim3(warps * 32), f32::rows_smem(rt, p.K), args);
}

// ---- steps of small fp32 models in one launch (f32_cluster.cuh) ------------------------------------------------------------
const void *const kClusterKernel = (const void *)f32::cluster_step_kernel;
cudaLaunchConfig_t cluster_config(const aed_dec_config_t &c, int cluster, int clusters, cudaLaunchAttribute *attr)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(clusters * cluster);
    cfg.blockDim = dim3(f32::kClusterThreads);
    cfg.dynamicSmemBytes = f32::cluster_smem(c.d_model, c.d_ffn, c.n_heads, cluster, c.n_layers);
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// The layers' weights as a table on the device, and how many clusters of either size find room at a time.
aed_status_t f32_setup(aed_dec *dec)
{
    const auto &c = dec->cfg;
    const char *v = getenv("AED_DEC_NO_CLUSTER");
    if ((v && v[0] == '1') || !f32::cluster_supports(c.d_model, c.d_ffn, c.n_layers)) return AED_OK;
    std::vector<f32::ClusterLayer> &table = dec->f32_table;            // (kept: the copy may be taken from it later)
    for (const LayerWeights &w : dec->layers) {
        auto f = [](const void *q) { return (const float *)q; };
        table.push_back({f(w.ln1_g), f(w.ln1_b), f(w.w_qkv), f(w.b_qkv), f(w.w_o), f(w.b_o), f(w.ln2_g), f(w.ln2_b), f(w.w_q_c), f(w.b_q_c), f(w.w_o_c),
                         f(w.b_o_c), f(w.ln3_g), f(w.ln3_b), f(w.w_ff1), f(w.b_ff1), f(w.w_ff2), f(w.b_ff2)});
    }
    const cudaError_t e = cudaMemcpyAsync(dec->ws + dec->lay.f32_layers, table.data(), table.size() * sizeof table[0], cudaMemcpyHostToDevice, dec->stream);
    if (e != cudaSuccess) return fail(nullptr, AED_ERR_CUDA, "fp32 set-up: %s", cudaGetErrorString(e));
    // (a GPU that does not have room for them is no error: steps run kernel by kernel)
    const size_t most = f32::cluster_smem(c.d_model, c.d_ffn, c.n_heads, f32::kClusterSizes[1], c.n_layers);
    if (cudaFuncSetAttribute(kClusterKernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most) != cudaSuccess) { cudaGetLastError(); return AED_OK; }
    bool larger = cudaFuncSetAttribute(kClusterKernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    for (int i = 0; i < 2; ++i) {
        cudaLaunchAttribute attr[2];
        const cudaLaunchConfig_t cfg = cluster_config(c, f32::kClusterSizes[i], 1, attr);
        int &fit = dec->f32_clusters[i];
        if ((i == 0 && !larger) || cudaOccupancyMaxActiveClusters(&fit, kClusterKernel, &cfg) != cudaSuccess) fit = 0;
    }
    cudaGetLastError();
    return AED_OK;
}

// Blocks per cluster for a step of rows_ub rows: the larger clusters while all of them find room, then the smaller; 0: kernel by kernel.
int cluster_of(const aed_dec *dec, int rows_ub)
{
    if (dec->partials_override) return 0;
    for (int i = 0; i < 2; ++i)
        if ((rows_ub + f32::kClusterRows - 1) / f32::kClusterRows <= dec->f32_clusters[i]) return f32::kClusterSizes[i];
    return 0;
}

aed_status_t launch_cluster_step(aed_dec *dec, int cluster, int rows_ub, const int32_t *tokens, float *logits_out)
{
    const auto &c = dec->cfg;
    const Layout &L = dec->lay;
    ProfScope ps(dec, KF_STEP);
    f32::ClusterArgs p{};
    p.state = dec->state();
    p.layers = dec->at<f32::ClusterLayer>(L.f32_layers);
    p.n_layers = c.n_layers; p.cluster_log = cluster == 16 ? 4 : 3; p.d = c.d_model; p.n_heads = c.n_heads; p.d_ffn = c.d_ffn; p.vocab = c.vocab;
    p.max_dec_len = c.max_dec_len; p.frame_capacity = c.max_total_enc_frames;
    p.eps = c.ln_eps; p.scale = sqrtf((float)c.d_model);
    p.row_info = dec->at<int4>(L.row_info);
    p.tokens = tokens;
    p.embed = (const float *)dec->embed; p.pe = dec->at<float>(L.pe);
    p.x = rows_ub <= kRowsInside ? dec->at<float>(L.x) : nullptr;          // made with the row table
    p.self_cache = dec->at<float>(L.self_cache); p.cross = dec->at<float>(L.cross_store);
    p.self_layer_elems = L.self_layer_elems; p.cross_layer_elems = L.cross_layer_elems;
    p.final_ln_g = (const float *)dec->final_ln_g; p.final_ln_b = (const float *)dec->final_ln_b;
    p.w_out = (const float *)dec->w_out; p.b_out = (const float *)dec->b_out;
    p.logits_out = logits_out;
    p.keys = dec->at<unsigned long long>(L.keys);
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = cluster_config(c, cluster, (rows_ub + f32::kClusterRows - 1) / f32::kClusterRows, attr);
    cfg.stream = dec->stream;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = dec->use_pdl ? 1 : 0;
    cfg.numAttrs = 2;
    void *args[] = {&p};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, kClusterKernel, args);
    if (e != cudaSuccess) return fail(dec, AED_ERR_CUDA, "step launch: %s", cudaGetErrorString(e));
    AED_LAUNCHED(dec);
    return AED_OK;
}

// The forward pass of one step in fp32 for the rows in the active list (at most rows_ub of them): 8 kernels per layer, chained
// with programmatic dependent launch.
//   tokens: by utterance.  self_len_ub: upper bound on t_u + 1.
aed_status_t forward_step_f32(aed_dec *dec, int rows_ub, int self_len_ub, const int32_t *tokens, float *logits_out)
{
    if (const int cluster = cluster_of(dec, rows_ub)) return launch_cluster_step(dec, cluster, rows_ub, tokens, logits_out);
    const auto &c = dec->cfg;
    const Layout &L = dec->lay;
    int d = c.d_model, V = c.vocab, zero = 0;
    const int F = c.d_ffn;
    float *x = dec->at<float>(L.x), *act = dec->at<float>(L.act), *qkv = dec->at<float>(L.qkv), *hid = dec->at<float>(L.hid), *none = nullptr;
    const int32_t *active_list = dec->at<int32_t>(L.active_list), *t_u = dec->at<int32_t>(L.t_u);
    const bool split = dec->partials_override != nullptr;        // aed_dec_step_static_scratch: attention split over chunks, with its scratch
    const bool embedded = rows_ub <= kRowsInside;          // by the kernel that made the row table
    if (!embedded) {
        ProfScope ps(dec, KF_EMBED);
        const DecState *state = dec->state();
        const float *emb = (const float *)dec->embed, *pe = dec->at<float>(L.pe);
        float sc = sqrtf((float)d);
        void *args[] = {&state, &active_list, &tokens, &t_u, &emb, &pe, &d, &V, &sc, &x, &none, &zero, &none, &zero};
        AED_TRY(launch_pdl_impl(dec, (const void *)embed_kernel<float>, dim3(rows_ub), dim3(256), 0, args));
    }
    auto rows = [&](const float *a, const void *ln_g, const void *ln_b, const void *w, const void *bias, int M, int K, float *out, int ldo) {
        f32::RowsArgs p{};
        p.rows_fixed = -1;
        p.a = a; p.ln_g = (const float *)ln_g; p.ln_b = (const float *)ln_b;
        p.w = (const float *)w; p.bias = (const float *)bias; p.M = M; p.K = K;
        p.out = out; p.ldo = ldo;
        return p;
    };
    for (int l = 0; l < c.n_layers; ++l) {
        const LayerWeights &w = dec->layers[l];
        float *self_cache = dec->at<float>(L.self_cache) + (size_t)l * L.self_layer_elems;
        const float *cross = dec->at<float>(L.cross_store) + (size_t)l * L.cross_layer_elems;
        // masked self-attention (which appends the new keys and values)
        AED_TRY(launch_f32<f32::EPI_STORE>(dec, KF_GEMM_QKV, rows_ub, rows(x, w.ln1_g, w.ln1_b, w.w_qkv, w.b_qkv, 3 * d, d, qkv, 3 * d), embedded && l == 0));
        if (split) AED_TRY((launch_attention<float, false, true>(dec, rows_ub, self_len_ub, qkv, 3 * d, self_cache, c.max_dec_len, act)));
        else AED_TRY((launch_attention_fused<float, false, true>(dec, rows_ub, self_len_ub, qkv, 3 * d, self_cache, c.max_dec_len, act, nullptr, nullptr, nullptr,
                                                                 nullptr, nullptr, dec->use_pdl)));
        AED_TRY(launch_f32<f32::EPI_RESID>(dec, KF_GEMM_O, rows_ub, rows(act, nullptr, nullptr, w.w_o, w.b_o, d, d, x, d)));
        // cross-attention over the utterance's own encoder frames
        AED_TRY(launch_f32<f32::EPI_STORE>(dec, KF_GEMM_QC, rows_ub, rows(x, w.ln2_g, w.ln2_b, w.w_q_c, w.b_q_c, d, d, qkv, d)));
        if (split) AED_TRY((launch_attention<float, true>(dec, rows_ub, c.max_enc_len, qkv, d, cross, c.max_total_enc_frames, act)));
        else AED_TRY((launch_attention_fused<float, true, false>(dec, rows_ub, c.max_enc_len, qkv, d, cross, c.max_total_enc_frames, act, nullptr, nullptr, nullptr,
                                                                 nullptr, nullptr, dec->use_pdl)));
        AED_TRY(launch_f32<f32::EPI_RESID>(dec, KF_GEMM_OC, rows_ub, rows(act, nullptr, nullptr, w.w_o_c, w.b_o_c, d, d, x, d)));
        // feed-forward
        AED_TRY(launch_f32<f32::EPI_RELU>(dec, KF_GEMM_FF1, rows_ub, rows(x, w.ln3_g, w.ln3_b, w.w_ff1, w.b_ff1, F, d, hid, F)));
        AED_TRY(launch_f32<f32::EPI_RESID>(dec, KF_GEMM_FF2, rows_ub, rows(hid, nullptr, nullptr, w.w_ff2, w.b_ff2, d, F, x, d)));
    }
    f32::RowsArgs p = rows(x, dec->final_ln_g, dec->final_ln_b, dec->w_out, dec->b_out, V, d, nullptr, 0);
    p.logits_out = logits_out;
    p.keys = dec->at<unsigned long long>(L.keys);
    p.active_list = active_list;
    return launch_f32<f32::EPI_LOGITS>(dec, KF_GEMM_VOCAB, rows_ub, p);
}


// ---- tensor-core path (bf16 mode) ----------------------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn()
{
    static EncodeTiledFn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// matrix [rows, cols] row-major; box = box_rows x 64 columns, zero fill out of bounds.  bf16 operands use the
// 128-byte swizzle the MMA descriptors name; fp32 staging tiles are copied unswizzled.
bool encode_map(CUtensorMap *map, const void *base, size_t rows, size_t cols, int box_rows, bool fp32 = false)
{
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const size_t esz = fp32 ? 4 : 2;
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {cols * esz};
    cuuint32_t box[2] = {(cuuint32_t)tc::kBlockK, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, fp32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base),
              dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              fp32 ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

using tc::kTcSmemBudget;

// The few-row projection for that many rows per CTA; wide: of up to four k-blocks (launches of 33 to 48 rows).
template <int MODE> const void *few_row_kernel(int rows, bool wide)
{
    if (wide) return rows == 20 ? (const void *)sv::step_gemv_staged_kernel<MODE, 20, 4> : rows == 24 ? (const void *)sv::step_gemv_staged_kernel<MODE, 24, 4> : nullptr;
    switch (rows) {
    case 4: return (const void *)sv::step_gemv_staged_kernel<MODE, 4>;
    case 8: return (const void *)sv::step_gemv_staged_kernel<MODE, 8>;
    case 12: return (const void *)sv::step_gemv_staged_kernel<MODE, 12>;
    case 16: return (const void *)sv::step_gemv_staged_kernel<MODE, 16>;
    case 20: return (const void *)sv::step_gemv_staged_kernel<MODE, 20>;
    case 24: return (const void *)sv::step_gemv_staged_kernel<MODE, 24>;
    case 28: return (const void *)sv::step_gemv_staged_kernel<MODE, 28>;
    default: return (const void *)sv::step_gemv_staged_kernel<MODE, 32>;
    }
}

aed_status_t tc_setup(aed_dec *dec)
{
    const auto &c = dec->cfg;
    const Layout &L = dec->lay;
    const size_t d = c.d_model, F = c.d_ffn;
    if (!encode_tiled_fn()) return fail(nullptr, AED_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
    bool ok = true;
    dec->tc_layers.resize(c.n_layers);
    std::vector<CUtensorMap> kvc_maps(c.n_layers);
    std::vector<const void *> kvc_bias(c.n_layers);
    for (int l = 0; l < c.n_layers; ++l) {
        const LayerWeights &w = dec->layers[l];
        aed_dec::TcLayerMaps &m = dec->tc_layers[l];
        ok = ok && encode_map(&m.qkv, w.w_qkv, 3 * d, d, tc::kTileM) && encode_map(&m.o, w.w_o, d, d, tc::kTileM) &&
             encode_map(&m.qc, w.w_q_c, d, d, tc::kTileM) && encode_map(&m.oc, w.w_o_c, d, d, tc::kTileM) &&
             encode_map(&m.ff1, w.w_ff1, F, d, tc::kTileM) && encode_map(&m.ff2, w.w_ff2, d, F, tc::kTileM) &&
             encode_map(&kvc_maps[l], w.w_kv_c, 2 * d, c.d_enc, ckv::kTileN / 2) &&
             encode_map(&m.o_qc, dec->ws + L.comp_w + (size_t)l * d * d * 2, d, d, tc::kTileM);
        kvc_bias[l] = w.b_kv_c;
    }
    ok = ok && encode_map(&dec->tc_w_out, dec->w_out, c.vocab, d, tc::kTileM);
    for (int i = 0; i < 16; ++i) {
        const int box = 16 * (i + 1);
        ok = ok && encode_map(&dec->tc_actd[i][0], dec->ws + L.actd_hi, L.rows_cap, d, box) &&
             encode_map(&dec->tc_actd[i][1], dec->ws + L.actd_lo, L.rows_cap, d, box) &&
             encode_map(&dec->tc_actf[i][0], dec->ws + L.actf_hi, L.rows_cap, F, box) &&
             encode_map(&dec->tc_actf[i][1], dec->ws + L.actf_lo, L.rows_cap, F, box);
    }
    if (!ok) return fail(nullptr, AED_ERR_CUDA, "cuTensorMapEncodeTiled failed (are all weight tensors 16-byte aligned?)");
    const int smem = kTcSmemBudget + 1024;
    cudaError_t e = cudaFuncSetAttribute(tc::tc_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(ckv::crosskv_gemm_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, ckv::kStages * ckv::kStageBytes + 1024);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(ckv::crosskv_gemm_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, ckv::kStages * ckv::kStageBytes + 1024);
    // tensor maps and bias pointers of the cross-K/V weights: read by the precompute kernel from the workspace
    if (e == cudaSuccess) e = cudaMemcpyAsync(dec->ws + L.ckv_maps, kvc_maps.data(), kvc_maps.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice, dec->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dec->ws + L.ckv_bias, kvc_bias.data(), kvc_bias.size() * sizeof(void *), cudaMemcpyHostToDevice, dec->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(dec->stream);       // the host vectors go away
    int dev = 0, sms = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return fail(nullptr, AED_ERR_CUDA, "tensor-core path set-up: %s", cudaGetErrorString(e));
    dec->sm_count = sms > 0 ? sms : 148;
    for (const void *k : {(const void *)sg::step_gemm_kernel<sg::B_PLAIN, 1>, (const void *)sg::step_gemm_kernel<sg::B_PLAIN, 2>, (const void *)sg::step_gemm_kernel<sg::B_PLAIN, 4>,
                          (const void *)sg::step_gemm_kernel<sg::B_GAMMA, 1>, (const void *)sg::step_gemm_kernel<sg::B_GAMMA, 2>, (const void *)sg::step_gemm_kernel<sg::B_GAMMA, 4>,
                          (const void *)sg::step_gemm_kernel<sg::B_LN_RELU, 1>, (const void *)sg::step_gemm_kernel<sg::B_LN_RELU, 2>, (const void *)sg::step_gemm_kernel<sg::B_LN_RELU, 4>})
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, sg::kSgSmem + 1024);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(pg::plane_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    for (int rows = 4; rows <= 32; rows += 4)
        for (int wide = 0; wide < 2; ++wide)
            for (const void *k : {few_row_kernel<sg::B_PLAIN>(rows, wide), few_row_kernel<sg::B_GAMMA>(rows, wide), few_row_kernel<sg::B_LN_RELU>(rows, wide)})
                if (e == cudaSuccess && k) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, sv::sv_smem(rows, wide ? 4 : sv::kSvMaxKb));
    if (e != cudaSuccess) return fail(nullptr, AED_ERR_CUDA, "tensor-core path set-up: %s", cudaGetErrorString(e));
    // LayerNorm-fold constants of every layer
    for (int l = 0; l < c.n_layers; ++l) {
        const LayerWeights &w = dec->layers[l];
        float *fc = dec->at<float>(L.fold_c) + (size_t)l * L.fold_layer_floats;
        typedef __nv_bfloat16 T;
        sg::ln_fold_constants_kernel<<<(3 * d + 7) / 8, 256, 0, dec->stream>>>((const T *)w.w_qkv, (const T *)w.ln1_g, (const T *)w.ln1_b,
                                                                               (const T *)w.b_qkv, 3 * (int)d, (int)d, fc, fc + 3 * d);
        sg::ln_fold_constants_kernel<<<(d + 7) / 8, 256, 0, dec->stream>>>((const T *)w.w_q_c, (const T *)w.ln2_g, (const T *)w.ln2_b,
                                                                           (const T *)w.b_q_c, (int)d, (int)d, fc + 6 * d, fc + 7 * d);
        sg::ln_fold_constants_kernel<<<(F + 7) / 8, 256, 0, dec->stream>>>((const T *)w.w_ff1, (const T *)w.ln3_g, (const T *)w.ln3_b,
                                                                           (const T *)w.b_ff1, (int)F, (int)d, fc + 8 * d, fc + 8 * d + F);
        // The self-attention output projection and the cross-attention query projection meet without a nonlinearity:
        // their composite lets one launch run both (see forward_step_fused).
        T *cw = dec->at<T>(L.comp_w) + (size_t)l * d * d;
        float *cb = dec->at<float>(L.comp_b) + (size_t)l * d;
        sg::compose_weights_kernel<<<dim3((unsigned)((d + 15) / 16), (unsigned)((d + 15) / 16)), 256, 0, dec->stream>>>(
            (const T *)w.w_q_c, (const T *)w.ln2_g, (const T *)w.w_o, (int)d, cw);
        sg::compose_bias_kernel<<<(d + 7) / 8, 256, 0, dec->stream>>>((const T *)w.w_q_c, (const T *)w.ln2_g, (const T *)w.b_o, (int)d, cb);
        dec->launches += 5;
    }
    {
        typedef __nv_bfloat16 T;
        float *fo = dec->at<float>(L.fold_out);
        sg::ln_fold_constants_kernel<<<(c.vocab + 7) / 8, 256, 0, dec->stream>>>((const T *)dec->w_out, (const T *)dec->final_ln_g, (const T *)dec->final_ln_b,
                                                                                (const T *)dec->b_out, c.vocab, (int)d, fo, fo + c.vocab);
        dec->launches += 1;
    }
    e = cudaGetLastError();
    // the few-row vocabulary kernel holds planes of the whole width: as wide as its shared memory, static and dynamic, allows
    cudaFuncAttributes attr;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&attr, vg::vocab_gemv_kernel<2>);
    dec->use_vocab_gemv = e == cudaSuccess && d % 128 == 0 && vg::vg_smem((int)d) + (int)attr.sharedSizeBytes <= 227 * 1024;
    if (dec->use_vocab_gemv) {
        e = cudaFuncSetAttribute(vg::vocab_gemv_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, vg::vg_smem((int)d));
        if (e == cudaSuccess) e = cudaFuncSetAttribute(vg::vocab_gemv_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, vg::vg_smem((int)d));
    }
    if (e != cudaSuccess) return fail(nullptr, AED_ERR_CUDA, "fold constants: %s", cudaGetErrorString(e));
    {
        const char *v = getenv("AED_DEC_NO_PDL");
        dec->use_pdl = !(v && v[0] == '1');
        v = getenv("AED_DEC_NO_ATTN_PIPE");
        dec->attn_pipe = !(v && v[0] == '1');
        v = getenv("AED_DEC_NO_GEMV");
        dec->use_gemv = !(v && v[0] == '1');
        v = getenv("AED_DEC_GEMV_ROWS");
        dec->gemv_rows = few_row_setting(v);
        v = getenv("AED_DEC_PLANES_ROWS");
        if (v && atoi(v) > 0) dec->planes_rows = atoi(v);

    }
    const char *ctas = getenv("AED_DEC_GEMM_CTAS");
    if (ctas && atoi(ctas) > 0) { dec->tc_target_ctas = atoi(ctas); dec->tc_target_fixed = true; }
    dec->use_tc = true;
    return AED_OK;
}

// The vocabulary projection on tensor cores: logits[r, v] = sum_k act[r, k] * Wout[v, k] (+ bias), argmax in the epilogue.
aed_status_t launch_vocab_gemm(aed_dec *dec, int rows_ub, tc::TcParams p, int rows_fixed = -1)
{
    ProfScope ps(dec, KF_GEMM_VOCAB);
    const VocabShape shape = vocab_shape(rows_ub, dec->cfg.d_model / tc::kBlockK);
    p.a_rows = dec->cfg.vocab;
    p.n_tile = shape.n_tile;
    p.k_blocks = dec->cfg.d_model / tc::kBlockK;
    p.from_state = dec->from_state;
    p.rows_fixed = rows_fixed;          // >= 0: only that many rows (a prefill pass projects its last-position rows only)
    p.state = dec->state();
    const CUtensorMap *acts = dec->tc_actd[shape.n_tile / 16 - 1];
    dim3 grid((p.a_rows + tc::kTileM - 1) / tc::kTileM, 1, shape.row_tiles);
    void *args[] = {(void *)&dec->tc_w_out, (void *)&acts[0], (void *)&acts[1], &p, (void *)&shape.stages, (void *)&shape.producers};
    return launch_pdl_impl(dec, (const void *)tc::tc_gemm_kernel, grid, dim3(tc::kThreads), shape.smem, args);
}

aed_status_t launch_ln_planes(aed_dec *dec, int rows_ub, const float *x, const void *g, const void *b)
{
    ProfScope ps(dec, KF_LAYERNORM);
    int d = dec->cfg.d_model;
    float eps = dec->cfg.ln_eps;
    const Layout &L = dec->lay;
    const DecState *state = dec->state();
    const __nv_bfloat16 *gp = (const __nv_bfloat16 *)g, *bp = (const __nv_bfloat16 *)b;
    __nv_bfloat16 *hi = dec->at<__nv_bfloat16>(L.actd_hi), *lo = dec->at<__nv_bfloat16>(L.actd_lo);
    void *args[] = {&state, &x, &gp, &bp, &d, &eps, &hi, &lo};
    return launch_pdl_impl(dec, (const void *)layernorm_planes_kernel, dim3(rows_ub), dim3(d <= 2048 ? 256 : 1024), 0, args);
}

// ---- fused step (bf16 mode): 7 kernels per layer, chained with programmatic dependent launch -------------------

template <int MODE>
aed_status_t launch_step_gemm(aed_dec *dec, int family, const CUtensorMap &map_w, int M,
                              int K, int rows_ub, sg::StepGemmParams p,
                              const CUtensorMap *map_w2 = nullptr, int M2 = 0, bool after_rows = false)
{
    // after_rows: the kernel before this launch makes the row table
    // map_w2, M2: a second weight matrix [M2, K] over the same rows (its output, gamma and bias are in p)
    p.after_rows = after_rows;
    p.a_rows2 = M2;
    const int k_blocks = K / tc::kBlockK;
    p.a_rows = M;
    p.k_blocks = k_blocks;
    p.state = dec->state();
    p.eps = dec->cfg.ln_eps;
    // k-splits: every split adds rows x features x 4 bytes of reductions, so the tcgen05 kernel stops at about one CTA per SM (256
    // CTAs instead of 128: 64 / 96 / 128 rows 1043 / 1297 / 1493 -> 1378 / 1726 / 1950 us per step of the 24-layer model; 64 instead of 128
    // at 64 / 128 rows 949 / 1356 -> 1027 / 1564).  For the
    // few-row kernels that traffic is small, and CTAs with one or two k-blocks need so little shared memory that the CTAs of the
    // next projection become resident beside them and fetch their weight tiles while this one still runs: there twice as many CTAs
    // are worth it (24-layer batch-64 workload: 129 ms per pass with a target of 128 CTAs, 121 ms with 256, 147 ms with 384).
    const bool few = dec->use_gemv && rows_ub <= dec->gemv_rows;
    const int target_ctas = dec->tc_target_fixed ? dec->tc_target_ctas : (few ? 256 : 128);
    int m_tiles = 0, splits = 0, kb_max = 0;
    // feature tiles come in multiples of `group`
    auto split = [&](int group, int row_tiles) {
        auto tiles = [&](int m) { return (m + group * tc::kTileM - 1) / (group * tc::kTileM) * group; };
        p.tiles_first = map_w2 ? tiles(M) : 0;
        m_tiles = tiles(M) + (map_w2 ? tiles(M2) : 0);
        splits = std::min(std::max(target_ctas / (m_tiles * row_tiles), 1), k_blocks);
        kb_max = (k_blocks + splits - 1) / splits;
    };
    split(1, 1);
    // Few rows: warp-level MMAs (step_gemv.cuh), rows of a CTA in multiples of 4, and from 33 rows two halves on grid.z with half the
    // k-splits, up to four k-blocks per CTA.  From 49 rows on the tcgen05 kernel takes over (20 / 24 / 32 / 40 / 48 rows 591 / 608 / 679 / 778 / 827
    // us per step of the 24-layer model here, at best 635 / 644 / 684 / 832 / 857 there; 49 / 56 / 64 rows 867 / 888 / 917 there).
    const int splits_wide = std::max((k_blocks + 3) / 4, splits / 2);
    const bool gemv = few && (rows_ub <= 32 ? kb_max <= sv::kSvMaxKb : (k_blocks + splits_wide - 1) / splits_wide <= 4);
    ProfScope ps(dec, family + KF_COUNT * (gemv ? KV_GEMV_STAGED : KV_NONE));
    if (gemv) {
        cudaLaunchConfig_t gc = {};
        gc.gridDim = dim3(m_tiles, splits, 1);
        gc.blockDim = dim3(sv::kSvThreads);
        const bool wide = rows_ub > 32;
        const int rows = ((wide ? (rows_ub + 1) / 2 : rows_ub) + 3) / 4 * 4;                  // of a CTA
        if (wide) gc.gridDim = dim3(m_tiles, splits_wide, 2);
        gc.dynamicSmemBytes = (size_t)sv::sv_smem(rows, wide ? 4 : sv::kSvMaxKb);
        gc.stream = dec->stream;
        cudaLaunchAttribute ga[1];
        ga[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        ga[0].val.programmaticStreamSerializationAllowed = dec->use_pdl ? 1 : 0;
        gc.attrs = ga;
        gc.numAttrs = 1;
        const CUtensorMap &second = map_w2 ? *map_w2 : map_w;
        void *args[] = {(void *)&map_w, (void *)&second, &p};
        const cudaError_t ge = cudaLaunchKernelExC(&gc, few_row_kernel<MODE>(rows, wide), args);
        if (ge != cudaSuccess) return fail(dec, AED_ERR_CUDA, "projection launch: %s", cudaGetErrorString(ge));
        AED_LAUNCHED(dec);
        return AED_OK;
    }
    // pairs of blocks
    p.n_tile = tc_pair_tile(rows_ub, sg::kSgMaxRows);
    const int row_tiles = (rows_ub + p.n_tile - 1) / p.n_tile, act_bytes = p.n_tile * tc::kBlockK * 2;      // of a k-block, both planes of half of the rows
    split(2, row_tiles);
    p.stages = std::min(kb_max, sg::kMaxKb);
    p.share = kb_max >= 4 ? 2 : kb_max >= 2 ? 1 : 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(m_tiles, splits, row_tiles);
    cfg.blockDim = dim3(sg::kSgThreads);
    cfg.dynamicSmemBytes = (size_t)p.stages * (tc::kATileBytes + act_bytes) + 1024;
    cfg.stream = dec->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = dec->use_pdl ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const CUtensorMap &second = map_w2 ? *map_w2 : map_w;
    const int rows_per_thread = (p.n_tile / 2 * (8 << p.share) + sg::kSgConvertThreads - 1) / sg::kSgConvertThreads;
    cudaError_t e = rows_per_thread <= 1   ? cudaLaunchKernelEx(&cfg, sg::step_gemm_kernel<MODE, 1>, map_w, second, p)
                    : rows_per_thread <= 2 ? cudaLaunchKernelEx(&cfg, sg::step_gemm_kernel<MODE, 2>, map_w, second, p)
                                           : cudaLaunchKernelEx(&cfg, sg::step_gemm_kernel<MODE, 4>, map_w, second, p);
    if (e != cudaSuccess) return fail(dec, AED_ERR_CUDA, "projection launch: %s", cudaGetErrorString(e));
    AED_LAUNCHED(dec);
    return AED_OK;
}

// A prefill pass (several prompt positions per utterance, rows = (utterance, position) pairs): the row table and the
// rows' tokens are already in place; keys and values are appended by a kernel of their own before any row attends; only
// the last chunk projects to the vocabulary, and only for the rows of the last position (rows 0 .. batch - 1).
//
// In the last layer the rows of earlier positions are done once their keys and values are in the cache: the rest of it
// runs for the rows of the last position only, or not at all before the last chunk.
struct PrefillPass { bool last_chunk; int batch; };

// Self-attention of a layer over raw [q | k | v] rows; a step appends the new position in the same launch, a prefill
// pass in one before it, because there a row reads positions that other rows append.  rows_out: rows that attend.
aed_status_t launch_self_attention(aed_dec *dec, int rows_ub, int rows_out, int self_len_ub, __nv_bfloat16 *self_cache, float *out, __nv_bfloat16 *out_hi,
                                   __nv_bfloat16 *out_lo, const float2 *stats, const float *c1, const float *c2, bool prefill)
{
    typedef __nv_bfloat16 T;
    const auto &c = dec->cfg;
    const float *qkv = dec->at<float>(dec->lay.qkv);
    const int d = c.d_model;
    if (!prefill)
        return launch_attention_fused<T, false, true>(dec, rows_ub, self_len_ub, qkv, 3 * d, self_cache, c.max_dec_len, out, out_hi, out_lo, stats, c1,
                                                      c2, dec->use_pdl);
    {
        ProfScope ps(dec, KF_ATTN_SELF);
        const DecState *state = dec->state();
        const int4 *ri = dec->at<int4>(dec->lay.row_info);
        int ldq = 3 * d, heads = c.n_heads, cap = c.max_dec_len;
        void *args[] = {&state, &ri, &qkv, &ldq, &self_cache, &heads, &cap, &stats, &c1, &c2};
        AED_TRY(launch_pdl_impl(dec, (const void *)append_kv_kernel<T>, dim3(rows_ub), dim3(256), 0, args));
    }
    if (rows_out == 0) return AED_OK;
    return launch_attention_fused<T, false, false>(dec, rows_out, self_len_ub, qkv, 3 * d, self_cache, c.max_dec_len, out, out_hi, out_lo, stats, c1, c2,
                                                   dec->use_pdl);
}

aed_status_t forward_step_fused(aed_dec *dec, int rows_ub, int self_len_ub, const int32_t *tokens, float *logits_out,
                                const PrefillPass *pf = nullptr)
{
    typedef __nv_bfloat16 T;
    const auto &c = dec->cfg;
    const Layout &L = dec->lay;
    const int d = c.d_model, F = c.d_ffn, V = c.vocab;
    float *x = dec->at<float>(L.x), *qkv = dec->at<float>(L.qkv), *hid = dec->at<float>(L.hid), *att = dec->at<float>(L.act);
    float *qc = dec->at<float>(L.qc);
    float2 *stats = dec->at<float2>(L.ln_stats);
    const int stats_stride = rows_bucket(c.max_batch);
    const int32_t *active_list = dec->at<int32_t>(L.active_list), *t_u = dec->at<int32_t>(L.t_u);
    const bool embedded = !pf && rows_ub <= kRowsInside;   // by the kernel that made the row table
    if (!embedded) {
        ProfScope ps(dec, KF_EMBED);
        if (pf)
            embed_rows_kernel<T><<<rows_ub, 256, 0, dec->stream>>>(dec->state(), dec->at<int4>(L.row_info), dec->at<int32_t>(L.row_tok),
                                                                   (const T *)dec->embed, dec->at<float>(L.pe), d, V, sqrtf((float)d), x, qkv, 3 * d,
                                                                   qc, d);
        else {
            // starts while the row compaction still runs and waits for it inside (programmatic launch)
            const DecState *state = dec->state();
            const T *emb = (const T *)dec->embed;
            const float *pe = dec->at<float>(L.pe);
            int dd = d, vv = V, zc = 3 * d, zc2 = d;
            float sc = sqrtf((float)d);
            float *zb = qkv, *zb2 = qc;
            void *args[] = {&state, &active_list, &tokens, &t_u, &emb, &pe, &dd, &vv, &sc, &x, &zb, &zc, &zb2, &zc2};
            AED_TRY(launch_pdl_impl(dec, (const void *)embed_kernel<T>, dim3(rows_ub), dim3(256), 0, args));
        }
        if (pf) AED_LAUNCHED(dec);
    }
    const bool pdl = dec->use_pdl;
    int rows = rows_ub;
    for (int l = 0; l < c.n_layers; ++l) {
        const LayerWeights &w = dec->layers[l];
        const aed_dec::TcLayerMaps &m = dec->tc_layers[l];
        T *self_cache = dec->at<T>(L.self_cache) + (size_t)l * L.self_layer_elems;
        const T *cross = dec->at<T>(L.cross_store) + (size_t)l * L.cross_layer_elems;
        const float *fc = dec->at<float>(L.fold_c) + (size_t)l * L.fold_layer_floats;
        const float *c1_qkv = fc, *c2_qkv = fc + 3 * d, *c1_qc = fc + 6 * d, *c2_qc = fc + 7 * d, *c1_ff = fc + 8 * d,
                    *c2_ff = fc + 8 * d + F;
        const LayerWeights &wn = dec->layers[(l + 1) % c.n_layers];     // next layer (or layer 0 of the next step)
        const size_t e2 = sizeof(T);
        sg::StepGemmParams p{};
        // 1. [q | k | v] raw = (gamma1 * x) Wqkv^T, and the part of the cross-attention query that this layer's input
        //    already fixes, q'A raw = (gamma2 * x) Wqc^T (the rest follows in 3) ; side: LN1 statistics of x
        p.src = x; p.ld_src = d; p.gamma = (const T *)w.ln1_g;
        p.out = qkv; p.ldo = 3 * d; p.bias = nullptr;
        p.gamma2 = (const T *)w.ln2_g; p.out2 = qc; p.ldo2 = d; p.bias2 = nullptr;
        p.stats_src = x; p.stats_out = stats; p.stats_d = d;
        p.prefetch_ptr = wn.w_qkv; p.prefetch_bytes = (size_t)3 * d * d * e2;
        p.prefetch2_ptr = wn.w_q_c; p.prefetch2_bytes = (size_t)d * d * e2;
        // the vocabulary matrix is as large as a layer: its way into L2 starts a whole layer ahead of the projection
        if (l == c.n_layers - 1) { p.prefetch2_ptr = dec->w_out; p.prefetch2_bytes = (size_t)V * d * e2; }
        AED_TRY(launch_step_gemm<sg::B_GAMMA>(dec, KF_GEMM_QKV, m.qkv, 3 * d, d, rows_ub, p, &m.qc, d, embedded && l == 0));
        // 2. self-attention (applies LN1 to q, k, v; appends k, v)
        if (pf && l == c.n_layers - 1) rows = pf->last_chunk ? pf->batch : 0;
        AED_TRY(launch_self_attention(dec, rows_ub, rows, self_len_ub, self_cache, att, nullptr, nullptr, stats, c1_qkv, c2_qkv, pf != nullptr));
        if (rows == 0) return AED_OK;
        // 3. x += att Wo^T + bo, and in the same launch the rest of the cross-attention query:
        //    (gamma2 * x_new) Wqc^T = q'A + att (Wqc diag(gamma2) Wo)^T + Wqc (gamma2 * bo), so the query projection does
        //    not wait for the sum over all features of x_new ; side: clear the FFN hidden rows
        p = sg::StepGemmParams{};
        p.src = att; p.ld_src = d;
        p.out = x; p.ldo = d; p.bias = (const T *)w.b_o;
        p.out2 = qc; p.ldo2 = d; p.bias2 = dec->at<float>(L.comp_b) + (size_t)l * d;
        p.zero_buf = hid; p.zero_cols = F;
        p.prefetch_ptr = wn.w_o; p.prefetch_bytes = (size_t)d * d * e2;
        p.prefetch2_ptr = dec->at<T>(L.comp_w) + (size_t)((l + 1) % c.n_layers) * d * d; p.prefetch2_bytes = (size_t)d * d * e2;
        AED_TRY(launch_step_gemm<sg::B_PLAIN>(dec, KF_GEMM_O, m.o, d, d, rows, p, &m.o_qc, d));
        // 4. cross-attention; every block computes the LN2 statistics of its row of x_new itself
        if (c.cross_kv_format == AED_CROSS_KV_E4M3) {
            const fp8e4m3 *cross8 = dec->at<fp8e4m3>(L.cross_store) + (size_t)l * L.cross_layer_elems;
            AED_TRY((launch_attention_fused<fp8e4m3, true, false>(dec, rows, c.max_enc_len, qc, d, cross8, c.max_total_enc_frames, att,
                                                                  nullptr, nullptr, nullptr, c1_qc, c2_qc, pdl, x)));
        } else {
            AED_TRY((launch_attention_fused<T, true, false>(dec, rows, c.max_enc_len, qc, d, cross, c.max_total_enc_frames, att,
                                                            nullptr, nullptr, nullptr, c1_qc, c2_qc, pdl, x)));
        }
        // 5. x += att Woc^T + boc ; side: clear the [q | k | v] rows for the next layer
        p = sg::StepGemmParams{};
        p.src = att; p.ld_src = d;
        p.out = x; p.ldo = d; p.bias = (const T *)w.b_o_c;
        p.zero_buf = qkv; p.zero_cols = 3 * d;
        p.prefetch_ptr = wn.w_o_c; p.prefetch_bytes = (size_t)d * d * e2;
        AED_TRY(launch_step_gemm<sg::B_PLAIN>(dec, KF_GEMM_OC, m.oc, d, d, rows, p));
        // 6. hidden raw = (gamma3 * x) W1^T ; side: LN3 statistics
        p = sg::StepGemmParams{};
        p.src = x; p.ld_src = d; p.gamma = (const T *)w.ln3_g;
        p.out = hid; p.ldo = F;
        p.stats_src = x; p.stats_out = stats + 2 * stats_stride; p.stats_d = d;
        p.prefetch_ptr = wn.w_ff1; p.prefetch_bytes = (size_t)F * d * e2;
        AED_TRY(launch_step_gemm<sg::B_GAMMA>(dec, KF_GEMM_FF1, m.ff1, F, d, rows, p));
        // 7. x += relu(LN3-corrected hidden) W2^T + b2 ; side: clear the cross-query rows
        p = sg::StepGemmParams{};
        p.src = hid; p.ld_src = F; p.c1 = c1_ff; p.c2 = c2_ff; p.stats_in = stats + 2 * stats_stride;
        p.out = x; p.ldo = d; p.bias = (const T *)w.b_ff2;
        p.zero_buf = qc; p.zero_cols = d;          // the next layer's first launch accumulates into it
        p.prefetch_ptr = wn.w_ff2; p.prefetch_bytes = (size_t)F * d * e2;
        AED_TRY(launch_step_gemm<sg::B_LN_RELU>(dec, KF_GEMM_FF2, m.ff2, d, F, rows, p));
    }
    if (!pf && dec->use_gemv && dec->use_vocab_gemv && rows <= vg::kVgRows) {
        // at most 16 rows: final LayerNorm, vocabulary projection and argmax keys in one kernel (vocab_gemv.cuh)
        ProfScope ps(dec, KF_GEMM_VOCAB + KF_COUNT * KV_GEMV);
        vg::VocabGemvParams vp{};
        vp.vocab = V; vp.d_model = d;
        vp.x = x; vp.gamma = (const T *)dec->final_ln_g;
        vp.c1 = dec->at<float>(L.fold_out); vp.c2 = vp.c1 + V;
        vp.eps = c.ln_eps;
        vp.logits_out = logits_out;
        vp.from_state = dec->from_state;
        vp.keys = dec->at<unsigned long long>(L.keys);
        vp.active_list = active_list;
        vp.state = dec->state();
        void *args[] = {(void *)&dec->tc_w_out, &vp};
        return launch_pdl_impl(dec, rows <= 8 ? (const void *)vg::vocab_gemv_kernel<1> : (const void *)vg::vocab_gemv_kernel<2>, dim3((V + tc::kTileM - 1) / tc::kTileM), dim3(vg::kVgThreads),
                               (size_t)vg::vg_smem(d), args);
    }
    AED_TRY(launch_ln_planes(dec, rows, x, dec->final_ln_g, dec->final_ln_b));
    tc::TcParams tp{};
    tp.bias = (const T *)dec->b_out;
    tp.logits_out = logits_out;
    tp.keys = dec->at<unsigned long long>(L.keys);
    tp.active_list = active_list;
    AED_TRY(launch_vocab_gemm(dec, rows, tp, pf ? rows : -1));
    return AED_OK;
}

// ---- steps with many rows (bf16 mode): activation planes made once per projection input, 11 kernels per layer -------
// With hundreds of rows every feature tile of the fused projections would convert the same activation rows again
// (24 times for the QKV projection) and that conversion, not the tensor cores, would set the pace.  Here a small kernel
// writes gamma * x as bf16 planes once, with the row statistics; attention writes its output as planes, FFN1's epilogue the
// ReLU of the corrected hidden layer; and the projections fetch both operands by TMA.

template <typename K, typename... Args>
aed_status_t launch_pdl(aed_dec *dec, K kernel, dim3 grid, dim3 block, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = dec->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = dec->use_pdl ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
    if (e != cudaSuccess) return fail(dec, AED_ERR_CUDA, "kernel launch: %s", cudaGetErrorString(e));
    AED_LAUNCHED(dec);
    return AED_OK;
}

// The shape of a projection of the many-rows path (plane_gemm.cuh).  n_tile: rows per pair of blocks; splits: k-splits.
//  * Two row tiles up to 320 rows, then tiles of at most 128: 136 rows 1872 us per step of the 24-layer model with one tile
//    of 160 and 1845 with two of 96; 304 rows 2701 with three of 128 and 2601 with two of 160; 448 rows 3284 with three of
//    160 and 3248 with four of 128.
//  * At most 128 blocks, one per SM: the pairs of a cluster launch must all find room at once (144 blocks at 384 rows: 3287 us
//    against 3015), and k-splits add rows x features x 4 bytes of reductions each.
//  * whole_k (FFN1, whose epilogue needs complete sums): more row tiles instead of k-splits (256 rows 2405 -> 2371 us).
struct PlaneShape { int n_tile, splits; };
constexpr int kPlaneBlocks = 128;
PlaneShape plane_shape(int M, int K, int rows_ub, bool whole_k)
{
    const int m_tiles = (M + 2 * tc::kTileM - 1) / (2 * tc::kTileM) * 2;
    int tiles = rows_ub <= 320 ? 2 : (rows_ub + 127) / 128;
    if (whole_k) tiles = std::max(tiles, kPlaneBlocks / m_tiles);
    const int n_tile = ((rows_ub + tiles - 1) / tiles + 31) / 32 * 32, row_tiles = (rows_ub + n_tile - 1) / n_tile;
    return {n_tile, whole_k ? 1 : std::min(std::max(kPlaneBlocks / (m_tiles * row_tiles), 1), K / tc::kBlockK)};
}

aed_status_t launch_plane_gemm(aed_dec *dec, int family, const CUtensorMap &map_w, const CUtensorMap (*planes)[2], int M, int K, int rows_ub, PlaneShape shape,
                               pg::PlaneGemmParams p)
{
    ProfScope ps(dec, family + KF_COUNT * KV_PLANE);
    p.a_rows = M;
    p.k_blocks = K / tc::kBlockK;
    p.n_tile = shape.n_tile;
    const int stage_bytes = tc::kATileBytes + p.n_tile * tc::kBlockK * 2, most = (p.k_blocks + shape.splits - 1) / shape.splits;
    p.stages = std::min({128 * 1024 / stage_bytes, pg::kPgStages, most});
    p.state = dec->state();
    // More than half of an SM's shared memory whatever the ring needs: two pairs on the same two SMs while others idle would
    // share what these take in (512 rows with 97 KB: 4150 us per step against 3500; 136 rows 1906 against 1845).
    const size_t smem = std::max({(size_t)p.stages * stage_bytes, (size_t)p.n_tile * (tc::kTileM + 4) * 4, (size_t)116 * 1024}) + 1024;
    const CUtensorMap *const maps = planes[p.n_tile / 32 - 1];
    void *args[] = {(void *)&map_w, (void *)&maps[0], (void *)&maps[1], &p};
    return launch_pdl_impl(dec, (const void *)pg::plane_gemm_kernel,
                           dim3((M + 2 * tc::kTileM - 1) / (2 * tc::kTileM) * 2, shape.splits, (rows_ub + p.n_tile - 1) / p.n_tile), dim3(pg::kPgThreads), smem, args);
}

aed_status_t forward_step_planes(aed_dec *dec, int rows_ub, int self_len_ub, const int32_t *tokens, float *logits_out,
                                 const PrefillPass *pf = nullptr)
{
    typedef __nv_bfloat16 T;
    const auto &c = dec->cfg;
    const Layout &L = dec->lay;
    const int d = c.d_model, F = c.d_ffn, V = c.vocab;
    float *x = dec->at<float>(L.x), *qkv = dec->at<float>(L.qkv), *qc = dec->at<float>(L.qc);
    T *ad_hi = dec->at<T>(L.actd_hi), *ad_lo = dec->at<T>(L.actd_lo), *af_hi = dec->at<T>(L.actf_hi), *af_lo = dec->at<T>(L.actf_lo);
    float2 *stats = dec->at<float2>(L.ln_stats);
    const int stats_stride = rows_bucket(c.max_batch);
    const int32_t *active_list = dec->at<int32_t>(L.active_list), *t_u = dec->at<int32_t>(L.t_u);
    {
        ProfScope ps(dec, KF_EMBED);
        if (pf)
            embed_rows_kernel<T><<<rows_ub, 256, 0, dec->stream>>>(dec->state(), dec->at<int4>(L.row_info), dec->at<int32_t>(L.row_tok), (const T *)dec->embed,
                                                                   dec->at<float>(L.pe), d, V, sqrtf((float)d), x, qkv, 3 * d);
        else
            embed_kernel<T><<<rows_ub, 256, 0, dec->stream>>>(dec->state(), active_list, tokens, t_u, (const T *)dec->embed,
                                                              dec->at<float>(L.pe), d, V, sqrtf((float)d), x, qkv, 3 * d);
        AED_LAUNCHED(dec);
    }
    const bool pdl = dec->use_pdl;
    int rows = rows_ub;
    const dim3 ln_block(d <= 2048 ? 256 : 1024);
    auto gamma_planes = [&](const void *g, float2 *st, float *zero_buf, int zero_cols) -> aed_status_t {
        ProfScope ps(dec, KF_LAYERNORM + KF_COUNT * KV_GAMMA);
        return launch_pdl(dec, gamma_planes_kernel, dim3(rows), ln_block, (const DecState *)dec->state(), (const float *)x,
                          (const T *)g, d, c.ln_eps, st, ad_hi, ad_lo, zero_buf, zero_cols);
    };
    const PlaneShape sh_qkv = plane_shape(3 * d, d, rows_ub, false), sh_o = plane_shape(d, d, rows_ub, false), sh_qc = sh_o,
                     sh_ff1 = plane_shape(F, d, rows_ub, true), sh_ff2 = plane_shape(d, F, rows_ub, false);
    // out: rows of their own, cleared before if there are k-splits; or null: the residual stream
    auto project = [&](int family, const CUtensorMap &map_w, const CUtensorMap (*planes)[2], int M, int K, PlaneShape shape, float *out, const void *bias) -> aed_status_t {
        pg::PlaneGemmParams p{};
        p.epi = out && shape.splits == 1 ? pg::PG_STORE : pg::PG_ADD;
        p.out = out ? out : x; p.ldo = M;
        p.bias = (const T *)bias;
        return launch_plane_gemm(dec, family, map_w, planes, M, K, rows, shape, p);
    };
    for (int l = 0; l < c.n_layers; ++l) {
        const LayerWeights &w = dec->layers[l];
        const aed_dec::TcLayerMaps &m = dec->tc_layers[l];
        T *self_cache = dec->at<T>(L.self_cache) + (size_t)l * L.self_layer_elems;
        const T *cross = dec->at<T>(L.cross_store) + (size_t)l * L.cross_layer_elems;
        const float *fc = dec->at<float>(L.fold_c) + (size_t)l * L.fold_layer_floats;
        const float *c1_qkv = fc, *c2_qkv = fc + 3 * d, *c1_qc = fc + 6 * d, *c2_qc = fc + 7 * d, *c1_ff = fc + 8 * d,
                    *c2_ff = fc + 8 * d + F;
        // self-attention block
        AED_TRY(gamma_planes(w.ln1_g, stats, sh_qc.splits > 1 ? qc : nullptr, d));
        AED_TRY(project(KF_GEMM_QKV, m.qkv, dec->tc_actd, 3 * d, d, sh_qkv, qkv, nullptr));
        if (pf && l == c.n_layers - 1) rows = pf->last_chunk ? pf->batch : 0;
        AED_TRY(launch_self_attention(dec, rows_ub, rows, self_len_ub, self_cache, nullptr, ad_hi, ad_lo, stats, c1_qkv, c2_qkv, pf != nullptr));
        if (rows == 0) return AED_OK;
        AED_TRY(project(KF_GEMM_O, m.o, dec->tc_actd, d, d, sh_o, nullptr, w.b_o));
        // cross-attention block
        AED_TRY(gamma_planes(w.ln2_g, stats + stats_stride, nullptr, 0));
        AED_TRY(project(KF_GEMM_QC, m.qc, dec->tc_actd, d, d, sh_qc, qc, nullptr));
        auto cross_attention = [&](const auto *store) -> aed_status_t {
            // Prefill, three positions of an utterance or more: its keys and values once for four of them.  4 warps per block; 2 where the blocks
            // are more than three times what the SMs hold.  (24 layers, us per prefill of utterances x positions at frames, a block per row and
            // head -> this: 37 x 9 at 110 2214 -> 2155, 20 x 24 at 110 / 400 2610 / 4099 -> 2323 / 3270, 96 x 5 at 110 2644 -> 2597, 130 x 3 at 60 2294 ->
            // 2139, 10 x 20 at 250 2088 -> 1926; 70 x 2 at 110 1510 -> 1594.)
            if (pf && rows > 2 * pf->batch) {
                ProfScope ps(dec, KF_ATTN_CROSS);
                const int chunk = rows / pf->batch;
                const dim3 grid(pf->batch * c.n_heads, (chunk + kPrompt - 1) / kPrompt);
                const int warps = (long long)grid.x * grid.y > 12ll * dec->sm_count ? 2 : 4;
                return launch_pdl(dec, prompt_cross_kernel<std::remove_const_t<std::remove_pointer_t<decltype(store)>>>, grid, dim3(32 * warps),
                                  (const int4 *)dec->at<int4>(L.row_info), (const float *)qc, d, store, c.n_heads, c.max_total_enc_frames,
                                  1.0f / sqrtf((float)kHeadDim), ad_hi, ad_lo, d, (const float2 *)(stats + stats_stride), c1_qc, c2_qc, pf->batch, chunk);
            }
            return launch_attention_fused<std::remove_const_t<std::remove_pointer_t<decltype(store)>>, true, false>(
                dec, rows, c.max_enc_len, qc, d, store, c.max_total_enc_frames, nullptr, ad_hi, ad_lo, stats + stats_stride, c1_qc, c2_qc, pdl);
        };
        if (c.cross_kv_format == AED_CROSS_KV_E4M3) AED_TRY(cross_attention((const fp8e4m3 *)(dec->at<fp8e4m3>(L.cross_store) + (size_t)l * L.cross_layer_elems)));
        else AED_TRY(cross_attention(cross));
        AED_TRY(project(KF_GEMM_OC, m.oc, dec->tc_actd, d, d, sh_o, nullptr, w.b_o_c));
        // feed-forward block; FFN1's epilogue makes the activation planes of FFN2
        AED_TRY(gamma_planes(w.ln3_g, stats + 2 * stats_stride, sh_qkv.splits > 1 ? qkv : nullptr, 3 * d));
        pg::PlaneGemmParams p{};
        p.epi = pg::PG_RELU_PLANES;
        p.c1 = c1_ff; p.c2 = c2_ff; p.stats = stats + 2 * stats_stride;
        p.out_hi = af_hi; p.out_lo = af_lo; p.ldo = F;
        AED_TRY(launch_plane_gemm(dec, KF_GEMM_FF1, m.ff1, dec->tc_actd, F, d, rows, sh_ff1, p));
        AED_TRY(project(KF_GEMM_FF2, m.ff2, dec->tc_actf, d, F, sh_ff2, nullptr, w.b_ff2));
    }
    AED_TRY(launch_ln_planes(dec, rows, x, dec->final_ln_g, dec->final_ln_b));
    tc::TcParams tp{};
    tp.bias = (const T *)dec->b_out;
    tp.logits_out = logits_out;
    tp.keys = dec->at<unsigned long long>(L.keys);
    tp.active_list = active_list;
    AED_TRY(launch_vocab_gemm(dec, rows, tp, pf ? rows : -1));
    return AED_OK;
}

aed_status_t forward_step_bf16(aed_dec *dec, int rows_ub, int self_len_ub, const int32_t *tokens, float *logits_out, const PrefillPass *pf = nullptr)
{
    return rows_ub > dec->planes_rows ? forward_step_planes(dec, rows_ub, self_len_ub, tokens, logits_out, pf)
                                      : forward_step_fused(dec, rows_ub, self_len_ub, tokens, logits_out, pf);
}

// Cross K/V of every layer on tensor cores, one persistent launch: D[frame, feature] = enc[frame, :] . w_kv_c[feature, :]
// Cross-K/V of runs of encoder frames: run i is rows src0[i] .. src0[i] + frames[i] - 1 of the tensor at enc_base
// (enc_rows rows in all) and goes to store rows dst0[i] .. (see ckv::CkvSegs; tile0 is filled here).
aed_status_t precompute_tc(aed_dec *dec, const void *enc_base, long long enc_rows, ckv::CkvSegs segs)
{
    typedef __nv_bfloat16 T;
    const auto &c = dec->cfg;
    const Layout &L = dec->lay;
    CUtensorMap map_enc;
    if (!encode_map(&map_enc, enc_base, (size_t)enc_rows, c.d_enc, tc::kTileM))
        return fail(dec, AED_ERR_CUDA, "cuTensorMapEncodeTiled failed for the encoder states");
    segs.tile0[0] = 0;
    for (int i = 0; i < segs.n; ++i) segs.tile0[i + 1] = segs.tile0[i] + (segs.frames[i] + tc::kTileM - 1) / tc::kTileM;
    ckv::CkvParams p{};
    p.segs = segs;
    p.frame_capacity = c.max_total_enc_frames;
    p.d_model = c.d_model; p.n_heads = c.n_heads; p.d_enc = c.d_enc;
    p.n_layers = c.n_layers;
    p.store = dec->ws + L.cross_store;
    p.layer_elems = L.cross_layer_elems;
    p.bias = dec->at<const T *>(L.ckv_bias);
    p.state = dec->state();
    const long long tiles = (long long)((segs.tile0[segs.n] + 1) / 2) * c.n_layers * ((2 * c.d_model + ckv::kTileN - 1) / ckv::kTileN);
    ProfScope ps(dec, KF_PRECOMPUTE);
    const unsigned grid = 2 * (unsigned)std::min<long long>(tiles, dec->sm_count / 2);
    const size_t smem = ckv::kStages * ckv::kStageBytes + 1024;
    if (c.cross_kv_format == AED_CROSS_KV_E4M3)
        ckv::crosskv_gemm_kernel<true><<<grid, ckv::kCkvThreads, smem, dec->stream>>>(map_enc, dec->at<CUtensorMap>(L.ckv_maps), p);
    else
        ckv::crosskv_gemm_kernel<false><<<grid, ckv::kCkvThreads, smem, dec->stream>>>(map_enc, dec->at<CUtensorMap>(L.ckv_maps), p);
    AED_LAUNCHED(dec);
    return AED_OK;
}

ckv::CkvSegs one_run(int frames, int dst0)
{
    ckv::CkvSegs g{};
    g.n = 1;
    g.src0[0] = 0; g.frames[0] = frames; g.dst0[0] = dst0;
    return g;
}

aed_status_t precompute_f32(aed_dec *dec, const void *enc_packed, int frames, int frame0)
{
    const auto &c = dec->cfg;
    const Layout &L = dec->lay;
    for (int l = 0; l < c.n_layers; ++l) {
        f32::RowsArgs p{};
        p.rows_fixed = frames;
        p.a = (const float *)enc_packed;
        p.w = (const float *)dec->layers[l].w_kv_c; p.bias = (const float *)dec->layers[l].b_kv_c;
        p.M = 2 * c.d_model; p.K = c.d_enc;
        p.out = dec->at<float>(L.cross_store) + (size_t)l * L.cross_layer_elems;
        p.d_model = c.d_model; p.n_heads = c.n_heads; p.frame_capacity = c.max_total_enc_frames; p.frame0 = frame0;
        AED_TRY(launch_f32<f32::EPI_CROSSKV>(dec, KF_PRECOMPUTE, frames, p));
    }
    return AED_OK;
}

// The row table of the next step (step_rows_kernel): after the bookkeeping of a greedy step that ends (finish), or on its
// own before the first one and before every step of the caller's loop.
template <typename T>
aed_status_t launch_step_rows_t(aed_dec *dec, bool finish, const uint8_t *mask, const int32_t *tokens, bool clear, int32_t *tokens_out, int32_t *out_lens,
                                float *step_logits, int32_t *step_next)
{
    const auto &c = dec->cfg;
    const Layout &L = dec->lay;
    StepRowsArgs<T> a{};
    a.state = dec->state();
    a.mask = mask; a.tokens = tokens;
    a.t_u = dec->at<int32_t>(L.t_u); a.retired = dec->at<int32_t>(L.retired); a.active_list = dec->at<int32_t>(L.active_list);
    a.max_dec_len = c.max_dec_len;
    a.enc_len = dec->at<int32_t>(L.enc_len); a.enc_off = dec->at<int32_t>(L.enc_off); a.order = dec->at<int32_t>(L.len_order);
    a.row_info = dec->at<int4>(L.row_info); a.row_slots = rows_bucket(c.max_batch);
    a.embed = (const T *)dec->embed; a.pe = dec->at<float>(L.pe); a.d = c.d_model; a.vocab = c.vocab; a.scale = sqrtf((float)c.d_model);
    a.x = dec->at<float>(L.x);
    if (clear && dec->use_tc) {
        a.zero_buf = dec->at<float>(L.qkv); a.zero_cols = 3 * c.d_model;
        a.zero_buf2 = dec->at<float>(L.qc); a.zero_cols2 = c.d_model;
    }
    a.keys = dec->at<unsigned long long>(L.keys); a.cur_tok = dec->at<int32_t>(L.cur_tok); a.max_len = dec->at<int32_t>(L.max_len); a.eos_id = c.eos_id;
    a.retired_host = dec->retired_host;
    a.tokens_out = tokens_out; a.out_lens = out_lens;
    a.step_logits = step_logits; a.step_next = step_next;
    void *args[] = {&a};
    ProfScope ps(dec, KF_BOOKKEEPING);
    return launch_pdl_impl(dec, finish ? (const void *)step_rows_kernel<T, true> : (const void *)step_rows_kernel<T, false>, dim3(1), dim3(1024), 0, args, !finish);
}
aed_status_t launch_step_rows(aed_dec *dec, bool finish, const uint8_t *mask, const int32_t *tokens, bool clear, int32_t *tokens_out = nullptr,
                              int32_t *out_lens = nullptr, float *step_logits = nullptr, int32_t *step_next = nullptr)
{
    return dec->use_tc ? launch_step_rows_t<__nv_bfloat16>(dec, finish, mask, tokens, clear, tokens_out, out_lens, step_logits, step_next)
                       : launch_step_rows_t<float>(dec, finish, mask, tokens, clear, tokens_out, out_lens, step_logits, step_next);
}

aed_status_t launch_finish(aed_dec *dec, int rows_ub, int32_t *next_out)
{
    const Layout &L = dec->lay;
    ProfScope ps(dec, KF_BOOKKEEPING);
    DecState *state = dec->state();
    const int32_t *active_list = dec->at<int32_t>(L.active_list);
    unsigned long long *keys = dec->at<unsigned long long>(L.keys);
    int32_t *t_u = dec->at<int32_t>(L.t_u);
    int from_state = dec->from_state;
    void *args[] = {&state, &active_list, &keys, &t_u, &next_out, &from_state};
    return launch_pdl_impl(dec, (const void *)finish_step_kernel, dim3((rows_ub + 127) / 128), dim3(128), 0, args);
}

// A new batch (or set of slots): lengths, offsets and visiting order in one copy, cleared bookkeeping in one kernel.
aed_status_t begin_batch(aed_dec *dec, const std::vector<int32_t> &order)
{
    const Layout &L = dec->lay;
    const size_t batch = dec->batch, at_len = (L.enc_len - L.enc_off) / 4, at_order = (L.len_order - L.enc_off) / 4;
    std::vector<int32_t> host(at_order + batch);
    std::copy(dec->enc_off.begin(), dec->enc_off.end(), host.begin());
    std::copy(dec->enc_len.begin(), dec->enc_len.end(), host.begin() + at_len);
    std::copy(order.begin(), order.end(), host.begin() + at_order);
    // Pageable host memory: cudaMemcpyAsync stages it before returning.
    AED_CUDA(dec, cudaMemcpyAsync(dec->ws + L.enc_off, host.data(), host.size() * 4, cudaMemcpyHostToDevice, dec->stream));
    ProfScope ps(dec, KF_BOOKKEEPING);
    begin_batch_kernel<<<1, 1024, 0, dec->stream>>>(dec->at<int4>(L.keys), (int)((L.enc_off - L.keys) / 16), dec->state(), dec->batch);      // keys, state, t_u, retired, lists
    AED_LAUNCHED(dec);
    dec->rows_ready = false;
    return AED_OK;
}

aed_status_t fill_i32(aed_dec *dec, int32_t *p, int32_t v, size_t n)
{
    if (n == 0) return AED_OK;
    ProfScope ps(dec, KF_BOOKKEEPING);
    fill_i32_kernel<<<(unsigned)((n + 255) / 256), 256, 0, dec->stream>>>(p, v, n);
    AED_LAUNCHED(dec);
    return AED_OK;
}

// One greedy step whose row table is in place, and the row table of the next one.
aed_status_t enqueue_greedy_step(aed_dec *dec, int rows_ub, int self_len_ub)
{
    const Layout &L = dec->lay;
    if (self_len_ub > dec->cfg.max_dec_len) self_len_ub = dec->cfg.max_dec_len;
    const int32_t *tok = dec->at<int32_t>(L.cur_tok);
    const bool planes = dec->use_tc && rows_ub > dec->planes_rows;
    aed_status_t st = dec->use_tc ? forward_step_bf16(dec, rows_ub, self_len_ub, tok, nullptr) : forward_step_f32(dec, rows_ub, self_len_ub, tok, nullptr);
    if (st != AED_OK) return st;
    // (the side jobs of the few-row projections leave the accumulators clear for the next step, the planes path does not)
    return launch_step_rows(dec, true, nullptr, tok, planes);
}

// Record greedy steps (or, with 0, a step of the caller's loop behind its first kernel) into a graph on the library's capture
// stream (nothing runs) and instantiate it.
aed_status_t capture_greedy_steps(aed_dec *dec, int rows_ub, int self_len_ub, int steps, aed_dec::Graphs::Entry *entry)
{
    if (!dec->capture_stream)
        AED_CUDA(dec, cudaStreamCreateWithFlags(&dec->capture_stream, cudaStreamNonBlocking));
    cudaStream_t user = dec->stream;
    const int64_t before = dec->launches;
    AED_CUDA(dec, cudaStreamBeginCapture(dec->capture_stream, cudaStreamCaptureModeThreadLocal));
    dec->stream = dec->capture_stream;
    aed_status_t st = AED_OK;
    for (int i = 0; i < steps && st == AED_OK; ++i) st = enqueue_greedy_step(dec, rows_ub, self_len_ub);
    if (steps == 0) {
        dec->from_state = true;
        st = forward_step_bf16(dec, rows_ub, std::min(self_len_ub, (int)dec->cfg.max_dec_len), nullptr, nullptr);
        if (st == AED_OK) st = launch_finish(dec, rows_ub, nullptr);
        dec->from_state = false;
    }
    dec->stream = user;
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamEndCapture(dec->capture_stream, &graph);
    entry->nodes = dec->launches - before;
    dec->launches = before;
    if (st != AED_OK) { if (graph) cudaGraphDestroy(graph); return st; }
    if (e != cudaSuccess || !graph) return fail(dec, AED_ERR_CUDA, "cudaStreamEndCapture: %s", cudaGetErrorString(e));
    e = cudaGraphInstantiate(&entry->exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) return fail(dec, AED_ERR_CUDA, "cudaGraphInstantiate: %s", cudaGetErrorString(e));
    return AED_OK;
}

// Steps of the same key per graph.  Inside a graph the kernels around a step's end overlap like all others (each starts
// while its predecessor runs and fetches its weights); between two graphs they do not, which costs about 3 us.  (4 steps
// instead of 1, 4-layer model: 93.5 -> 90.6 us per step of 1 row, 105.5 -> 102.1 of 8, 135.3 -> 133.9 of 24, 319.7 -> 318.5
// of 128; 24 layers: 460 -> 457 us of 1 row, nothing beyond 8; fp32, 2 layers: 51.7 -> 47.1.)  A longer graph takes longer
// to record, so deep models have them up to 8 rows and shallow ones up to 64.
constexpr int kGraphSteps = 4;
int steps_per_graph(const aed_dec *dec, int rows_b) { return rows_b <= (dec->cfg.n_layers <= 8 ? 64 : kRowsInside) ? kGraphSteps : 1; }

// The graph of `steps` greedy steps (0: a step of the caller's loop, behind its first kernel) of at most rows_b rows and chunks *
// kAttnChunk positions, recorded at first use; null if it cannot be recorded.
const aed_dec::Graphs::Entry *step_graph(aed_dec *dec, int rows_b, int chunks, int steps)
{
    return dec->graphs.get(aed_dec::GraphKey(rows_b, chunks, steps, dec->short_cross), [&](aed_dec::Graphs::Entry &entry) {
        std::string err = dec->err;
        if (capture_greedy_steps(dec, rows_b, chunks * kAttnChunk, steps, &entry) == AED_OK) return true;
        dec->err.swap(err);               // the steps are launched kernel by kernel instead: nothing has failed yet
        cudaGetLastError();
        return false;
    });
}
aed_status_t launch_graph(aed_dec *dec, const aed_dec::Graphs::Entry &graph)
{
    AED_CUDA(dec, cudaGraphLaunch(graph.exec, dec->stream));
    dec->launches += graph.nodes;
    return AED_OK;
}

}  // namespace

// ---- C ABI -------------------------------------------------------------------------------------------------

extern "C" size_t aed_dec_workspace_bytes(const aed_dec_config_t *config)
{
    if (!config || !config_supported(*config, nullptr) || !shape_supported(*config, nullptr)) return 0;
    return make_layout(*config).total;
}

extern "C" aed_status_t aed_dec_create(const aed_dec_config_t *config, const aed_dec_weights_t *w, aed_dec_t **out)
{
    if (out) *out = nullptr;
    if (!config || !w || !out) return fail(nullptr, AED_ERR_INVALID_ARG, "config, weights and out must not be NULL");
    std::string why;
    if (!config_supported(*config, &why)) return fail(nullptr, AED_ERR_INVALID_ARG, "%s", why.c_str());
    if (!shape_supported(*config, &why)) return fail(nullptr, AED_ERR_UNSUPPORTED, "%s", why.c_str());
    Layout lay = make_layout(*config);
    if (!config->workspace) return fail(nullptr, AED_ERR_INVALID_ARG, "workspace is NULL");
    if (reinterpret_cast<uintptr_t>(config->workspace) % 256) return fail(nullptr, AED_ERR_INVALID_ARG, "workspace must be 256-byte aligned");
    if (config->workspace_bytes < lay.total)
        return fail(nullptr, AED_ERR_CAPACITY, "workspace has %zu bytes, %zu needed", config->workspace_bytes, lay.total);
    const void *const *required[] = {w->ln1_g, w->ln1_b, w->w_qkv, w->w_o, w->ln2_g, w->ln2_b, w->w_q_c, w->w_kv_c,
                                     w->w_o_c, w->ln3_g, w->ln3_b, w->w_ff1, w->w_ff2};
    if (!w->embed || !w->final_ln_g || !w->final_ln_b || !w->w_out)
        return fail(nullptr, AED_ERR_INVALID_ARG, "embed, final_ln_g, final_ln_b and w_out must not be NULL");
    for (auto arr : required) {
        if (!arr) return fail(nullptr, AED_ERR_INVALID_ARG, "a required per-layer weight array is NULL");
        for (int l = 0; l < config->n_layers; ++l)
            if (!arr[l]) return fail(nullptr, AED_ERR_INVALID_ARG, "a required weight of layer %d is NULL", l);
    }
    if (config->dtype == AED_DTYPE_F32) {
        // (in the bf16 configuration the tensor maps refuse the same)
        bool ok = aligned16(w->w_out);
        for (auto arr : {w->w_qkv, w->w_o, w->w_q_c, w->w_kv_c, w->w_o_c, w->w_ff1, w->w_ff2})
            for (int l = 0; l < config->n_layers; ++l) ok = ok && aligned16(arr[l]);
        if (!ok) return fail(nullptr, AED_ERR_INVALID_ARG, "weight matrices must be 16-byte aligned");
    }
    aed_dec *dec = new (std::nothrow) aed_dec();
    if (!dec) return fail(nullptr, AED_ERR_INVALID_ARG, "out of host memory");
    dec->cfg = *config;
    dec->lay = lay;
    dec->stream = static_cast<cudaStream_t>(config->stream);
    dec->ws = static_cast<char *>(config->workspace);
    dec->embed = w->embed; dec->final_ln_g = w->final_ln_g; dec->final_ln_b = w->final_ln_b;
    dec->w_out = w->w_out; dec->b_out = w->b_out;
    dec->layers.resize(config->n_layers);
    auto opt = [](const void *const *arr, int l) -> const void * { return arr ? arr[l] : nullptr; };
    for (int l = 0; l < config->n_layers; ++l) {
        LayerWeights &lw = dec->layers[l];
        lw.ln1_g = w->ln1_g[l]; lw.ln1_b = w->ln1_b[l]; lw.w_qkv = w->w_qkv[l]; lw.b_qkv = opt(w->b_qkv, l);
        lw.w_o = w->w_o[l]; lw.b_o = opt(w->b_o, l);
        lw.ln2_g = w->ln2_g[l]; lw.ln2_b = w->ln2_b[l]; lw.w_q_c = w->w_q_c[l]; lw.b_q_c = opt(w->b_q_c, l);
        lw.w_kv_c = w->w_kv_c[l]; lw.b_kv_c = opt(w->b_kv_c, l); lw.w_o_c = w->w_o_c[l]; lw.b_o_c = opt(w->b_o_c, l);
        lw.ln3_g = w->ln3_g[l]; lw.ln3_b = w->ln3_b[l]; lw.w_ff1 = w->w_ff1[l]; lw.b_ff1 = opt(w->b_ff1, l);
        lw.w_ff2 = w->w_ff2[l]; lw.b_ff2 = opt(w->b_ff2, l);
    }
    // positional table and zeroed state
    int n = config->max_dec_len * config->d_model;
    fill_pe_kernel<<<(n + 255) / 256, 256, 0, dec->stream>>>(dec->at<float>(lay.pe), config->max_dec_len, config->d_model);
    dec->launches++;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemsetAsync(dec->ws + lay.keys, 0, lay.total - lay.keys, dec->stream);
    if (e != cudaSuccess) {
        aed_status_t s = fail(nullptr, AED_ERR_CUDA, "create: %s", cudaGetErrorString(e));
        delete dec;
        return s;
    }
    {
        const char *no_graph = getenv("AED_DEC_NO_GRAPH");
        dec->use_graphs = !(no_graph && no_graph[0] == '1');
    }
    if (config->eos_id >= 0) {
        e = cudaHostAlloc(reinterpret_cast<void **>(&dec->retired_host), sizeof(int32_t), cudaHostAllocDefault);
        for (int i = 0; i < aed_dec::kProbeSlots && e == cudaSuccess; ++i) e = cudaEventCreateWithFlags(&dec->probe_event[i], cudaEventDisableTiming);
        if (e != cudaSuccess) {
            aed_status_t s = fail(nullptr, AED_ERR_CUDA, "create: %s", cudaGetErrorString(e));
            aed_dec_destroy(dec);
            return s;
        }
    }
    if (config->dtype == AED_DTYPE_BF16) {
        aed_status_t s = tc_setup(dec);
        if (s != AED_OK) {
            aed_dec_destroy(dec);
            return s;
        }
    }
    if (config->dtype == AED_DTYPE_F32) {
        aed_status_t s = f32_setup(dec);
        if (s != AED_OK) {
            aed_dec_destroy(dec);
            return s;
        }
    }
    *out = dec;
    return AED_OK;
}

// (both configurations read the states 16 bytes at a time)
static aed_status_t check_encoder_states(aed_dec *dec, const void *enc)
{
    return aligned16(enc) ? AED_OK : fail(dec, AED_ERR_INVALID_ARG, "the encoder states must be 16-byte aligned");
}

extern "C" aed_status_t aed_dec_precompute_cross_kv(aed_dec_t *dec, const void *enc_packed, const int32_t *enc_lens,
                                                    int32_t batch)
{
    if (!dec) return AED_ERR_INVALID_ARG;
    if (!enc_packed || !enc_lens) return fail(dec, AED_ERR_INVALID_ARG, "enc_packed and enc_lens must not be NULL");
    AED_TRY(check_encoder_states(dec, enc_packed));
    if (batch < 1) return fail(dec, AED_ERR_INVALID_ARG, "batch must be at least 1");
    if (batch > dec->cfg.max_batch) return fail(dec, AED_ERR_CAPACITY, "batch %d exceeds max_batch %d", batch, dec->cfg.max_batch);
    long long total = 0;
    for (int u = 0; u < batch; ++u) {
        if (enc_lens[u] < 1) return fail(dec, AED_ERR_INVALID_ARG, "enc_lens[%d] = %d: every utterance needs at least one frame", u, enc_lens[u]);
        if (enc_lens[u] > dec->cfg.max_enc_len) return fail(dec, AED_ERR_CAPACITY, "enc_lens[%d] = %d exceeds max_enc_len %d", u, enc_lens[u], dec->cfg.max_enc_len);
        total += enc_lens[u];
    }
    if (total > dec->cfg.max_total_enc_frames)
        return fail(dec, AED_ERR_CAPACITY, "%lld encoder frames exceed max_total_enc_frames %d", total, dec->cfg.max_total_enc_frames);

    std::vector<int32_t> off(batch + 1, 0);
    for (int u = 0; u < batch; ++u) off[u + 1] = off[u] + enc_lens[u];
    // From here on the old batch is gone.
    dec->have_batch = false;
    dec->enc_len.assign(enc_lens, enc_lens + batch);
    dec->enc_off = off;
    dec->batch = batch;
    dec->frames = EncoderFrames{};
    for (int u = 0; u < batch; ++u) dec->frames.add(enc_lens[u]);
    {
        // visiting order of the row compaction: longest encoder output first (ties by utterance index)
        std::vector<int32_t> order(batch);
        for (int u = 0; u < batch; ++u) order[u] = u;
        std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) { return enc_lens[a] > enc_lens[b]; });
        AED_TRY(begin_batch(dec, order));
    }
    dec->slot_mode = false;
    aed_status_t s = dec->use_tc ? precompute_tc(dec, enc_packed, total, one_run((int)total, 0)) : precompute_f32(dec, enc_packed, (int)total, 0);
    if (s != AED_OK) return s;
    dec->have_batch = true;
    dec->fresh_batch = true;
    dec->steps_issued = 0;
    dec->full_steps = 0;
    return AED_OK;
}

extern "C" aed_status_t aed_dec_step(aed_dec_t *dec, const int32_t *tokens_in, const uint8_t *active, float *logits_out,
                                     int32_t *next_out)
{
    if (!dec) return AED_ERR_INVALID_ARG;
    if (!tokens_in) return fail(dec, AED_ERR_INVALID_ARG, "tokens_in must not be NULL");
    if (!dec->have_batch) return fail(dec, AED_ERR_STATE, "aed_dec_step needs a batch: call aed_dec_precompute_cross_kv first");
    if (dec->slot_mode) return fail(dec, AED_ERR_STATE, "aed_dec_step does not run on slots: use aed_dec_greedy_steps");
    if (dec->full_steps >= dec->cfg.max_dec_len)
        return fail(dec, AED_ERR_CAPACITY, "every utterance already holds max_dec_len = %d tokens", dec->cfg.max_dec_len);
    const int self_len_ub = dec->steps_issued + 1 < dec->cfg.max_dec_len ? dec->steps_issued + 1 : dec->cfg.max_dec_len;
    // A step of a size that keeps coming is replayed as a graph (see step_graphs.h for when and why).  Everything that a call
    // passes goes through the step's first kernel, which is launched as it is; inside a capture of the caller's own all of them are.
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    if (dec->use_tc && dec->use_graphs && !dec->profiling && !dec->partials_override) AED_CUDA(dec, cudaStreamIsCapturing(dec->stream, &capturing));
    else capturing = cudaStreamCaptureStatusActive;
    const int chunks = (self_len_ub + kAttnChunk - 1) / kAttnChunk, rows_b = rows_key(dec->batch);
    const aed_dec::Graphs::Entry *graph = nullptr;
    if (capturing == cudaStreamCaptureStatusNone) {
        dec->short_cross = few_cross_warps(dec, rows_b, dec->frames);
        if (dec->graphs.due(aed_dec::GraphKey(rows_b, chunks, 0, dec->short_cross), steps_before_recording(rows_b > dec->planes_rows)))
            graph = step_graph(dec, rows_b, chunks, 0);
    }
    AED_TRY(launch_step_rows(dec, false, active, tokens_in, true, nullptr, nullptr, logits_out, next_out));
    if (graph) {
        AED_TRY(launch_graph(dec, *graph));
    } else {
        const int rows_ub = dec->batch;
        dec->short_cross = few_cross_warps(dec, rows_ub, dec->frames);
        AED_TRY(dec->use_tc ? forward_step_bf16(dec, rows_ub, self_len_ub, tokens_in, logits_out)
                            : forward_step_f32(dec, rows_ub, self_len_ub, tokens_in, logits_out));
        AED_TRY(launch_finish(dec, rows_ub, next_out));
    }
    dec->steps_issued++;
    if (!active) dec->full_steps++;
    dec->fresh_batch = false;
    return AED_OK;
}

// ---- prompt prefill: several positions per utterance in one pass ---------------------------------------------------
extern "C" aed_status_t aed_dec_prefill(aed_dec_t *dec, const int32_t *prompt, int32_t prompt_len, float *logits_out,
                                        int32_t *next_out)
{
    if (!dec) return AED_ERR_INVALID_ARG;
    if (!prompt) return fail(dec, AED_ERR_INVALID_ARG, "prompt must not be NULL");
    if (prompt_len < 1) return fail(dec, AED_ERR_INVALID_ARG, "prompt_len must be at least 1");
    if (!dec->have_batch) return fail(dec, AED_ERR_STATE, "aed_dec_prefill needs a batch: call aed_dec_precompute_cross_kv first");
    if (!dec->fresh_batch) return fail(dec, AED_ERR_STATE, "aed_dec_prefill must directly follow aed_dec_precompute_cross_kv");
    if (prompt_len > dec->cfg.max_dec_len)
        return fail(dec, AED_ERR_CAPACITY, "prompt_len %d exceeds max_dec_len %d", prompt_len, dec->cfg.max_dec_len);
    if (!dec->use_tc) return fail(dec, AED_ERR_UNSUPPORTED, "aed_dec_prefill needs the bf16 configuration (feed the prompt with aed_dec_step in fp32 mode)");
    const Layout &L = dec->lay;
    const int B = dec->batch;
    // (utterance, position) rows share the step's row buffers: max_batch rows per pass
    const int chunk_max = std::max(1, dec->cfg.max_batch / B);
    for (int j0 = 0; j0 < prompt_len; j0 += chunk_max) {
        const int chunk = std::min(chunk_max, prompt_len - j0), rows = B * chunk;
        const bool last = j0 + chunk == prompt_len;
        {
            ProfScope ps(dec, KF_BOOKKEEPING);
            const int slots = rows_bucket(dec->cfg.max_batch);
            build_prefill_rows_kernel<<<(slots + 255) / 256, 256, 0, dec->stream>>>(
                dec->state(), chunk, j0, prompt_len, prompt, dec->at<int32_t>(L.t_u), dec->at<int32_t>(L.enc_len),
                dec->at<int32_t>(L.enc_off), dec->at<int32_t>(L.len_order), dec->at<int32_t>(L.active_list),
                dec->at<int4>(L.row_info), dec->at<int32_t>(L.row_tok), slots);
            AED_LAUNCHED(dec);
        }
        PrefillPass pf{last, B};
        dec->short_cross = few_cross_warps(dec, rows, dec->frames);
        AED_TRY(forward_step_bf16(dec, rows, j0 + chunk, nullptr, logits_out, &pf));
        {
            ProfScope ps(dec, KF_BOOKKEEPING);
            DecState *state = dec->state();
            const int32_t *active_list = dec->at<int32_t>(L.active_list);
            unsigned long long *keys = dec->at<unsigned long long>(L.keys);
            int32_t *t_u = dec->at<int32_t>(L.t_u), *cur_tok = dec->at<int32_t>(L.cur_tok);
            int chunk_arg = chunk, last_arg = last ? 1 : 0;
            void *args[] = {&state, &active_list, &keys, &t_u, &chunk_arg, &last_arg, &next_out, &cur_tok};
            AED_TRY(launch_pdl_impl(dec, (const void *)prefill_finish_kernel, dim3((B + 127) / 128), dim3(128), 0, args));
        }
    }
    dec->steps_issued = prompt_len;
    dec->full_steps = prompt_len;
    dec->fresh_batch = false;
    return AED_OK;
}

// ---- step variant for callers that cannot allocate device memory ---------------------------------------------
// The flash-decoding partials (running max, running sum and 64 accumulators per (row, head, chunk)) are the one
// piece of scratch a step needs beyond activations.  This variant keeps them in a fixed array that is part of
// the library image, so a caller that has no allocator at hand can run steps without carving room for them.
constexpr size_t kStaticScratchBytes = size_t(8) << 20;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_static_mutex;
void *g_static_scratch_addr[kMaxDevices] = {};

// Device address of the array on the current device.  In host code the array's name is only a handle for the
// runtime; the address a kernel can use has to be asked for, once per device, with that device current.
aed_status_t static_scratch_address(aed_dec *dec, float **out)
{
    int dev = -1;
    AED_CUDA(dec, cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return fail(dec, AED_ERR_UNSUPPORTED, "device index %d is out of range", dev);
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_scratch_addr[dev]) {
        void *ptr = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&ptr, g_static_scratch);
        if (e != cudaSuccess || !ptr)
            return fail(dec, AED_ERR_CUDA, "cudaGetSymbolAddress(static scratch): %s", cudaGetErrorString(e));
        g_static_scratch_addr[dev] = ptr;
    }
    *out = static_cast<float *>(g_static_scratch_addr[dev]);
    return AED_OK;
}
}  // namespace

extern "C" size_t aed_dec_static_scratch_bytes(void) { return kStaticScratchBytes; }

extern "C" aed_status_t aed_dec_step_static_scratch(aed_dec_t *dec, const int32_t *tokens_in, const uint8_t *active,
                                                    float *logits_out, int32_t *next_out)
{
    if (!dec) return AED_ERR_INVALID_ARG;
    if (!dec->have_batch)
        return fail(dec, AED_ERR_STATE, "aed_dec_step_static_scratch needs a batch: call aed_dec_precompute_cross_kv first");
    // Only the fp32 path splits attention over chunks and writes partials; the bf16 step merges inside one block
    // and touches no scratch, so no batch is refused there.
    const size_t need = dec->use_tc ? 0 : (size_t)dec->batch * dec->cfg.n_heads * dec->lay.max_chunks * kPartialStride * sizeof(float);
    if (need > kStaticScratchBytes)
        return fail(dec, AED_ERR_CAPACITY,
                    "batch %d x %d heads x %d chunks needs %zu bytes of attention scratch; the built-in array holds %zu",
                    dec->batch, dec->cfg.n_heads, dec->lay.max_chunks, need, kStaticScratchBytes);
    float *scratch = nullptr;
    AED_TRY(static_scratch_address(dec, &scratch));
    dec->partials_override = scratch;
    aed_status_t s = aed_dec_step(dec, tokens_in, active, logits_out, next_out);
    dec->partials_override = nullptr;
    return s;
}

extern "C" aed_status_t aed_dec_greedy_decode(aed_dec_t *dec, const int32_t *max_len, int32_t *tokens_out, int32_t *out_lens)
{
    if (!dec) return AED_ERR_INVALID_ARG;
    if (!max_len || !tokens_out || !out_lens) return fail(dec, AED_ERR_INVALID_ARG, "max_len, tokens_out and out_lens must not be NULL");
    if (!dec->have_batch) return fail(dec, AED_ERR_STATE, "aed_dec_greedy_decode needs a batch: call aed_dec_precompute_cross_kv first");
    if (!dec->fresh_batch || dec->slot_mode) return fail(dec, AED_ERR_STATE, "aed_dec_greedy_decode must directly follow aed_dec_precompute_cross_kv");
    const int B = dec->batch;
    int longest = 0;
    for (int u = 0; u < B; ++u) {
        if (max_len[u] < 1) return fail(dec, AED_ERR_INVALID_ARG, "max_len[%d] = %d: must be at least 1", u, max_len[u]);
        if (max_len[u] > dec->cfg.max_dec_len) return fail(dec, AED_ERR_CAPACITY, "max_len[%d] = %d exceeds max_dec_len %d", u, max_len[u], dec->cfg.max_dec_len);
        if (max_len[u] > longest) longest = max_len[u];
    }
    const Layout &L = dec->lay;
    // rows still alive at step s: utterances with max_len > s (exact without EOS, an upper bound with it)
    std::vector<int> alive(longest + 1, 0);
    for (int u = 0; u < B; ++u) alive[max_len[u] - 1]++;
    std::vector<EncoderFrames> frames_alive(longest + 1);
    for (int u = 0; u < B; ++u) frames_alive[max_len[u] - 1].add(dec->enc_len[u]);
    for (int s = longest - 1; s >= 0; --s) { alive[s] += alive[s + 1]; frames_alive[s].add(frames_alive[s + 1]); }

    dec->fresh_batch = false;
    AED_CUDA(dec, cudaMemcpyAsync(dec->ws + L.max_len, max_len, B * 4, cudaMemcpyHostToDevice, dec->stream));
    const bool probe = dec->cfg.eos_id >= 0;
    {
        ProfScope ps(dec, KF_BOOKKEEPING);
        const size_t n = (size_t)B * dec->cfg.max_dec_len;
        begin_greedy_kernel<<<(unsigned)((n + 255) / 256), 256, 0, dec->stream>>>(dec->at<int32_t>(L.cur_tok), dec->cfg.bos_id, B, tokens_out, n, out_lens);
        AED_LAUNCHED(dec);
    }
    AED_TRY(launch_step_rows(dec, false, nullptr, dec->at<int32_t>(L.cur_tok), true, tokens_out, out_lens));
    // With an end-of-sequence id the forced lengths are only upper bounds.  The host then stays at most kWindow steps
    // ahead of the device (an event behind every launch) and stops once every utterance has retired, as the steps report
    // in pinned memory.
    constexpr int kWindow = 8;
    int done = 0, oldest = 0, newest = 0;                   // steps known to be over; ring of launches in flight
    int ends[aed_dec::kProbeSlots];
    for (int s = 0; s < longest;) {
        // grids are sized for the keyed row count; kernels leave rows beyond the device-side row count alone
        const int rows_b = rows_key(alive[s]), chunks = s / kAttnChunk + 1;
        dec->short_cross = few_cross_warps(dec, rows_b, frames_alive[s]);
        const aed_dec::Graphs::Entry *graph = nullptr;
        int n = 1;
        if (dec->use_graphs && !dec->profiling) {
            const int most = steps_per_graph(dec, rows_b);
            while (n < most && s + n < longest && rows_key(alive[s + n]) == rows_b && (s + n) / kAttnChunk + 1 == chunks) ++n;
            if (n < most) n = 1;
            graph = step_graph(dec, rows_b, chunks, n);
            if (!graph) n = 1;
        }
        if (probe) {
            while (s + n - done > kWindow) {
                AED_CUDA(dec, cudaEventSynchronize(dec->probe_event[oldest % aed_dec::kProbeSlots]));
                done = ends[oldest++ % aed_dec::kProbeSlots];
            }
            // (looked at only behind an event of this decode; steps already issued beyond the last retirement do nothing)
            if (done > 0 && *static_cast<volatile int32_t *>(dec->retired_host) >= B) break;
        }
        if (graph) AED_TRY(launch_graph(dec, *graph));
        else AED_TRY(enqueue_greedy_step(dec, alive[s], s + 1));
        s += n;
        dec->steps_issued = s;
        if (probe) {
            AED_CUDA(dec, cudaEventRecord(dec->probe_event[newest % aed_dec::kProbeSlots], dec->stream));
            ends[newest++ % aed_dec::kProbeSlots] = s;
        }
    }
    dec->full_steps = dec->cfg.max_dec_len;   // every utterance is retired: further steps are refused
    return aed_dec_sync_status(dec);
}

// ---- continuous batching: utterances enter and leave slots one by one -----------------------------------------------

extern "C" aed_status_t aed_dec_open_slots(aed_dec_t *dec, int32_t slots)
{
    if (!dec) return AED_ERR_INVALID_ARG;
    const auto &c = dec->cfg;
    if (slots < 1) return fail(dec, AED_ERR_INVALID_ARG, "slots must be at least 1");
    if (slots > c.max_batch) return fail(dec, AED_ERR_CAPACITY, "%d slots exceed max_batch %d", slots, c.max_batch);
    if ((long long)slots * c.max_enc_len > c.max_total_enc_frames)
        return fail(dec, AED_ERR_CAPACITY, "%d slots of max_enc_len %d frames exceed max_total_enc_frames %d", slots, c.max_enc_len,
                    c.max_total_enc_frames);
    const Layout &L = dec->lay;
    dec->have_batch = false;
    dec->batch = slots;
    dec->frames = EncoderFrames{};
    dec->enc_len.assign(slots, 0);
    dec->enc_off.assign(slots + 1, 0);
    for (int u = 0; u <= slots; ++u) dec->enc_off[u] = u * c.max_enc_len;       // every slot owns max_enc_len store rows
    dec->slot_t.assign(slots, -1);
    dec->slot_max.assign(slots, 0);
    {
        std::vector<int32_t> order(slots);
        for (int u = 0; u < slots; ++u) order[u] = u;
        AED_TRY(begin_batch(dec, order));
    }
    AED_TRY(fill_i32(dec, dec->at<int32_t>(L.retired), 1, slots));      // empty slots take no part in a step
    dec->slot_mode = true;
    dec->have_batch = true;
    dec->fresh_batch = false;
    dec->steps_issued = 0;
    dec->full_steps = 0;
    return AED_OK;
}

namespace {

struct Admission { int slot; long long src_row; int frames, max_len; };

aed_status_t check_admission(aed_dec *dec, const Admission &a)
{
    const auto &c = dec->cfg;
    if (a.slot < 0 || a.slot >= dec->batch) return fail(dec, AED_ERR_INVALID_ARG, "slot %d is outside 0..%d", a.slot, dec->batch - 1);
    if (a.frames < 1) return fail(dec, AED_ERR_INVALID_ARG, "enc_len = %d: an utterance needs at least one frame", a.frames);
    if (a.frames > c.max_enc_len) return fail(dec, AED_ERR_CAPACITY, "enc_len = %d exceeds max_enc_len %d", a.frames, c.max_enc_len);
    if (a.max_len < 1) return fail(dec, AED_ERR_INVALID_ARG, "max_len = %d: must be at least 1", a.max_len);
    if (a.max_len > c.max_dec_len) return fail(dec, AED_ERR_CAPACITY, "max_len = %d exceeds max_dec_len %d", a.max_len, c.max_dec_len);
    // Without an end-of-sequence id the host knows when a slot's utterance ends; with one the caller has seen
    // out_lens[slot] > 0 before it reuses the slot.
    if (c.eos_id < 0 && dec->slot_t[a.slot] >= 0 && dec->slot_t[a.slot] < dec->slot_max[a.slot])
        return fail(dec, AED_ERR_STATE, "slot %d still decodes (%d of %d tokens)", a.slot, dec->slot_t[a.slot], dec->slot_max[a.slot]);
    return AED_OK;
}

// Up to ckv::kMaxSegs utterances enter their slots with one cross-K/V launch and one bookkeeping launch.  The encoder
// states of admission i are rows src_row .. src_row + frames - 1 of the tensor at enc_base (enc_rows rows).
aed_status_t admit_many(aed_dec *dec, const void *enc_base, long long enc_rows, const Admission *adm, int n, int32_t *out_lens)
{
    static_assert(kMaxAdmit == ckv::kMaxSegs, "one bookkeeping entry per run of frames");
    const auto &c = dec->cfg;
    const Layout &L = dec->lay;
    const size_t row_bytes = (size_t)c.d_enc * (c.dtype == AED_DTYPE_BF16 ? 2 : 4);
    ckv::CkvSegs segs{};
    AdmitBatch ab{};
    segs.n = ab.n = n;
    for (int i = 0; i < n; ++i) {
        AED_TRY(check_admission(dec, adm[i]));
        for (int k = 0; k < i; ++k)
            if (adm[k].slot == adm[i].slot) return fail(dec, AED_ERR_INVALID_ARG, "slot %d is admitted into twice", adm[i].slot);
        segs.src0[i] = (int)adm[i].src_row; segs.frames[i] = adm[i].frames; segs.dst0[i] = adm[i].slot * c.max_enc_len;
        ab.slot[i] = adm[i].slot; ab.n_frames[i] = adm[i].frames; ab.frame0[i] = segs.dst0[i]; ab.forced_len[i] = adm[i].max_len;
    }
    dec->rows_ready = false;
    if (dec->use_tc) {
        AED_TRY(precompute_tc(dec, enc_base, enc_rows, segs));
    } else {
        for (int i = 0; i < n; ++i)
            AED_TRY(precompute_f32(dec, static_cast<const char *>(enc_base) + (size_t)adm[i].src_row * row_bytes, adm[i].frames, segs.dst0[i]));
    }
    {
        ProfScope ps(dec, KF_BOOKKEEPING);
        admit_slots_kernel<<<1, 32, 0, dec->stream>>>(ab, c.bos_id, dec->at<int32_t>(L.enc_len), dec->at<int32_t>(L.enc_off),
                                                      dec->at<int32_t>(L.t_u), dec->at<int32_t>(L.retired), dec->at<int32_t>(L.cur_tok),
                                                      dec->at<int32_t>(L.max_len), out_lens);
        AED_LAUNCHED(dec);
    }
    for (int i = 0; i < n; ++i) {
        dec->enc_len[adm[i].slot] = adm[i].frames;
        dec->slot_t[adm[i].slot] = 0;
        dec->slot_max[adm[i].slot] = adm[i].max_len;
    }
    return AED_OK;
}

}  // namespace

extern "C" aed_status_t aed_dec_admit(aed_dec_t *dec, int32_t slot, const void *enc, int32_t enc_len, int32_t max_len,
                                      int32_t *out_lens)
{
    if (!dec) return AED_ERR_INVALID_ARG;
    if (!dec->have_batch || !dec->slot_mode) return fail(dec, AED_ERR_STATE, "aed_dec_admit needs slots: call aed_dec_open_slots first");
    if (!enc) return fail(dec, AED_ERR_INVALID_ARG, "enc must not be NULL");
    AED_TRY(check_encoder_states(dec, enc));
    const Admission a{slot, 0, enc_len, max_len};
    AED_TRY(check_admission(dec, a));           // before enc_len is used as the extent of the tensor
    return admit_many(dec, enc, enc_len, &a, 1, out_lens);
}

extern "C" aed_status_t aed_dec_greedy_steps(aed_dec_t *dec, int32_t n_steps, int32_t *tokens_out, int32_t *out_lens,
                                             int32_t *steps_done)
{
    if (steps_done) *steps_done = 0;
    if (!dec) return AED_ERR_INVALID_ARG;
    if (!dec->have_batch || !dec->slot_mode) return fail(dec, AED_ERR_STATE, "aed_dec_greedy_steps needs slots: call aed_dec_open_slots first");
    if (!tokens_out || !out_lens) return fail(dec, AED_ERR_INVALID_ARG, "tokens_out and out_lens must not be NULL");
    if (n_steps < 0) return fail(dec, AED_ERR_INVALID_ARG, "n_steps must not be negative");
    for (int s = 0; s < n_steps;) {
        // what the host knows: a slot decodes until its forced length (with an end-of-sequence id it may stop earlier
        // on the device; its row then simply is not there any more)
        EncoderFrames frames;
        auto rows_at = [&](int ahead, int &longest) {
            int rows = 0;
            longest = 0;
            frames = EncoderFrames{};
            for (int u = 0; u < dec->batch; ++u)
                if (dec->slot_t[u] >= 0 && dec->slot_t[u] + ahead < dec->slot_max[u]) { ++rows; longest = std::max(longest, dec->slot_t[u] + ahead + 1); frames.add(dec->enc_len[u]); }
            return rows;
        };
        int longest;
        const int rows_ub = rows_at(0, longest);
        if (rows_ub == 0) break;
        dec->short_cross = few_cross_warps(dec, rows_key(rows_ub), frames);
        if (!dec->rows_ready || dec->rows_tokens != tokens_out || dec->rows_lens != out_lens) {
            AED_TRY(launch_step_rows(dec, false, nullptr, dec->at<int32_t>(dec->lay.cur_tok), true, tokens_out, out_lens));
            dec->rows_ready = true;
            dec->rows_tokens = tokens_out; dec->rows_lens = out_lens;
        }
        const aed_dec::Graphs::Entry *graph = nullptr;
        int n = 1;
        if (dec->use_graphs && !dec->profiling) {
            const int rows_b = rows_key(rows_ub), chunks = (longest + kAttnChunk - 1) / kAttnChunk, most = steps_per_graph(dec, rows_b);
            if (most <= n_steps - s) {
                int last;
                const int rows_last = rows_at(most - 1, last);       // (rows only leave in between, positions only grow)
                if (rows_last > 0 && rows_key(rows_last) == rows_b && (last + kAttnChunk - 1) / kAttnChunk == chunks && last == longest + most - 1) n = most;
            }
            graph = step_graph(dec, rows_b, chunks, n);
            if (!graph) n = 1;
        }
        if (graph) AED_TRY(launch_graph(dec, *graph));
        else AED_TRY(enqueue_greedy_step(dec, rows_ub, longest));
        for (int u = 0; u < dec->batch; ++u)
            if (dec->slot_t[u] >= 0 && dec->slot_t[u] < dec->slot_max[u]) dec->slot_t[u] = std::min(dec->slot_t[u] + n, dec->slot_max[u]);
        s += n;
        if (steps_done) *steps_done += n;
    }
    return AED_OK;
}

extern "C" aed_status_t aed_dec_decode_stream(aed_dec_t *dec, const void *enc_packed, const int32_t *enc_lens,
                                              const int32_t *max_lens, const int32_t *order, int32_t n, int32_t slots,
                                              int32_t poll_steps, int32_t *tokens_out, int32_t *out_lens,
                                              int64_t *steps_out, int64_t *row_steps_out)
{
    if (steps_out) *steps_out = 0;
    if (row_steps_out) *row_steps_out = 0;
    if (!dec) return AED_ERR_INVALID_ARG;
    if (!enc_packed || !enc_lens || !max_lens || !tokens_out || !out_lens)
        return fail(dec, AED_ERR_INVALID_ARG, "enc_packed, enc_lens, max_lens, tokens_out and out_lens must not be NULL");
    AED_TRY(check_encoder_states(dec, enc_packed));
    if (n < 1) return fail(dec, AED_ERR_INVALID_ARG, "n must be at least 1");
    const auto &c = dec->cfg;
    const bool eos = c.eos_id >= 0;
    if (eos && poll_steps < 1) return fail(dec, AED_ERR_INVALID_ARG, "poll_steps must be at least 1 when eos_id >= 0");
    std::vector<long long> off(n + 1, 0);
    std::vector<char> seen(n, 0);
    for (int i = 0; i < n; ++i) {
        if (enc_lens[i] < 1 || enc_lens[i] > c.max_enc_len)
            return fail(dec, enc_lens[i] < 1 ? AED_ERR_INVALID_ARG : AED_ERR_CAPACITY, "enc_lens[%d] = %d is outside 1..max_enc_len = %d", i, enc_lens[i], c.max_enc_len);
        if (max_lens[i] < 1 || max_lens[i] > c.max_dec_len)
            return fail(dec, max_lens[i] < 1 ? AED_ERR_INVALID_ARG : AED_ERR_CAPACITY, "max_lens[%d] = %d is outside 1..max_dec_len = %d", i, max_lens[i], c.max_dec_len);
        off[i + 1] = off[i] + enc_lens[i];
        if (order) {
            if (order[i] < 0 || order[i] >= n || seen[order[i]]) return fail(dec, AED_ERR_INVALID_ARG, "order is not a permutation of 0..n-1");
            seen[order[i]] = 1;
        }
    }
    AED_TRY(aed_dec_open_slots(dec, slots));
    const Layout &L = dec->lay;
    if (off[n] > 0x7fffffffLL) return fail(dec, AED_ERR_CAPACITY, "the stream has %lld encoder frames; at most 2^31 - 1 per call", off[n]);
    // The scheduling decisions are in stream_schedule.h; here are its operations on the device.
    struct Ops {
        aed_dec *dec;
        const void *enc_packed;
        const std::vector<long long> &off;
        const int32_t *enc_lens, *max_lens;
        int32_t *toks, *lens, *tokens_out, *out_lens;
        int ld, slots;
        int admit(const StreamAdmission *a, int k)
        {
            Admission adm[ckv::kMaxSegs];
            for (int i = 0; i < k; ++i) adm[i] = Admission{a[i].slot, off[a[i].utterance], enc_lens[a[i].utterance], max_lens[a[i].utterance]};
            return admit_many(dec, enc_packed, off.back(), adm, k, lens);
        }
        int steps(int want, int *done)
        {
            int32_t d = 0;
            const aed_status_t st = aed_dec_greedy_steps(dec, want, toks, lens, &d);
            *done = d;
            return st;
        }
        int read_lens(int32_t *host)
        {
            if (cudaMemcpyAsync(host, lens, (size_t)slots * 4, cudaMemcpyDeviceToHost, dec->stream) != cudaSuccess ||
                cudaStreamSynchronize(dec->stream) != cudaSuccess)
                return fail(dec, AED_ERR_CUDA, "reading the slot lengths: %s", cudaGetErrorString(cudaGetLastError()));
            return AED_OK;
        }
        // The finished utterance's tokens and length go to the host behind the steps that produced them and before
        // the slot's next occupant (stream order); with pinned host buffers the host does not wait for them.
        int harvest(int s, int u)
        {
            if (cudaMemcpyAsync(tokens_out + (size_t)u * ld, toks + (size_t)s * ld, (size_t)max_lens[u] * 4, cudaMemcpyDeviceToHost, dec->stream) != cudaSuccess ||
                cudaMemcpyAsync(out_lens + u, lens + s, 4, cudaMemcpyDeviceToHost, dec->stream) != cudaSuccess)
                return fail(dec, AED_ERR_CUDA, "copying a finished utterance out: %s", cudaGetErrorString(cudaGetLastError()));
            return AED_OK;
        }
    } ops{dec, enc_packed, off, enc_lens, max_lens, dec->at<int32_t>(L.slot_tokens), dec->at<int32_t>(L.slot_lens), tokens_out,
          out_lens, c.max_dec_len, slots};
    StreamTotals tot;
    const int rc = run_stream_schedule(n, slots, order, max_lens, eos, poll_steps, ckv::kMaxSegs, ops, &tot);
    if (rc < 0) return static_cast<aed_status_t>(rc);
    const long long steps = tot.steps, row_steps = tot.row_steps;
    if (steps_out) *steps_out = steps;
    if (row_steps_out) *row_steps_out = row_steps;
    return aed_dec_sync_status(dec);
}

extern "C" aed_status_t aed_dec_sync_status(aed_dec_t *dec)
{
    if (!dec) return AED_ERR_INVALID_ARG;
    DecState host{};
    AED_CUDA(dec, cudaMemcpyAsync(&host, dec->state(), sizeof host, cudaMemcpyDeviceToHost, dec->stream));
    AED_CUDA(dec, cudaStreamSynchronize(dec->stream));
    const aed_status_t s = aed_dec_status_of_error_word(host.error);
    if (s == AED_ERR_CAPACITY) return fail(dec, s, "a step was asked of an utterance whose self-attention cache is full");
    if (s != AED_OK) return fail(dec, s, "a bounded wait on the device ran out (device-side error %d)", host.error);
    return AED_OK;
}

// The sticky error word of the device-side decode state as a status: 0 = fine, 1 = a self-attention cache was full,
// anything else = a kernel gave up waiting.
extern "C" aed_status_t aed_dec_status_of_error_word(int32_t error_word)
{
    if (error_word == 0) return AED_OK;
    if (error_word == 1) return AED_ERR_CAPACITY;
    return AED_ERR_TIMEOUT;
}

extern "C" aed_status_t aed_dec_profile_enable(aed_dec_t *dec, int32_t enable)
{
    if (!dec) return AED_ERR_INVALID_ARG;
    AED_CUDA(dec, cudaStreamSynchronize(dec->stream));
    dec->profiling = enable != 0;
    dec->prof_used = 0;
    dec->prof_family.clear();
    return AED_OK;
}

extern "C" int32_t aed_dec_profile_read(aed_dec_t *dec, int32_t max_families, const char **names, double *ms,
                                        int64_t *launches)
{
    if (!dec || !names || !ms || !launches || max_families < 1) return AED_ERR_INVALID_ARG;
    if (cudaStreamSynchronize(dec->stream) != cudaSuccess) return AED_ERR_CUDA;
    double sum[KF_COUNT * KV_COUNT] = {0};
    int64_t cnt[KF_COUNT * KV_COUNT] = {0};
    static std::string variant_names[KF_COUNT * KV_COUNT];
    static std::once_flag once;
    std::call_once(once, [] {
        for (int v = 0; v < KV_COUNT; ++v)
            for (int f = 0; f < KF_COUNT; ++f) variant_names[f + KF_COUNT * v] = std::string(kFamilyNames[f]) + kVariantSuffix[v];
    });
    for (size_t i = 0; i < dec->prof_family.size() && 2 * i + 1 < dec->prof_used + 1; ++i) {
        float t = 0.f;
        if (cudaEventElapsedTime(&t, dec->prof_events[2 * i], dec->prof_events[2 * i + 1]) != cudaSuccess) continue;
        sum[dec->prof_family[i]] += t;
        cnt[dec->prof_family[i]]++;
    }
    int n = 0;
    for (int f = 0; f < KF_COUNT * KV_COUNT && n < max_families; ++f) {
        if (!cnt[f]) continue;
        names[n] = variant_names[f].c_str(); ms[n] = sum[f]; launches[n] = cnt[f];
        ++n;
    }
    return n;
}

extern "C" int64_t aed_dec_launch_count(const aed_dec_t *dec) { return dec ? dec->launches : 0; }

extern "C" void aed_dec_destroy(aed_dec_t *dec)
{
    if (!dec) return;
    for (cudaEvent_t e : dec->prof_events) cudaEventDestroy(e);
    dec->graphs.clear([](cudaGraphExec_t g) { cudaGraphExecDestroy(g); });
    if (dec->capture_stream) cudaStreamDestroy(dec->capture_stream);
    for (cudaEvent_t e : dec->probe_event) if (e) cudaEventDestroy(e);
    if (dec->retired_host) cudaFreeHost(dec->retired_host);
    delete dec;
}

extern "C" const char *aed_dec_last_error(const aed_dec_t *dec) { return dec ? dec->err.c_str() : ""; }

extern "C" const char *aed_dec_create_error(void) { return g_create_error.c_str(); }

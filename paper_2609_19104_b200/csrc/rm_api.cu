// C-ABI entry points: argument validation and dispatch.  Every step of the path runs in the library's kernels.
#include <new>
#include <cstring>
#include <cstdlib>
#include <string>

#include "rm_common.cuh"

int rm_last_cuda_error = 0;

namespace {

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

inline bool all_aligned(std::initializer_list<const void*> ps) {
    for (const void* p : ps)
        if (p && !rm_aligned16(p)) return false;
    return true;
}

inline bool use_fused(const rm_ctx* ctx, int B, int T) {
    return ctx->path != 1 && rm_fused_supported(ctx, B, T);
}

// The whole-step kernel (variant 5).  Chosen by itself where it is measured ahead of the per-layer kernels (single episodes).
// Its time per layer is ~11 us at H = 1024 and ~15 us at H = 2048, with little growth in K or T (chains between CTAs); the
// lean per-layer kernel's grows with T (tiles of 32 or 64 token columns; T > 52: one CTA per SM) and by a step at every
// 64-neuron tile that makes a cluster's run longer; the streaming kernel's by a step at every wave of tiles over the SMs.
// us per step of 6 layers, whole-step / per-layer kernels (s: streaming), by T (I = 4096 and 16384):
//   H = 1024  K =  500: 8: 62/35    32: 64/40    52: 66/53    56: 66/59    64: 67/62
//                  900: 8: 62/37    32: 65/43    52: 66/55    56: 67/67    64: 67/70
//                 1024: 8: 65/42    32: 67/48    48: 68/63    52: 69/63    64: 69/84
//                 1152: 33: 67/62   48: 69/70    52: 69/70    64: 70/98s
//                 1280: 8: 66/47    32: 68/54    33: 68/65    52: 69/72    64: 70/98s
//                 1900: 8: 68/55    32: 70/63    33: 70/72    52: 72/82
//                 2048: 8: 70/58    32: 72/65    33: 72/74    52: 73/85
//   H = 2048  K =  500: 8: 83/50    32: 88/61    48: 91/73    64: 94/80
//                  960: 8: 84/60    32: 89/69    48: 92/83    56: 93/87    64: 95/90
//                 1024: 8: 86/85    32: 91/94    48: 94/108   64: 97/119
//                 4600: 8: 144/137s 32: 150/147s 51: 154/161s
//                 4900: 8: 149/139s 32: 155/148s 51: 158/161s
//                 6100: 8: 158/141s 32: 165/151s 40: 167/162s 64: 171/165s
//                 6500: 8: 162/141s 32: 168/152s 40: 170/163s 64: 174/166s
//                 9400: 8: 223/157s 32: 231/194s 64: 237/207s   (10000, beyond a wave of 148 tiles: 225/265s, 239/324s)
// with the anchor update (Eq. 4), whose sums the streaming kernel is slow at:
//   H = 1024  K =  600: 8: 67/41    32: 72/46    51: 74/59    60: 75/68    64: 76/70
//                  900: 8: 68/42    32: 73/48    51: 74/61    60: 75/74    64: 76/76
//                 1400: 8: 71/51    32: 77/59    40: 78/73    51: 78/79    64: 80/95
//                 2048: 8: 76/62    32: 82/70    33: 81/83
//   H = 2048  K =  960: 8: 92/63    32: 103/75   64: 116/106      1100: 8: 94/88   32: 107/97
// So, in tiles of 64 neurons, with K the caller's count hint (the whole layer for a dense pass): up to the bounds below the
// layer kernels; from the bounds of H = 2048 up to one wave the streaming kernel.  The bounds were drawn where the columns crossed when
// the layer kernels took 3 to 8 us more; they now lie a few tiles on the low side (H = 1024: 16 to 24 tiles of 33 to 52
// tokens, 30 and more of up to 32).  Without a hint the whole-step kernel at
// H = 2048 (it adapts to the counts on the device), the lean kernel at H = 1024.  Batches stay with the streaming kernel.
// `steps`: a whole stack (false: the one-layer entry, which pays the kernel's set-up for a single layer, and only where a streaming
// tile takes longer still; H = 2048, us, whole-step / streaming / two-tile kernel (T = 64: the lean kernel in its place):
//   T =  8: 36 tiles 20.8/22.8/17.5   57: 22.7/22.8/20.9     T = 32: 36: 18.3/24.0/19.2   48: 19.2/24.0/23.2   57: 19.6/24.0/23.3
//   T = 48: 30 tiles 18.4/26.1/17.8   33: 18.6/26.2/22.2   57: 19.9/26.2/27.0   63: 26.9/26.2/31.3     T = 64: 33: 18.5/26.3/26.2   57: 19.8/26.3/32.3;
// up to 4 tiles of 64 to a cluster: its tile is one of 256).  It takes 120 SMs for that time, the streaming kernel one per tile:
// calls on several streams overlap less (33 tiles of 48 tokens, us a round of 1 / 2 / 4 streams: 18.8/34.4/68 against 26.2/27.2/35).
inline bool use_persist(const rm_ctx* ctx, int B, int T, bool masked, bool eq4, bool steps) {
    if (ctx->path == 1 || !rm_persist_supported(ctx, B, T)) return false;
    if (ctx->variant_override == 5) return true;
    if ((ctx->variant_override != 0 && ctx->variant_override != 7) || B > ctx->persist_max_b) return false;
    const long long K = masked ? rm_effective_count_hint(ctx) : ctx->g.I, tiles = (K + 63) / 64;
    if (!steps) return ctx->g.H == 2048 && ctx->stream_min_tiles == 0 && T > 16 && tiles >= (T > 32 ? 31 : 46) && tiles < 4 * ctx->persist_clusters;
    if (K <= 0) return ctx->g.H == 2048;
    if (ctx->g.H == 2048) {
        if (tiles <= (eq4 || T <= 55 ? 15 : 13)) return false;
        return eq4 || tiles < (T <= 32 ? 77 : 101) || tiles > ctx->sm_count;
    }
    if (T <= 32) return tiles > (eq4 ? 32 : 29);
    if (rm_fused_two_per_sm(ctx, T)) return tiles > (eq4 ? 20 : T <= 48 ? 16 : 15);
    return tiles > (eq4 ? 13 : 8);
}

inline void* persist_ws(const rm_ctx* ctx, void* ws, int B, int T) {
    const size_t r_bytes = align_up((size_t)B * T * ctx->g.H * sizeof(float), 256);
    return static_cast<char*>(ws) + 4 * r_bytes + align_up(rm_ref_workspace_bytes(ctx, B, T), 256);
}

// The slice kernel (variant 6): where the tcgen05 kernels do not reach (widths other than 1024 and 2048, chunks of more than
// 64 tokens), instead of the CUDA-core kernels.  One step of 12 layers of 1536/6144 with 25 % of the neurons and 51 tokens:
// 272 us against 9335.
inline bool use_slice(const rm_ctx* ctx, int B, int T, bool record) {
    if (ctx->path == 1 || !rm_slice_supported(ctx, B, T, record)) return false;
    return ctx->variant_override == 6 || (ctx->path == 0 && !rm_fused_supported(ctx, B, T));
}

// The sweep kernel (variant 7): dense steps of one episode, where a cluster of the whole-step kernel would walk more than one
// tile of 256 neurons per layer.  us per step of 18 layers, 51 tokens, whole-step / sweep: H = 1024, I = 3000: 213 / 248,
// 3500: 220 / 263, 4096: 282 / 255, 6000: 309 / 279; H = 2048, I = 8000: 540 / 430, 16384: 1085 / 750.
// The line lies at the same place from 8 to 64 tokens (6 layers, 8 tokens: 3840 72 / 85, 3900 93 / 86) and at H = 2048 (51 tokens:
// 3840 110 / 124, 3900 150 / 124, 4500 152 / 125, 6000 165 / 133).
inline bool use_sweep(const rm_ctx* ctx, int B, int T, bool dense) {
    if (ctx->path == 1 || !dense || !rm_sweep_supported(ctx, B, T)) return false;
    if (ctx->variant_override != 0) return ctx->variant_override == 7;
    return ctx->g.I > 256 * ctx->persist_clusters;
}
inline void* sweep_ws(const rm_ctx* ctx, void* ws, int B, int T) {
    char* p = static_cast<char*>(persist_ws(ctx, ws, B, T)) + align_up(rm_persist_workspace_bytes(ctx), 256) + rm_slice_workspace_bytes(ctx, B, T);
    return reinterpret_cast<void*>(align_up(reinterpret_cast<size_t>(p), 1024));
}

// the slice kernel's control block and partial sums in a workspace of (B, T)
inline void slice_buffers(const rm_ctx* ctx, rm_step_args& sa, void* ws, int B, int T) {
    sa.ctrl = reinterpret_cast<int*>(static_cast<char*>(persist_ws(ctx, ws, B, T)) + align_up(rm_persist_workspace_bytes(ctx), 256));
}

// The streaming variant (whole tiles per CTA): a tile costs an SM ~16 us at H = 1024 (its gathers run at ~20 bytes per clock,
// its adds at 16), however few tiles there are; the cluster kernels, which spread a tile over 8 SMs, win while every cluster
// has a single tile.  Measured crossover, us a step of 18 layers and 51 tokens, lean / streaming kernel (the lean kernel's time steps up
// with every round of its 32 (H = 1024) or 15 (H = 2048) co-resident clusters): H = 1024: 32 tiles 269 / 291, 36 tiles 363 / 293 (20
// tokens: 285 / 251), 46 tiles 408 / 294.  H = 2048: up to 30 tiles 360 to 380 / ~470, 32 tiles 531 / 475, 52 tiles 658 / 491.
// The option stream_min_tiles, when set, stands for these lines, and for a single layer's (which it then keeps off the whole-step kernel).
// `masked` says whether a count is in play.
// With the anchor state of Eq. 4 the tiles do more (the anchor step adds two boxes per block and stores h_anchor, an update step reads
// it), in the layer kernels beside other tiles.  us per 6 layers, 4 episodes, streaming / layer kernels:
//   anchor step, H = 1024, T = 20: 40 tiles 112 / 100, 44 116 / 116     T = 51: 56 168 / 144, 60 168 / 158     T = 60: 32 162 / 137
//                H = 2048, T = 20: 32 tiles 219 / 201     T = 51: 32 307 / 279     T = 56: 48 315 / 240, 56 316 / 277, 64 312 / 318
//   update step, H = 1024, T = 20: 36 tiles 115 / 99     T = 51: 36 132 / 149
//                H = 2048, T = 8: 32 tiles 218 / 170, 52 219 / 180, 64 217 / 220     T = 20: 32 219 / 177, 52 217 / 188     T = 51: 32 236 / 248
// Where the lean kernel fits an SM only once (H = 1024, T > 52), clusters walk two tiles from 16 tiles on: half the threshold.  The
// two-tile kernel takes those launches; 2 episodes of 60 tokens, us per 6 layers, streaming / two-tile / lean kernel: 16 tiles 97 / 80 / 89,
// 18 97 / 93 / 104, 20 97 / 82 / 91, 28 98 / 89 / 99, 32 98 / 115 / 132 (from 17 to 30 tiles half the threshold is on the low side); with
// the gate alone 18 99 / 96 / 107, 32 100 / 118 / 135; update steps 16 115 / 88 / 97, 18 116 / 107 / 117, 32 129 / 134 / 151; anchor steps 32
// 162 / 137 / 151.  One layer alone: T = 56, 18 tiles 17.0 / 13.7, 30 17.1 / 14.2, 31 17.2 / 17.0; at H = 2048 the two-tile kernel
// takes up to 59 tiles of short chunks.
inline bool use_stream(const rm_ctx* ctx, bool masked, int B, int T, int anchor_mode = RM_ANCHOR_NONE, bool eq4 = false, bool steps = true) {
    if (ctx->path == 1 || !rm_stream_supported(ctx, B, T)) return false;
    if (ctx->variant_override == 4) return true;
    if (ctx->variant_override != 0 && ctx->variant_override != 5 && ctx->variant_override != 7) return false;   // 5, 7: a call the whole-step kernel does not cover
    const int per_episode = masked ? rm_effective_count_hint(ctx) : ctx->g.I;
    if (per_episode <= 0) return false;
    const long long tiles = (long long)((per_episode + 63) / 64) * B;
    const bool wide = ctx->g.H == 2048, once = !wide && !rm_fused_two_per_sm(ctx, T);
    const int line = ctx->stream_min_tiles > 0 ? ctx->stream_min_tiles : wide ? 31 : 33;
    int least = !eq4 && once ? line / 2 + line % 2 : line, eq4_least = 0;
    if (!steps && ctx->stream_min_tiles == 0) least = wide ? (T <= 32 ? 4 * ctx->fused_clusters : line) : once ? 2 * ctx->fused_clusters + 1 : line;
    if (anchor_mode == RM_ANCHOR_WRITE) eq4_least = wide ? (T > 52 ? 53 : 0) : T <= 32 ? 41 : once ? 0 : 57;
    if (anchor_mode == RM_ANCHOR_UPDATE && wide && T <= 32) eq4_least = 64;
    return tiles >= (least > eq4_least ? least : eq4_least);
}

}  // namespace

extern "C" {

int rm_create(rm_ctx** out, const rm_model_desc* desc) {
    if (!out) return RM_ERR_INVALID_ARG;
    *out = nullptr;
    if (!desc) return RM_ERR_INVALID_ARG;
    if (desc->L < 1 || desc->H < 64 || desc->I < 1 || desc->T_max < 1 || desc->B_max < 1) return RM_ERR_INVALID_ARG;
    if (desc->H % 64 != 0) return RM_ERR_SHAPE;
    if (desc->act != RM_ACT_GELU_TANH) return RM_ERR_UNSUPPORTED;
    rm_ctx* c = new (std::nothrow) rm_ctx();
    if (!c) return RM_ERR_CUDA;
    c->desc = *desc;
    c->g.L = desc->L;
    c->g.H = desc->H;
    c->g.I = desc->I;
    c->g.Hs = desc->H / RM_NS;
    c->launches = 0;
    c->status_detail = 0;
    c->stream_min_tiles = 0;
    c->d_status = nullptr;
    int major = 0;                         // (two attributes: cudaGetDeviceProperties takes milliseconds)
    if (cudaGetDevice(&c->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, c->device) != cudaSuccess ||
        cudaMalloc(&c->d_status, (RM_STATUS_INTS + RM_ALONE_INTS) * sizeof(int)) != cudaSuccess ||
        cudaMemset(c->d_status, 0, (RM_STATUS_INTS + RM_ALONE_INTS) * sizeof(int)) != cudaSuccess) {
        if (c->d_status) cudaFree(c->d_status);
        delete c;
        return RM_ERR_CUDA;
    }
    c->path = 0;
    c->use_pdl = 1;
    c->npc_target = 64;
    c->count_hint = 0;
    c->count_hint_seen = 0;
    c->max_clusters_override = 0;
    c->variant_override = 0;
    c->l2_prefetch = 0;
    c->fused_clusters = 0;
    c->fused_blocks_per_sm = 0;
    c->last_variant = 0;
    c->persist_clusters = 0;
    c->slice_clusters = 0;
    c->stream_pairs = 0;
    c->persist_max_b = 1;
    c->persist_prefetch_kb = 0;
    for (int l = 0; l < 64; ++l) c->sweep_key[l] = nullptr;
    if (major == 10) { rm_fused_init(c); rm_persist_init(c); rm_slice_init(c); rm_stream_init(c); }   // failure leaves the portable path in charge
    cudaGetLastError();
    *out = c;
    return RM_OK;
}

int rm_destroy(rm_ctx* ctx) {
    if (!ctx) return RM_ERR_INVALID_ARG;
    cudaFree(ctx->d_status);
    delete ctx;
    return RM_OK;
}

size_t rm_packed_layer_bytes(const rm_ctx* ctx) {
    return ctx ? (size_t)ctx->g.I * 3 * ctx->g.H * sizeof(__nv_bfloat16) : 0;
}

size_t rm_workspace_bytes(const rm_ctx* ctx, int B, int T) {
    if (!ctx || B < 1 || T < 1) return 0;
    // three rotating residual-stream buffers, the host variant's staging buffer, then the portable path's scratch
    size_t r_bytes = align_up((size_t)B * T * ctx->g.H * sizeof(float), 256);
    return 4 * r_bytes + align_up(rm_ref_workspace_bytes(ctx, B, T), 256) + align_up(rm_persist_workspace_bytes(ctx), 256) +
           align_up(rm_slice_workspace_bytes(ctx, B, T), 1024) + 1024 + rm_sweep_workspace_bytes(ctx);
}

int rm_pack_weights(rm_ctx* ctx, const void* Wg, const void* Wu, const void* Wd, void* packed_out,
                    float* down_colnorm, rm_stream_t stream) {
    if (!ctx || !Wg || !Wu || !Wd || !packed_out) return RM_ERR_INVALID_ARG;
    if (!all_aligned({Wg, Wu, Wd, packed_out, down_colnorm})) return RM_ERR_ALIGN;
    return rm_launch_pack(ctx, Wg, Wu, Wd, packed_out, down_colnorm, static_cast<cudaStream_t>(stream));
}

int rm_debug_gather_read(rm_ctx* ctx, const void* packed_layer, const int32_t* idx, const int32_t* count_dev,
                         int64_t list_cap, rm_stream_t stream) {
    if (!ctx || !packed_layer || (idx && !count_dev) || list_cap < 0) return RM_ERR_INVALID_ARG;
    if (!all_aligned({packed_layer, idx})) return RM_ERR_ALIGN;
    return rm_launch_gather_read(ctx, packed_layer, idx, count_dev, idx ? list_cap : ctx->g.I,
                                 static_cast<cudaStream_t>(stream));
}

int rm_debug_gather_read_step(rm_ctx* ctx, const void* const* packed_layers, const int32_t* idx, const int32_t* count_dev,
                              int64_t stride, rm_stream_t stream) {
    if (!ctx || !packed_layers || (idx && (!count_dev || stride < 1))) return RM_ERR_INVALID_ARG;
    for (int l = 0; l < ctx->g.L; ++l) {
        if (!packed_layers[l]) return RM_ERR_INVALID_ARG;
        if (!rm_aligned16(packed_layers[l])) return RM_ERR_ALIGN;
    }
    if (!all_aligned({idx})) return RM_ERR_ALIGN;
    return rm_launch_gather_read_step(ctx, packed_layers, idx, count_dev, stride, static_cast<cudaStream_t>(stream));
}

int rm_debug_wait_timeout(rm_ctx* ctx, int polls, rm_stream_t stream) {
    if (!ctx || polls < 1 || polls > (1 << 20)) return RM_ERR_INVALID_ARG;
    return rm_launch_wait_timeout(ctx, (unsigned)polls, static_cast<cudaStream_t>(stream));
}

int rm_gather_weights(rm_ctx* ctx, const void* packed_layer, const int32_t* idx, const int32_t* count_dev,
                      int64_t list_cap, void* compact_out, rm_stream_t stream) {
    if (!ctx || !packed_layer || !idx || !count_dev || !compact_out || list_cap < 0) return RM_ERR_INVALID_ARG;
    if (!all_aligned({packed_layer, idx, compact_out})) return RM_ERR_ALIGN;
    if (compact_out == packed_layer) return RM_ERR_INVALID_ARG;
    return rm_launch_gather_rows(ctx, packed_layer, idx, count_dev, list_cap, compact_out,
                                 static_cast<cudaStream_t>(stream));
}

int rm_context_drift(rm_ctx* ctx, const void* x, const void* x_ref, int P, float* score_out, rm_stream_t stream) {
    if (!ctx || !x || !x_ref || !score_out || P < 0) return RM_ERR_INVALID_ARG;
    if (ctx->g.H % 8 != 0) return RM_ERR_UNSUPPORTED;
    if (!all_aligned({x, x_ref, score_out})) return RM_ERR_ALIGN;
    if (P == 0) return RM_OK;
    return rm_launch_context_drift(ctx, x, x_ref, P, score_out, static_cast<cudaStream_t>(stream));
}

constexpr int RM_CONTEXT_MAX_ROWS = 1024;      // four passes of 256 rows over the weights

size_t rm_context_workspace_bytes(const rm_ctx* ctx, int R_max) {
    if (!ctx || R_max < 1 || R_max > RM_CONTEXT_MAX_ROWS || !rm_context_supported(ctx)) return 0;
    return rm_context_workspace_bytes_impl(ctx, R_max);
}

int rm_context_ffn(rm_ctx* ctx, const void* Wg, const void* Wu, const void* Wd, const void* x, const int32_t* rows,
                   const int32_t* count_dev, int P, int S, int R_max, const float* y_ref, float* y_out, void* ws,
                   size_t ws_bytes, rm_stream_t stream) {
    if (!ctx || !Wg || !Wu || !Wd || !x || !rows || !count_dev || !y_ref || !y_out || P < 0 || S < 0) return RM_ERR_INVALID_ARG;
    if (!rm_context_supported(ctx)) return RM_ERR_UNSUPPORTED;
    if (R_max < 1 || R_max > RM_CONTEXT_MAX_ROWS || S > R_max) return RM_ERR_SHAPE;
    if (!all_aligned({Wg, Wu, Wd, x, rows, y_ref, y_out, ws})) return RM_ERR_ALIGN;
    if (!ws || ws_bytes < rm_context_workspace_bytes(ctx, R_max)) return RM_ERR_WORKSPACE;
    // rows beyond 256 take further passes; the capacity is rounded up to what the passes hold (the rows that this adds are zero)
    return rm_launch_context_ffn(ctx, Wg, Wu, Wd, x, rows, count_dev, P, S, R_max, y_ref, y_out, ws,
                                 static_cast<cudaStream_t>(stream));
}

int rm_mask_compact(rm_ctx* ctx, const rm_mask_src* src, int32_t* idx_out, int32_t* count_out, int64_t stride,
                    rm_stream_t stream) {
    if (!ctx || !src || !idx_out || !count_out || !src->records) return RM_ERR_INVALID_ARG;
    if (src->n_lists < 0 || src->I < 1 || stride < 1) return RM_ERR_INVALID_ARG;
    if (src->n_records < 1 || src->n_records > 16) return RM_ERR_INVALID_ARG;
    if (src->kind == RM_SRC_BOOL_U8) {
        if (src->reduce != RM_REDUCE_NONE) return RM_ERR_INVALID_ARG;
    } else if (src->kind == RM_SRC_SCORE_F32) {
        if (src->reduce != RM_REDUCE_THRESHOLD && src->reduce != RM_REDUCE_TOPK && src->reduce != RM_REDUCE_GROUP)
            return RM_ERR_INVALID_ARG;
    } else {
        return RM_ERR_INVALID_ARG;
    }
    if (src->reduce != RM_REDUCE_GROUP && (src->min_votes < 1 || src->min_votes > src->n_records))
        return RM_ERR_INVALID_ARG;
    if ((src->reduce == RM_REDUCE_TOPK || src->reduce == RM_REDUCE_GROUP) && src->k < 0) return RM_ERR_INVALID_ARG;
    for (int w = 0; w < src->n_records; ++w) {
        if (!src->records[w]) return RM_ERR_INVALID_ARG;
        if (!rm_aligned16(src->records[w])) return RM_ERR_ALIGN;
    }
    if (!all_aligned({idx_out, src->scale})) return RM_ERR_ALIGN;
    if (src->scale && src->kind != RM_SRC_SCORE_F32) return RM_ERR_INVALID_ARG;
    if ((src->reduce == RM_REDUCE_TOPK || src->reduce == RM_REDUCE_GROUP) && src->I == ctx->g.I)
        ctx->count_hint_seen = src->k < src->I ? src->k : src->I;
    return rm_launch_mask_compact(ctx, src, idx_out, count_out, stride, static_cast<cudaStream_t>(stream));
}

int rm_sparse_mlp(rm_ctx* ctx, const void* packed_layer, const void* x, const float* residual, const int32_t* idx,
                  const int32_t* count_dev, float* y, float* record_out, const float* record_scale, int T, void* ws,
                  size_t ws_bytes, rm_stream_t stream) {
    if (!ctx || !packed_layer || !x || !y || T < 0) return RM_ERR_INVALID_ARG;
    if (idx && !count_dev) return RM_ERR_INVALID_ARG;
    if (idx && record_out) return RM_ERR_INVALID_ARG;       // records are emitted by dense passes only
    if (T > ctx->desc.T_max) return RM_ERR_SHAPE;
    if (!all_aligned({packed_layer, x, residual, idx, y, record_out, record_scale, ws})) return RM_ERR_ALIGN;
    if (T == 0) return RM_OK;
    if (!ws || ws_bytes < rm_workspace_bytes(ctx, 1, T)) return RM_ERR_WORKSPACE;
    rm_layer_args a{};
    a.packed = static_cast<const __nv_bfloat16*>(packed_layer);
    a.x = static_cast<const __nv_bfloat16*>(x);
    a.r_in = residual;
    a.r_out = y;
    a.idx = idx;
    a.count = count_dev;
    a.idx_stride = ctx->g.I;
    a.list_cap = ctx->g.I;
    a.count_stride = 1;
    a.record = record_out;
    a.record_stride = ctx->g.I;
    a.record_scale = record_scale;
    a.B = 1;
    a.T = T;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t r_bytes = align_up((size_t)T * ctx->g.H * sizeof(float), 256);
    if (use_slice(ctx, 1, T, record_out != nullptr)) {
        const void* one[1] = {packed_layer};
        rm_step_args sa{};
        sa.packed_layers = one;
        sa.L = 1;
        sa.r = y;
        sa.r_in = residual;
        sa.idx = idx;
        sa.count = count_dev;
        sa.list_cap = ctx->g.I;
        sa.record = record_out;
        sa.record_scale = record_scale;
        sa.B = 1;
        sa.T = T;
        sa.x_ext = x;
        slice_buffers(ctx, sa, ws, 1, T);
        ctx->last_variant = 6;
        return rm_launch_step_slice(ctx, sa, s);
    }
    if (use_fused(ctx, 1, T)) {
        // y accumulates the CTAs' partial sums with atomics: start it from the residual (or zero)
        // (a kernel of its own, so that the layer's CTAs can set up and gather their first weights while it runs)
        if (y != residual) {
            const int rc = rm_launch_copy(ctx, y, residual, nullptr, (size_t)T * ctx->g.H, s);
            if (rc != RM_OK) return rc;
        }
        if (use_persist(ctx, 1, T, count_dev != nullptr, false, false)) {
            // the whole-step kernel on a stack of one layer whose input is the caller's x
            const void* one[1] = {packed_layer};
            rm_step_args sa{};
            sa.packed_layers = one;
            sa.L = 1;
            sa.r = y;
            sa.idx = idx;
            sa.count = count_dev;
            sa.idx_b_stride = 0;
            sa.idx_l_stride = 0;
            sa.list_cap = ctx->g.I;
            sa.count_b_stride = 0;
            sa.record = record_out;
            sa.rec_b_stride = 0;
            sa.record_scale = record_scale;
            sa.B = 1;
            sa.T = T;
            sa.x_ext = x;
            ctx->last_variant = 5;
            return rm_launch_step_persist(ctx, sa, nullptr, s);      // (the workspace stays untouched, as by the layer kernels)
        }
        if (use_stream(ctx, count_dev != nullptr, 1, T, RM_ANCHOR_NONE, false, false)) {
            ctx->last_variant = 4;
            return rm_launch_layer_stream(ctx, a, nullptr, y == residual, s);
        }
        return rm_launch_layer_fused(ctx, a, nullptr, false, ctx->use_pdl && y != residual, s);
    }
    if (ctx->path == 2) return RM_ERR_UNSUPPORTED;
    ctx->last_variant = 0;
    return rm_launch_layer_ref(ctx, a, static_cast<char*>(ws) + 4 * r_bytes, s);
}

namespace {
struct AnchorIO {                      // whole-stack anchor state (Eq. 4); mode RM_ANCHOR_NONE and NULLs for none
    int mode = RM_ANCHOR_NONE;
    float* y = nullptr;                // [L,B,T,H]
    float* h = nullptr;                // [L,B,I,h_stride]
    int64_t h_stride = 0;
    const float* gate = nullptr;       // [L,B,H]
};
}  // namespace

static int step_device(rm_ctx* ctx, const void* const* packed_layers, const float* r_in, const int32_t* idx,
                       const int32_t* count_dev, int64_t stride, float* r_out, float* records_out,
                       const float* record_scale, int B, int T, void* ws, cudaStream_t s,
                       const AnchorIO& an = AnchorIO(), const float** result = nullptr) {
    // `result` (or NULL): where the output is, instead of a copy into r_out when the step runs in place
    const rm_geom& g = ctx->g;
    const size_t n_bytes = (size_t)B * T * g.H * sizeof(float);
    const size_t r_bytes = align_up(n_bytes, 256);
    if (result) *result = r_out;
    char* layer_ws = static_cast<char*>(ws) + 4 * r_bytes;
    const bool slice = use_slice(ctx, B, T, records_out != nullptr);
    const bool sweep = !slice && use_sweep(ctx, B, T, !idx && !count_dev && an.mode != RM_ANCHOR_UPDATE);
    if (slice || sweep || use_persist(ctx, B, T, count_dev != nullptr, an.mode != RM_ANCHOR_NONE || an.gate, true)) {
        // the whole step in one launch: the layers add into r_out in place (the kernel starts it as a copy of r_in)
        rm_step_args sa{};
        sa.packed_layers = packed_layers;
        sa.L = g.L;
        sa.r = r_out;
        sa.r_in = r_out != r_in ? r_in : nullptr;
        sa.idx = idx;
        sa.count = count_dev;
        sa.idx_b_stride = (int64_t)g.L * stride;
        sa.idx_l_stride = stride;
        sa.list_cap = idx ? stride : g.I;
        sa.count_b_stride = g.L;
        sa.record = records_out;
        sa.rec_b_stride = (int64_t)g.L * g.I;
        sa.record_scale = record_scale;
        sa.B = B;
        sa.T = T;
        sa.anchor_mode = an.mode;
        sa.y_anchor = an.y;
        sa.h_anchor = an.h;
        sa.h_stride = an.h_stride;
        sa.gate = an.gate;
        if (sweep) {
            ctx->last_variant = 7;
            return rm_launch_step_sweep(ctx, sa, sweep_ws(ctx, ws, B, T), s);
        }
        if (slice) {
            slice_buffers(ctx, sa, ws, B, T);
            ctx->last_variant = 6;
            return rm_launch_step_slice(ctx, sa, s);
        }
        ctx->last_variant = 5;
        return rm_launch_step_persist(ctx, sa, persist_ws(ctx, ws, B, T), s);
    }
    const bool fused = use_fused(ctx, B, T);
    if (!fused && ctx->path == 2) return RM_ERR_UNSUPPORTED;
    float* rot[3] = {reinterpret_cast<float*>(static_cast<char*>(ws)),
                     reinterpret_cast<float*>(static_cast<char*>(ws) + r_bytes),
                     reinterpret_cast<float*>(static_cast<char*>(ws) + 2 * r_bytes)};
    // Fused path: layer l reads rot[l%3] (the caller's r_in for l = 0), accumulates into rot[(l+1)%3] and clears
    // rot[(l+2)%3] for the layer after next; the last layer accumulates straight into r_out when that is a
    // different buffer from r_in.
    const bool stream = fused && use_stream(ctx, count_dev != nullptr, B, T, an.mode,
                                             an.mode != RM_ANCHOR_NONE || an.gate);
    const bool direct_out = fused && r_out != r_in;
    if (fused && !stream) {
        const int rc = rm_launch_copy(ctx, g.L == 1 && direct_out ? r_out : rot[1], nullptr, direct_out && g.L > 1 ? r_out : nullptr,
                                      n_bytes / sizeof(float), s);
        if (rc != RM_OK) return rc;
    }
    // the anchor step's outputs are accumulated by the CTAs' atomics: start them from zero
    if (fused && an.mode == RM_ANCHOR_WRITE)
        RM_CUDA_TRY(cudaMemsetAsync(an.y, 0, (size_t)g.L * n_bytes, s));
    const float* cur = r_in;
    for (int l = 0; l < g.L; ++l) {
        rm_layer_args a{};
        a.packed = static_cast<const __nv_bfloat16*>(packed_layers[l]);
        a.x = nullptr;
        a.r_in = cur;
        a.idx = idx ? idx + (size_t)l * stride : nullptr;
        a.count = count_dev ? count_dev + l : nullptr;
        a.idx_stride = (int64_t)g.L * stride;
        a.list_cap = idx ? stride : g.I;
        a.count_stride = g.L;
        a.record = records_out ? records_out + (size_t)l * g.I : nullptr;
        a.record_stride = (int64_t)g.L * g.I;
        a.record_scale = record_scale ? record_scale + (size_t)l * g.I : nullptr;
        a.B = B;
        a.T = T;
        a.anchor_mode = an.mode;
        a.y_anchor = an.y ? an.y + (size_t)l * B * T * g.H : nullptr;
        a.h_anchor = an.h ? an.h + (size_t)l * B * g.I * an.h_stride : nullptr;
        a.h_stride = an.h_stride;
        a.gate = an.gate ? an.gate + (size_t)l * B * g.H : nullptr;
        int rc;
        if (stream) {
            // two buffers in turn: the preparation kernel writes the residual part of the output, the tiles add theirs
            const bool last = l == g.L - 1;
            a.r_out = (last && direct_out) ? r_out : rot[l & 1];
            ctx->last_variant = 4;
            rc = rm_launch_layer_stream(ctx, a, reinterpret_cast<__nv_bfloat16*>(layer_ws), l == 0, s);
            cur = a.r_out;
        } else if (fused) {
            const bool last = l == g.L - 1;
            a.r_out = (last && direct_out) ? r_out : rot[(l + 1) % 3];
            // the buffer cleared here is the output of layer l+1 (unless that layer writes to r_out directly); it
            // was the input of layer l-1, which has completed by the time this layer passes its dependency wait
            float* zero = (l + 1 < g.L && !(l + 1 == g.L - 1 && direct_out)) ? rot[(l + 2) % 3] : nullptr;
            rc = rm_launch_layer_fused(ctx, a, zero, true, ctx->use_pdl && (l > 0 || an.mode != RM_ANCHOR_WRITE), s);
            cur = a.r_out;
        } else {
            a.r_out = r_out;                               // in place after the first layer
            ctx->last_variant = 0;
            rc = rm_launch_layer_ref(ctx, a, layer_ws, s);
            cur = r_out;
        }
        if (rc != RM_OK) return rc;
    }
    if (result) *result = cur;
    else if (fused && !direct_out) return rm_launch_copy(ctx, r_out, cur, nullptr, n_bytes / sizeof(float), s);
    return RM_OK;
}

int rm_action_expert_step(rm_ctx* ctx, const void* const* packed_layers, const float* r_in, const int32_t* idx,
                          const int32_t* count_dev, int64_t stride, float* r_out, float* records_out,
                          const float* record_scale, int B, int T, void* ws, size_t ws_bytes, rm_stream_t stream) {
    if (!ctx || !packed_layers || !r_in || !r_out || B < 0 || T < 0) return RM_ERR_INVALID_ARG;
    if (idx && (!count_dev || stride < 1)) return RM_ERR_INVALID_ARG;
    if (idx && records_out) return RM_ERR_INVALID_ARG;
    if (B > ctx->desc.B_max || T > ctx->desc.T_max) return RM_ERR_SHAPE;
    for (int l = 0; l < ctx->g.L; ++l) {
        if (!packed_layers[l]) return RM_ERR_INVALID_ARG;
        if (!rm_aligned16(packed_layers[l])) return RM_ERR_ALIGN;
    }
    if (!all_aligned({r_in, idx, r_out, records_out, record_scale, ws})) return RM_ERR_ALIGN;
    if (idx && (stride % 4) != 0) return RM_ERR_ALIGN;       // every list must start 16-byte aligned
    if (B == 0 || T == 0) return RM_OK;
    if (!ws || ws_bytes < rm_workspace_bytes(ctx, B, T)) return RM_ERR_WORKSPACE;
    return step_device(ctx, packed_layers, r_in, idx, count_dev, stride, r_out, records_out, record_scale, B, T, ws,
                       static_cast<cudaStream_t>(stream));
}

int rm_action_expert_step_ex(rm_ctx* ctx, const void* const* packed_layers, const float* r_in, const int32_t* idx,
                             const int32_t* count_dev, int64_t stride, float* r_out, float* records_out,
                             const float* record_scale, int B, int T, int anchor_mode, float* y_anchor,
                             float* h_anchor, int64_t h_stride, const float* out_gate, void* ws, size_t ws_bytes,
                             rm_stream_t stream) {
    if (!ctx || !packed_layers || !r_in || !r_out || B < 0 || T < 0) return RM_ERR_INVALID_ARG;
    if (idx && (!count_dev || stride < 1)) return RM_ERR_INVALID_ARG;
    if (idx && records_out) return RM_ERR_INVALID_ARG;
    if (anchor_mode != RM_ANCHOR_NONE && anchor_mode != RM_ANCHOR_WRITE && anchor_mode != RM_ANCHOR_UPDATE)
        return RM_ERR_INVALID_ARG;
    if (anchor_mode != RM_ANCHOR_NONE) {
        if (!y_anchor || !h_anchor || h_stride < T) return RM_ERR_INVALID_ARG;
        if (h_stride % 4 != 0) return RM_ERR_ALIGN;
        // the anchor state is read (or accumulated) while the outputs are written: no overlap with them
        if (y_anchor == r_out || y_anchor == r_in) return RM_ERR_INVALID_ARG;
    }
    if (B > ctx->desc.B_max || T > ctx->desc.T_max) return RM_ERR_SHAPE;
    for (int l = 0; l < ctx->g.L; ++l) {
        if (!packed_layers[l]) return RM_ERR_INVALID_ARG;
        if (!rm_aligned16(packed_layers[l])) return RM_ERR_ALIGN;
    }
    if (!all_aligned({r_in, idx, r_out, records_out, record_scale, ws, y_anchor, h_anchor, out_gate}))
        return RM_ERR_ALIGN;
    if (idx && (stride % 4) != 0) return RM_ERR_ALIGN;
    if (B == 0 || T == 0) return RM_OK;
    if (!ws || ws_bytes < rm_workspace_bytes(ctx, B, T)) return RM_ERR_WORKSPACE;
    AnchorIO an;
    an.mode = anchor_mode;
    if (anchor_mode != RM_ANCHOR_NONE) { an.y = y_anchor; an.h = h_anchor; an.h_stride = h_stride; }
    an.gate = out_gate;
    return step_device(ctx, packed_layers, r_in, idx, count_dev, stride, r_out, records_out, record_scale, B, T, ws,
                       static_cast<cudaStream_t>(stream), an);
}

// The device's address of a pinned host buffer, or NULL (pageable, not host memory, or not 16-byte aligned)
static void* pinned_device_pointer(const void* p, size_t bytes) {
    cudaPointerAttributes first, last;
    if (!rm_aligned16(p) || cudaPointerGetAttributes(&first, p) != cudaSuccess ||
        cudaPointerGetAttributes(&last, static_cast<const char*>(p) + bytes - 1) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    const bool whole = first.type == cudaMemoryTypeHost && last.type == cudaMemoryTypeHost && first.devicePointer &&
                       static_cast<char*>(last.devicePointer) - static_cast<char*>(first.devicePointer) == (ptrdiff_t)(bytes - 1);
    return whole && rm_aligned16(first.devicePointer) ? first.devicePointer : nullptr;
}

int rm_action_expert_step_host(rm_ctx* ctx, const void* const* packed_layers, const float* r_in_host,
                               const int32_t* idx, const int32_t* count_dev, int64_t stride, float* r_out_host, int B,
                               int T, void* ws, size_t ws_bytes, rm_stream_t stream) {
    if (!ctx || !packed_layers || !r_in_host || !r_out_host || B < 0 || T < 0) return RM_ERR_INVALID_ARG;
    if (idx && (!count_dev || stride < 1)) return RM_ERR_INVALID_ARG;
    if (B > ctx->desc.B_max || T > ctx->desc.T_max) return RM_ERR_SHAPE;
    for (int l = 0; l < ctx->g.L; ++l) {
        if (!packed_layers[l]) return RM_ERR_INVALID_ARG;
        if (!rm_aligned16(packed_layers[l])) return RM_ERR_ALIGN;
    }
    if (!all_aligned({idx, ws})) return RM_ERR_ALIGN;
    if (idx && (stride % 4) != 0) return RM_ERR_ALIGN;
    if (B == 0 || T == 0) return RM_OK;
    if (!ws || ws_bytes < rm_workspace_bytes(ctx, B, T)) return RM_ERR_WORKSPACE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t n_bytes = (size_t)B * T * ctx->g.H * sizeof(float);
    // the fourth residual-stream buffer of the workspace is the staging copy
    float* stage = reinterpret_cast<float*>(static_cast<char*>(ws) + 3 * align_up(n_bytes, 256));
    // pinned buffers are copied by a kernel (rm_launch_copy), others by the copy engine
    const float* in_dev = static_cast<const float*>(pinned_device_pointer(r_in_host, n_bytes));
    float* out_dev = static_cast<float*>(pinned_device_pointer(r_out_host, n_bytes));
    if (in_dev) {
        const int rc = rm_launch_copy(ctx, stage, in_dev, nullptr, n_bytes / sizeof(float), s);
        if (rc != RM_OK) return rc;
    } else {
        RM_CUDA_TRY(cudaMemcpyAsync(stage, r_in_host, n_bytes, cudaMemcpyHostToDevice, s));
    }
    const float* out = nullptr;
    int rc = step_device(ctx, packed_layers, stage, idx, count_dev, stride, stage, nullptr, nullptr, B, T, ws, s, AnchorIO(), &out);
    if (rc != RM_OK) return rc;
    if (out_dev) {
        rc = rm_launch_copy(ctx, out_dev, out, nullptr, n_bytes / sizeof(float), s);
        if (rc != RM_OK) return rc;
    } else {
        RM_CUDA_TRY(cudaMemcpyAsync(r_out_host, out, n_bytes, cudaMemcpyDeviceToHost, s));
    }
    RM_CUDA_TRY(cudaStreamSynchronize(s));
    return RM_OK;
}

int rm_device_status(rm_ctx* ctx, int* host_out, rm_stream_t stream) {
    if (!ctx || !host_out) return RM_ERR_INVALID_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int v[RM_STATUS_INTS] = {0};
    RM_CUDA_TRY(cudaMemcpyAsync(v, ctx->d_status, sizeof(v), cudaMemcpyDeviceToHost, s));
    RM_CUDA_TRY(cudaMemsetAsync(ctx->d_status, 0, sizeof(v), s));
    RM_CUDA_TRY(cudaStreamSynchronize(s));
    *host_out = v[0];
    ctx->status_detail = v[0] ? v[1] : 0;
    std::memcpy(ctx->status_log, v, sizeof(v));
    return RM_OK;
}

int64_t rm_launch_count(const rm_ctx* ctx) { return ctx ? ctx->launches : 0; }

int rm_set_option(rm_ctx* ctx, const char* name, int value) {
    if (!ctx || !name) return RM_ERR_INVALID_ARG;
    const std::string n(name);
    if (n == "path") {
        if (value < 0 || value > 2) return RM_ERR_INVALID_ARG;
        ctx->path = value;
    } else if (n == "pdl") {
        ctx->use_pdl = value != 0;
    } else if (n == "neurons_per_cluster") {
        if (value < 1) return RM_ERR_INVALID_ARG;
        ctx->npc_target = value;
    } else if (n == "count_hint") {
        if (value < 0) return RM_ERR_INVALID_ARG;
        ctx->count_hint = value;
    } else if (n == "variant") {
        if (value < 0 || value > 7) return RM_ERR_INVALID_ARG;
        ctx->variant_override = value;
    } else if (n == "persist_prefetch_kb") {
        if (value < 0 || value > 4096) return RM_ERR_INVALID_ARG;
        ctx->persist_prefetch_kb = value;
    } else if (n == "persist_max_batch") {
        if (value < 0 || value > 16) return RM_ERR_INVALID_ARG;
        ctx->persist_max_b = value;
    } else if (n == "stream_min_tiles") {
        if (value < 1) return RM_ERR_INVALID_ARG;
        ctx->stream_min_tiles = value;
    } else if (n == "l2_prefetch") {
        if (value < 0 || value > 16) return RM_ERR_INVALID_ARG;
        ctx->l2_prefetch = value;
    } else if (n == "max_clusters") {
        if (value < 0) return RM_ERR_INVALID_ARG;
        ctx->max_clusters_override = value;
    } else {
        return RM_ERR_INVALID_ARG;
    }
    return RM_OK;
}

int rm_get_info(const rm_ctx* ctx, const char* name, int* out) {
    if (!name || !out) return RM_ERR_INVALID_ARG;
    const std::string n(name);
    if (n == "last_cuda_error") { *out = rm_last_cuda_error; return RM_OK; }   // process-wide: needs no context
    if (!ctx) return RM_ERR_INVALID_ARG;
    if (n == "fused_clusters") *out = ctx->fused_clusters;
    else if (n == "fused_blocks_per_sm") *out = ctx->fused_blocks_per_sm;
    else if (n == "sm_count") *out = ctx->sm_count;
    else if (n == "persist_clusters") *out = ctx->persist_clusters;
    else if (n == "stream_pairs") *out = ctx->stream_pairs;
    else if (n == "slice_clusters") *out = ctx->slice_clusters;
    else if (n == "last_variant") *out = ctx->last_variant;
    else if (n == "path") *out = ctx->path;
    else if (n == "status_detail") *out = ctx->status_detail;
    else if (n == "status_log_count") *out = ctx->status_log[2] < RM_STATUS_LOG ? ctx->status_log[2] : RM_STATUS_LOG;
    else if (n.rfind("status_log:", 0) == 0) {
        const int i = std::atoi(n.c_str() + 11);
        if (i < 0 || i >= RM_STATUS_LOG) return RM_ERR_INVALID_ARG;
        *out = ctx->status_log[4 + i];
    }
    else return RM_ERR_INVALID_ARG;
    return RM_OK;
}

int rm_debug_phase_times(rm_ctx* ctx, long long* host_out, int n) {
    if (!ctx || !host_out) return RM_ERR_INVALID_ARG;
    if (n == -64) return rm_stream_debug_stamps(host_out);      // the streaming kernel's stamps (first tile of CTA 0)
    if (n <= -(1 << 20)) return rm_persist_debug_stamps(host_out, -n - (1 << 20));   // the whole-step kernel's stamps
    return rm_fused_debug_stamps(host_out, n);
}

const char* rm_status_string(int status) {
    switch (status) {
        case RM_OK: return "ok";
        case RM_ERR_INVALID_ARG: return "invalid argument";
        case RM_ERR_SHAPE: return "shape outside the context's limits";
        case RM_ERR_ALIGN: return "pointer not 16-byte aligned";
        case RM_ERR_WORKSPACE: return "workspace missing or too small";
        case RM_ERR_CUDA: return "CUDA runtime error";
        case RM_ERR_INDEX: return "neuron index out of range or count exceeds stride";
        case RM_ERR_TIMEOUT: return "bounded device wait expired";
        case RM_ERR_UNSUPPORTED: return "not supported by this build";
        default: return "unknown status";
    }
}

}  // extern "C"

// pc_attend_frame and the prepare / prepared pair: argument checks and the choice of attention kernel.
#include "pc_common.cuh"

namespace {

constexpr int STEP_TILE = 128;        // rows of the rotated-key scratch start on multiples of this

// anchors ++ history ++ current, empty segments dropped
pc_status gather_segments(pc_ctx *ctx, const pc_cache *cache, const pc_segment *current, pc_segment *segs, int *n_seg) {
    *n_seg = 0;
    int64_t n_keys = 0;
    const pc_segment *cand[3] = {&cache->anchors, &cache->history, current};
    for (int i = 0; i < 3; ++i) {
        if (!cand[i]) continue;
        pc_status st = pc_check_segment(cand[i], true);
        if (st != PC_OK) return st;
        if (cand[i]->n_tokens == 0) continue;
        segs[(*n_seg)++] = *cand[i];
        n_keys += cand[i]->n_tokens;
    }
    if (n_keys == 0) return PC_ERR_INVALID_ARG;
    if (n_keys > ctx->desc.max_keys) return PC_ERR_CAPACITY;
    return PC_OK;
}

pc_status check_queries(pc_ctx *ctx, const void *q, const int32_t *q_pos, int32_t n_q, const void *out, const float *lse) {
    if (!q || !q_pos || !out || n_q <= 0) return PC_ERR_INVALID_ARG;
    if (!pc_aligned16(q) || !pc_aligned16(q_pos) || !pc_aligned16(out) || (lse && !pc_aligned16(lse))) return PC_ERR_INVALID_ARG;
    if (n_q > ctx->desc.max_q) return PC_ERR_CAPACITY;
    return PC_OK;
}

bool tensor_core_path(const pc_ctx *ctx) {
    return ctx->attend_impl != 1 && pc_tensor_core_shape(ctx);
}

// Tensor-core attention of all n_q rows, the output in parts if somebody waits for them.  `what` holds what is still to be rotated.
pc_status attend_tc(pc_ctx *ctx, int n_seg, const pc_segment *segs, const void *q, const int32_t *q_pos, int32_t n_q, void *out,
                    float *lse, cudaStream_t stream, int what, const pc_step_hooks *hooks) {
    const int part = hooks ? pc_attend_part_rows(ctx, n_q) : n_q;
    if (part >= n_q) {
        const pc_status st = pc_launch_attend_tc(ctx, n_seg, segs, q, q_pos, n_q, out, lse, stream, what);
        return st == PC_OK && hooks ? hooks->part_done(hooks->self, 0, n_q, stream) : st;
    }
    pc_status st = pc_launch_attend_tc(ctx, n_seg, segs, q, q_pos, n_q, out, lse, stream, what & ~PC_TC_ATTEND);
    const size_t row_bytes = (size_t)ctx->desc.n_q_heads * ctx->desc.head_dim * ctx->elem_size;
    for (int r = 0; r < n_q && st == PC_OK; r += part) {
        const int n = part < n_q - r ? part : n_q - r;
        st = pc_launch_attend_tc(ctx, n_seg, segs, nullptr, nullptr, n, static_cast<char *>(out) + r * row_bytes,
                                 lse ? lse + (size_t)r * ctx->desc.n_q_heads : nullptr, stream, PC_TC_ATTEND | PC_TC_GOES_ON, r);
        if (st == PC_OK) st = hooks->part_done(hooks->self, r, n, stream);
    }
    if (st == PC_OK) ctx->last_n_q = n_q;
    return st;
}

pc_status attend_simt(pc_ctx *ctx, int n_seg, const pc_segment *segs, const void *q, const int32_t *q_pos, int32_t n_q, void *out,
                      float *lse, cudaStream_t stream, const pc_step_hooks *hooks) {
    const pc_status st = pc_launch_attend_simt(ctx, n_seg, segs, q, q_pos, n_q, out, lse, stream);
    return st == PC_OK && hooks ? hooks->part_done(hooks->self, 0, n_q, stream) : st;
}

// The checks of a fused step up to the pack stage (scoring has its own): what the pack stage would refuse (a destination that
// overlaps the source, a misaligned or missing buffer) is refused before the scoring stage enqueues anything.
pc_status check_frame_step(pc_ctx *ctx, const pc_cache *src, const int32_t *budget, const pc_cache *dst, const void *q, const int32_t *q_pos,
                           int32_t n_q, const int32_t *sel_idx, const void *out, const float *lse, int64_t *n_sel_out) {
    if (!ctx || !src || !dst || !budget) return PC_ERR_INVALID_ARG;
    pc_status st = check_queries(ctx, q, q_pos, n_q, out, lse);
    if (st != PC_OK) return st;
    if (src->n_frames < 0 || (src->n_frames > 0 && !src->frame_count)) return PC_ERR_INVALID_ARG;
    int64_t n_sel = 0;
    for (int f = 0; f < src->n_frames; ++f) {
        if (budget[f] < 0) return PC_ERR_INVALID_ARG;
        n_sel += budget[f];
    }
    if (n_sel > dst->history.capacity) return PC_ERR_CAPACITY;
    st = pc_check_segment(&src->anchors, true);
    if (st != PC_OK) return st;
    const int n_anchor = src->anchors.n_tokens;
    if (n_anchor + n_sel == 0) return PC_ERR_INVALID_ARG;
    if (n_anchor + n_sel > ctx->desc.max_keys) return PC_ERR_CAPACITY;
    if (tensor_core_path(ctx) && (size_t)((n_anchor + STEP_TILE - 1) / STEP_TILE + (n_sel + STEP_TILE - 1) / STEP_TILE) * STEP_TILE > ctx->k_rot_rows)
        return PC_ERR_CAPACITY;
    *n_sel_out = n_sel;
    return pc_compact_check(ctx, src, sel_idx, budget, dst, nullptr, nullptr);
}

}  // namespace

pc_status pc_attend_frame_check(pc_ctx *ctx, const pc_cache *cache, const pc_segment *current, const void *q, const int32_t *q_pos,
                                int32_t n_q, const void *out, const float *lse) {
    if (!ctx || !cache) return PC_ERR_INVALID_ARG;
    const pc_status st = check_queries(ctx, q, q_pos, n_q, out, lse);
    if (st != PC_OK) return st;
    pc_segment segs[PC_MAX_SEGMENTS];
    int n_seg = 0;
    return gather_segments(ctx, cache, current, segs, &n_seg);
}

pc_status pc_frame_step_check(pc_ctx *ctx, const pc_cache *src, const int32_t *budget, const pc_cache *dst, const void *q, const int32_t *q_pos,
                              int32_t n_q, const float *scores, const int32_t *sel_idx, const void *out, const float *lse) {
    int64_t n_sel = 0;
    const pc_status st = check_frame_step(ctx, src, budget, dst, q, q_pos, n_q, sel_idx, out, lse, &n_sel);
    return st != PC_OK ? st : pc_score_check(ctx, src, q, q_pos, n_q, budget, nullptr, scores, sel_idx);
}

pc_status pc_attend_frame_impl(pc_ctx *ctx, const pc_cache *cache, const pc_segment *current, const void *q, const int32_t *q_pos,
                               int32_t n_q, void *out, float *lse, cudaStream_t stream, const pc_step_hooks *hooks) {
    if (!ctx || !cache) return PC_ERR_INVALID_ARG;
    pc_status st = check_queries(ctx, q, q_pos, n_q, out, lse);
    if (st != PC_OK) return st;
    pc_segment segs[PC_MAX_SEGMENTS];
    int n_seg = 0;
    st = gather_segments(ctx, cache, current, segs, &n_seg);
    if (st != PC_OK) return st;
    if (hooks && hooks->kv_ready) PC_CUDA_TRY(cudaStreamWaitEvent(stream, hooks->kv_ready, 0));
    ctx->last_n_q = 0;
    if (tensor_core_path(ctx)) {
        ctx->prepared_n_seg = 0;                       // the rotated-key scratch is about to be overwritten
        ctx->anchor_rot_n = 0;
        return attend_tc(ctx, n_seg, segs, q, q_pos, n_q, out, lse, stream, PC_TC_ALL, hooks);
    }
    return attend_simt(ctx, n_seg, segs, q, q_pos, n_q, out, lse, stream, hooks);
}

extern "C" pc_status pc_attend_frame(pc_ctx *ctx, const pc_cache *cache, const pc_segment *current, const void *q,
                                     const int32_t *q_pos, int32_t n_q, void *out, float *lse, void *stream) {
    return pc_attend_frame_impl(ctx, cache, current, q, q_pos, n_q, out, lse, static_cast<cudaStream_t>(stream), nullptr);
}

extern "C" pc_status pc_attend_prepare(pc_ctx *ctx, const pc_cache *cache, const pc_segment *current, void *stream_) {
    if (!ctx || !cache) return PC_ERR_INVALID_ARG;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    pc_segment segs[PC_MAX_SEGMENTS];
    int n_seg = 0;
    pc_status st = gather_segments(ctx, cache, current, segs, &n_seg);
    if (st != PC_OK) return st;
    ctx->prepared_n_seg = 0;
    ctx->last_n_q = 0;
    if (tensor_core_path(ctx)) {
        ctx->anchor_rot_n = 0;
        st = pc_launch_attend_tc(ctx, n_seg, segs, nullptr, nullptr, 0, nullptr, nullptr, stream, PC_TC_ROPE_K);
        if (st != PC_OK) return st;
    }
    for (int i = 0; i < n_seg; ++i) ctx->prepared_seg[i] = segs[i];
    ctx->prepared_n_seg = n_seg;
    return PC_OK;
}

extern "C" pc_status pc_attend_prepared(pc_ctx *ctx, const void *q, const int32_t *q_pos, int32_t n_q, void *out, float *lse,
                                        void *stream_) {
    if (!ctx) return PC_ERR_INVALID_ARG;
    if (ctx->prepared_n_seg <= 0) return PC_ERR_INVALID_ARG;      // no key set prepared (or overwritten since)
    pc_status st = check_queries(ctx, q, q_pos, n_q, out, lse);
    if (st != PC_OK) return st;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    ctx->last_n_q = 0;
    if (tensor_core_path(ctx))
        return pc_launch_attend_tc(ctx, ctx->prepared_n_seg, ctx->prepared_seg, q, q_pos, n_q, out, lse, stream,
                                   PC_TC_ROPE_Q | PC_TC_ATTEND);
    return pc_launch_attend_simt(ctx, ctx->prepared_n_seg, ctx->prepared_seg, q, q_pos, n_q, out, lse, stream);
}

// One frame of the steady state in one call: score -> select -> pack -> attend over anchors ++ packed history.  On the
// tensor-core path the intermediate passes of the separate calls disappear: the query pass that pools for the scores also
// leaves the rotated queries, the pack kernel also leaves the rotated keys of what it packs, and the anchors' rotated
// keys stay in the scratch from the first step that saw them, so attention starts without a rotary pre-pass.
pc_status pc_frame_step_impl(pc_ctx *ctx, const pc_cache *src, const int32_t *budget, int32_t delta_t, pc_cache *dst, const void *q,
                             const int32_t *q_pos, int32_t n_q, float *scores, int32_t *sel_idx, void *out, float *lse,
                             cudaStream_t stream, const pc_step_hooks *hooks) {
    int64_t n_sel = 0;
    pc_status st = check_frame_step(ctx, src, budget, dst, q, q_pos, n_q, sel_idx, out, lse, &n_sel);
    if (st != PC_OK) return st;
    const int n_anchor = src->anchors.n_tokens;
    const bool tc = tensor_core_path(ctx);
    void *k_rot_dst = nullptr;
    if (tc) {
        const size_t row_bytes = (size_t)ctx->desc.n_kv_heads * ctx->desc.head_dim * sizeof(__nv_bfloat16);
        k_rot_dst = static_cast<char *>(ctx->k_rot) + (size_t)((n_anchor + STEP_TILE - 1) / STEP_TILE) * STEP_TILE * row_bytes;
        ctx->prepared_n_seg = 0;                       // the scratch no longer holds a key set of pc_attend_prepare
    }
    // (with values still on their way the selection need not wait for them; stage marks tell the two stages apart)
    const bool on_the_way = hooks && hooks->kv_ready;
    const bool one_launch = !on_the_way && !ctx->timing_on && pc_select_pack_fits(ctx, src, budget);
    ctx->last_n_q = 0;
    ctx->q_rot_n = 0;
    pc_front_args args{src, budget, nullptr, scores, sel_idx, delta_t, &dst->history, k_rot_dst, {}};
    const pc_front_args *front = !on_the_way && n_sel > 0 && pc_front_fits(ctx, src, true, &args.plan) ? &args : nullptr;
    st = pc_score_impl(ctx, src, q, q_pos, n_q, budget, nullptr, nullptr, scores, sel_idx, tc ? ctx->q_rot : nullptr, stream, !one_launch, front);
    if (st != PC_OK) return st;
    if (on_the_way) PC_CUDA_TRY(cudaStreamWaitEvent(stream, hooks->kv_ready, 0));
    if (!front)
        st = one_launch ? pc_launch_select_pack(ctx, scores, src, budget, delta_t, &dst->history, sel_idx, k_rot_dst, stream)
                    : pc_compact_impl(ctx, src, sel_idx, budget, delta_t, dst, k_rot_dst, stream);
    if (st != PC_OK) return st;
    dst->history.n_tokens = (int32_t)n_sel;
    dst->n_frames = src->n_frames;

    pc_segment segs[PC_MAX_SEGMENTS];
    int n_seg = 0;
    if (n_anchor > 0) segs[n_seg++] = src->anchors;
    if (n_sel > 0) segs[n_seg++] = dst->history;
    if (!tc) return attend_simt(ctx, n_seg, segs, q, q_pos, n_q, out, lse, stream, hooks);
    int what = PC_TC_ATTEND;
    if (ctx->q_rot_n != n_q) what |= PC_TC_ROPE_Q;    // nothing was scored, so no query pass ran: rotate the queries now
    const bool anchors_cached = n_anchor > 0 && ctx->anchor_rot_n == n_anchor && ctx->anchor_rot_k == src->anchors.k &&
                                ctx->anchor_rot_pos == src->anchors.pos;
    if (n_anchor > 0 && !anchors_cached) what |= PC_TC_ROPE_K0;
    ctx->anchor_rot_n = 0;
    st = attend_tc(ctx, n_seg, segs, q, q_pos, n_q, out, lse, stream, what, hooks);
    if (st != PC_OK) return st;
    if (n_anchor > 0) {
        ctx->anchor_rot_k = src->anchors.k;
        ctx->anchor_rot_pos = src->anchors.pos;
        ctx->anchor_rot_n = n_anchor;
    }
    return PC_OK;
}

extern "C" pc_status pc_frame_step(pc_ctx *ctx, const pc_cache *src, const int32_t *budget, int32_t delta_t, pc_cache *dst,
                                   const void *q, const int32_t *q_pos, int32_t n_q, float *scores, int32_t *sel_idx, void *out,
                                   float *lse, void *stream) {
    return pc_frame_step_impl(ctx, src, budget, delta_t, dst, q, q_pos, n_q, scores, sel_idx, out, lse, static_cast<cudaStream_t>(stream),
                              nullptr);
}

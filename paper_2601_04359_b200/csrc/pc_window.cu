// Cache window: the Fill / Pack / Slide regimes (Sec. 3.4, Fig. 6) and the temporal rebase (Eq. 9) as a host-side state
// machine around pc_plan_budget, pc_score and pc_compact; its one kernel turns a cache mask (Eq. 1) into row indices.
#include <cuda.h>

#include <algorithm>
#include <vector>

#include "pc_common.cuh"

struct pc_window {
    pc_ctx *ctx;
    pc_window_params p;
    pc_segment anchors;
    pc_segment buf[2];
    int active;
    std::vector<int32_t> count;      // tokens per retained frame, oldest -> newest
    std::vector<int32_t> budget;     // scratch of the last plan
    int64_t t_shift;
    float *scores;
    int32_t *sel_idx;
    int32_t scratch_capacity;
    // the step from host memory: V and the output travel on a stream of their own, beside the kernels
    cudaStream_t side;
    cudaEvent_t main_ev, keys_ev, side_ev;
};

extern "C" pc_status pc_window_create(pc_ctx *ctx, const pc_window_params *params, const pc_segment *anchors,
                                      const pc_segment *hist_a, const pc_segment *hist_b, float *scores, int32_t *sel_idx,
                                      pc_window **out) {
    if (!ctx || !params || !anchors || !hist_a || !hist_b || !scores || !sel_idx || !out) return PC_ERR_INVALID_ARG;
    *out = nullptr;
    if (params->window < 1 || params->window >= PC_MAX_FRAMES || params->t_step < 0 || params->budget.total < 0)
        return PC_ERR_INVALID_ARG;
    if (!pc_aligned16(scores) || !pc_aligned16(sel_idx)) return PC_ERR_INVALID_ARG;
    pc_status st = pc_check_segment(anchors, true);
    if (st != PC_OK) return st;
    const pc_segment *hb[2] = {hist_a, hist_b};
    for (int i = 0; i < 2; ++i) {
        if (hb[i]->capacity <= 0 || !hb[i]->k || !hb[i]->v || !hb[i]->pos) return PC_ERR_INVALID_ARG;
        if (!pc_aligned16(hb[i]->k) || !pc_aligned16(hb[i]->v) || !pc_aligned16(hb[i]->pos)) return PC_ERR_INVALID_ARG;
    }
    pc_window *w = new (std::nothrow) pc_window();
    if (!w) return PC_ERR_CUDA;
    w->ctx = ctx;
    w->p = *params;
    w->anchors = *anchors;
    w->buf[0] = *hist_a;
    w->buf[1] = *hist_b;
    w->buf[0].n_tokens = w->buf[1].n_tokens = 0;
    w->active = 0;
    w->t_shift = 0;
    w->scores = scores;
    w->sel_idx = sel_idx;
    w->scratch_capacity = std::min(hist_a->capacity, hist_b->capacity);
    // The stream and the events belong to the context's device, whichever is current here: the steps' own stream is on it, and an
    // event is recorded on a stream of its own device only.
    const auto on_device = [&]() -> pc_status {
        PC_CUDA_TRY(cudaStreamCreateWithFlags(&w->side, cudaStreamNonBlocking));
        PC_CUDA_TRY(cudaEventCreateWithFlags(&w->main_ev, cudaEventDisableTiming));
        PC_CUDA_TRY(cudaEventCreateWithFlags(&w->keys_ev, cudaEventDisableTiming));
        PC_CUDA_TRY(cudaEventCreateWithFlags(&w->side_ev, cudaEventDisableTiming));
        return PC_OK;
    };
    int current = ctx->device;
    st = cudaGetDevice(&current) == cudaSuccess && (current == ctx->device || cudaSetDevice(ctx->device) == cudaSuccess) ? on_device() : PC_ERR_CUDA;
    if (current != ctx->device && cudaSetDevice(current) != cudaSuccess && st == PC_OK) st = PC_ERR_CUDA;
    if (st != PC_OK) {
        pc_window_destroy(w);
        return st;
    }
    *out = w;
    return PC_OK;
}

extern "C" pc_status pc_window_destroy(pc_window *w) {
    if (!w) return PC_ERR_INVALID_ARG;
    if (w->side) cudaStreamDestroy(w->side);
    if (w->main_ev) cudaEventDestroy(w->main_ev);
    if (w->keys_ev) cudaEventDestroy(w->keys_ev);
    if (w->side_ev) cudaEventDestroy(w->side_ev);
    delete w;
    return PC_OK;
}

namespace {

constexpr int APPEND_THREADS = 256, APPEND_CHUNKS = 4;

// A finished frame's K, V and position rows to the end of the history: three runs of 16-byte chunks in one launch, four chunks
// of a thread in flight.  Bound by launches and latency (4.1 MB each way for 1,008 tokens of 2 KB rows): three copies by the
// runtime were three launches with a drained GPU between them.  Back to back, 63 tokens 2.98 -> 1.44 us, 1,008 tokens
// 3.71 -> 2.74 us, 4,032 tokens 8.10 -> 6.40 us; append, update and attention over 8,064 kept tokens 152.1 -> 147.8 us.
__global__ void __launch_bounds__(APPEND_THREADS) k_append(const uint4 *__restrict__ k, const uint4 *__restrict__ v,
                                                           const uint4 *__restrict__ pos, uint4 *__restrict__ dst_k,
                                                           uint4 *__restrict__ dst_v, uint4 *__restrict__ dst_pos, long long n_kv /* chunks of K, and of V */,
                                                           int n_pos) {
    pc_grid_dep_launch();
    const long long i0 = (long long)blockIdx.x * (APPEND_THREADS * APPEND_CHUNKS) + threadIdx.x, n = 2 * n_kv + n_pos;
    pc_grid_dep_wait();
    uint4 x[APPEND_CHUNKS];
#pragma unroll
    for (int c = 0; c < APPEND_CHUNKS; ++c) {
        const long long i = i0 + c * APPEND_THREADS;
        if (i < n) x[c] = pc_ldg_stream(i < n_kv ? k + i : (i < 2 * n_kv ? v + (i - n_kv) : pos + (i - 2 * n_kv)));
    }
#pragma unroll
    for (int c = 0; c < APPEND_CHUNKS; ++c) {
        const long long i = i0 + c * APPEND_THREADS;
        if (i < n) *(i < n_kv ? dst_k + i : (i < 2 * n_kv ? dst_v + (i - n_kv) : dst_pos + (i - 2 * n_kv))) = x[c];
    }
}

// Memory that a kernel on the context's device reads as it is.
bool on_device(const pc_ctx *ctx, const void *p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice && a.device == ctx->device;
}

}  // namespace

extern "C" pc_status pc_window_append(pc_window *w, const pc_segment *frame, void *stream_) {
    if (!w || !frame) return PC_ERR_INVALID_ARG;
    pc_status st = pc_check_segment(frame, false);
    if (st != PC_OK) return st;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    pc_segment &A = w->buf[w->active];
    const int n = frame->n_tokens;
    if ((int64_t)A.n_tokens + n > A.capacity || (int64_t)A.n_tokens + n > w->scratch_capacity) return PC_ERR_CAPACITY;
    if ((int)w->count.size() + 1 > PC_MAX_FRAMES) return PC_ERR_CAPACITY;
    const size_t row = (size_t)w->ctx->desc.n_kv_heads * w->ctx->desc.head_dim * w->ctx->elem_size;
    const size_t at = (size_t)A.n_tokens * row;
    char *k = static_cast<char *>(A.k) + at, *v = static_cast<char *>(A.v) + at;
    int32_t *pos = A.pos + 4 * (size_t)A.n_tokens;
    if (on_device(w->ctx, frame->k) && on_device(w->ctx, frame->v) && on_device(w->ctx, frame->pos)) {
        const long long n_kv = (long long)(n * row / 16), chunks = 2 * n_kv + n, per_block = APPEND_THREADS * APPEND_CHUNKS;   // rows are multiples of 16 bytes
        PC_LAUNCH(k_append, dim3((unsigned)((chunks + per_block - 1) / per_block)), dim3(APPEND_THREADS), 0, stream,
                  static_cast<const uint4 *>(frame->k), static_cast<const uint4 *>(frame->v), reinterpret_cast<const uint4 *>(frame->pos),
                  reinterpret_cast<uint4 *>(k), reinterpret_cast<uint4 *>(v), reinterpret_cast<uint4 *>(pos), n_kv, n);
        PC_CUDA_TRY(cudaGetLastError());
    } else {
        // a frame on another GPU, in host memory, or nowhere the driver knows of: the runtime's copies reach the former and refuse the rest
        PC_CUDA_TRY(cudaMemcpyAsync(k, frame->k, (size_t)n * row, cudaMemcpyDeviceToDevice, stream));
        PC_CUDA_TRY(cudaMemcpyAsync(v, frame->v, (size_t)n * row, cudaMemcpyDeviceToDevice, stream));
        PC_CUDA_TRY(cudaMemcpyAsync(pos, frame->pos, (size_t)n * 16, cudaMemcpyDeviceToDevice, stream));
    }
    A.n_tokens += n;
    w->count.push_back(n);
    return PC_OK;
}

namespace {

// Indices of the non-zero bytes of valid[0..n), ascending, into idx; one block, a scan per 1024 bytes.  The host states how
// many there are (it sizes the frame table without a device round trip): a different count is recorded as an error.
__global__ void __launch_bounds__(1024) k_mask_to_index(const uint8_t *__restrict__ valid, int n, int32_t *__restrict__ idx,
                                                        int expected, int32_t *status) {
    pc_grid_dep_launch();
    pc_grid_dep_wait();
    __shared__ int warp_sums[32];
    __shared__ int carry;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int j0 = 0; j0 < n; j0 += 1024) {
        const int j = j0 + threadIdx.x;
        const int keep = j < n && valid[j] != 0;
        int inc = keep;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        if (lane == 31) warp_sums[w] = inc;
        __syncthreads();
        int base = carry;
        for (int i = 0; i < w; ++i) base += warp_sums[i];
        const int at = base + inc - keep;
        if (keep && at < expected) idx[at] = j;
        __syncthreads();
        if (threadIdx.x == 1023) carry = base + inc;
        __syncthreads();
    }
    if (threadIdx.x == 0 && carry != expected) pc_flag(status, PC_ERR_INVALID_ARG, PC_WHERE_MASK_COUNT);
}

}  // namespace

extern "C" pc_status pc_window_append_masked(pc_window *w, const pc_segment *frame, const uint8_t *valid, int32_t n_valid,
                                             void *stream_) {
    if (!w || !frame || !valid) return PC_ERR_INVALID_ARG;
    pc_status st = pc_check_segment(frame, false);
    if (st != PC_OK) return st;
    if (n_valid < 0 || n_valid > frame->n_tokens) return PC_ERR_INVALID_ARG;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    pc_segment &A = w->buf[w->active];
    // the grown buffer must fit the caller's score / index scratch as well (the next update scores every token of it), and
    // the mask's row indices go through that index scratch
    if ((int64_t)A.n_tokens + n_valid > A.capacity || (int64_t)A.n_tokens + n_valid > w->scratch_capacity ||
        frame->n_tokens > w->scratch_capacity)
        return PC_ERR_CAPACITY;
    if ((int)w->count.size() + 1 > PC_MAX_FRAMES) return PC_ERR_CAPACITY;
    if (n_valid > 0) {
        const size_t row = (size_t)w->ctx->desc.n_kv_heads * w->ctx->desc.head_dim * w->ctx->elem_size;
        PC_LAUNCH(k_mask_to_index, dim3(1), dim3(1024), 0, stream, valid, (int)frame->n_tokens, w->sel_idx, (int)n_valid,
                  w->ctx->status);
        st = pc_launch_pack(w->ctx, frame->k, frame->v, frame->pos, w->sel_idx, n_valid, frame->n_tokens, 0,
                            static_cast<char *>(A.k) + (size_t)A.n_tokens * row, static_cast<char *>(A.v) + (size_t)A.n_tokens * row,
                            A.pos + 4 * (size_t)A.n_tokens, nullptr, stream);
        if (st != PC_OK) return st;
    }
    A.n_tokens += n_valid;
    w->count.push_back(n_valid);
    return PC_OK;
}

namespace {

// What an update has to do, worked out on the host before anything is enqueued.
struct WindowPlan {
    bool fill;               // everything still fits: nothing to do
    pc_cache src;            // source of the pack: the active buffer past the frames that leave
    const int32_t *budget;   // quotas of the frames that stay (points into the window's plan)
    int stay, left;          // frames that stay / leave (beyond the window, or starved by the plan at the old end)
    int64_t n_sel;           // tokens kept
    int32_t delta_t;         // temporal rebase (Eq. 9)
    const float *scores_override;
};

pc_status window_plan(pc_window *w, const float *scores_override, WindowPlan *pl) {
    const int n_frames = (int)w->count.size();
    const int drop = std::max(0, n_frames - w->p.window);          // frames beyond the window leave first (FIFO)
    int64_t dropped_tokens = 0, kept_tokens = 0;
    for (int f = 0; f < n_frames; ++f) (f < drop ? dropped_tokens : kept_tokens) += w->count[f];
    pl->fill = drop == 0 && kept_tokens <= w->p.budget.total;      // Fill: everything still fits
    if (pl->fill) return PC_OK;
    const int kept = n_frames - drop;
    pc_segment &A = w->buf[w->active], &B = w->buf[w->active ^ 1];
    const size_t row = (size_t)w->ctx->desc.n_kv_heads * w->ctx->desc.head_dim * w->ctx->elem_size;
    // source: the active buffer past the dropped frames
    pc_cache &src = pl->src;
    src.anchors = w->anchors;
    src.history.k = static_cast<char *>(A.k) + (size_t)dropped_tokens * row;
    src.history.v = static_cast<char *>(A.v) + (size_t)dropped_tokens * row;
    src.history.pos = A.pos + 4 * (size_t)dropped_tokens;
    src.history.n_tokens = (int32_t)kept_tokens;
    src.history.capacity = (int32_t)(A.capacity - dropped_tokens);
    src.n_frames = kept;
    src.frame_count = w->count.data() + drop;
    w->budget.assign((size_t)std::max(kept, 1), 0);
    pc_status st = pc_plan_budget(&w->p.budget, kept, src.frame_count, w->budget.data());
    if (st != PC_OK) return st;
    // Frames that the plan leaves with nothing at the old end (a minimum quota starves the oldest frames first) leave the
    // window like frames beyond W: first in, first out, counted in the rebase.
    int lead = 0;
    int64_t lead_tokens = 0;
    while (lead < kept && w->budget[lead] == 0) lead_tokens += src.frame_count[lead++];
    pl->budget = w->budget.data() + lead;
    pl->left = drop + lead;
    pl->stay = kept - lead;
    src.history.k = static_cast<char *>(src.history.k) + (size_t)lead_tokens * row;
    src.history.v = static_cast<char *>(src.history.v) + (size_t)lead_tokens * row;
    src.history.pos += 4 * (size_t)lead_tokens;
    src.history.n_tokens -= (int32_t)lead_tokens;
    src.history.capacity -= (int32_t)lead_tokens;
    src.n_frames = pl->stay;
    src.frame_count += lead;
    pl->scores_override = scores_override ? scores_override + lead_tokens : nullptr;
    pl->n_sel = 0;
    for (int f = 0; f < pl->stay; ++f) pl->n_sel += pl->budget[f];
    if (pl->n_sel > B.capacity) return PC_ERR_CAPACITY;
    pl->delta_t = w->p.rebase ? pl->left * w->p.t_step : 0;        // Eq. 9: t falls by the number of frames that left
    return PC_OK;
}

// the other buffer becomes the active one and holds what was kept
void window_commit(pc_window *w, const WindowPlan &pl) {
    pc_segment &A = w->buf[w->active], &B = w->buf[w->active ^ 1];
    B.n_tokens = (int32_t)pl.n_sel;
    A.n_tokens = 0;
    w->active ^= 1;
    w->count.assign(pl.budget, pl.budget + pl.stay);
    w->t_shift += pl.delta_t;
}

}  // namespace

extern "C" pc_status pc_window_update(pc_window *w, const void *q, const int32_t *q_pos, int32_t n_q,
                                      const float *scores_override, int32_t *regime, void *stream) {
    if (!w) return PC_ERR_INVALID_ARG;
    WindowPlan pl;
    pc_status st = window_plan(w, scores_override, &pl);
    if (st != PC_OK) return st;
    if (pl.fill) {
        if (regime) *regime = PC_WINDOW_FILL;
        return PC_OK;
    }
    if (pl.stay > 0) {
        st = pc_score(w->ctx, &pl.src, q, q_pos, n_q, pl.budget, nullptr, pl.scores_override, w->scores, w->sel_idx, stream);
        if (st != PC_OK) return st;
        pc_cache dst;
        dst.anchors = w->anchors;
        dst.history = w->buf[w->active ^ 1];
        dst.n_frames = pl.stay;
        dst.frame_count = pl.budget;
        st = pc_compact(w->ctx, &pl.src, w->sel_idx, pl.budget, pl.delta_t, &dst, stream);
        if (st != PC_OK) return st;
    }
    window_commit(w, pl);
    if (regime) *regime = pl.left ? PC_WINDOW_SLIDE : PC_WINDOW_PACK;
    return PC_OK;
}

namespace {

// what attention runs over where nothing is packed: the window as it is, or (every frame leaves) none of it
pc_cache unpacked_cache(const pc_window *w, const WindowPlan &pl) {
    pc_cache cache;
    cache.anchors = w->anchors;
    cache.history = w->buf[w->active];
    if (!pl.fill) cache.history.n_tokens = 0;
    cache.n_frames = pl.fill ? (int32_t)w->count.size() : 0;
    cache.frame_count = w->count.data();
    return cache;
}
pc_cache pack_destination(const pc_window *w, const WindowPlan &pl) {
    pc_cache dst;
    dst.anchors = w->anchors;
    dst.history = w->buf[w->active ^ 1];
    dst.n_frames = pl.stay;
    dst.frame_count = pl.budget;
    return dst;
}

// The plan and every other host-side check of a step, nothing enqueued.
pc_status window_step_check(pc_window *w, const void *q, const int32_t *q_pos, int32_t n_q, const void *out) {
    WindowPlan pl;
    const pc_status st = window_plan(w, nullptr, &pl);
    if (st != PC_OK) return st;
    if (pl.fill || pl.stay == 0) {
        const pc_cache cache = unpacked_cache(w, pl);
        return pc_attend_frame_check(w->ctx, &cache, nullptr, q, q_pos, n_q, out, nullptr);
    }
    const pc_cache dst = pack_destination(w, pl);
    return pc_frame_step_check(w->ctx, &pl.src, pl.budget, &dst, q, q_pos, n_q, w->scores, w->sel_idx, out, nullptr);
}

// A step that fails leaves the window as it was.
pc_status window_step(pc_window *w, const void *q, const int32_t *q_pos, int32_t n_q, void *out, float *lse, int32_t *regime,
                      cudaStream_t stream, const pc_step_hooks *hooks) {
    WindowPlan pl;
    pc_status st = window_plan(w, nullptr, &pl);
    if (st != PC_OK) return st;
    if (pl.fill || pl.stay == 0) {
        const pc_cache cache = unpacked_cache(w, pl);
        st = pc_attend_frame_impl(w->ctx, &cache, nullptr, q, q_pos, n_q, out, lse, stream, hooks);
        if (st != PC_OK) return st;
        if (!pl.fill) window_commit(w, pl);
        if (regime) *regime = pl.fill ? PC_WINDOW_FILL : (pl.left ? PC_WINDOW_SLIDE : PC_WINDOW_PACK);
        return PC_OK;
    }
    pc_cache dst = pack_destination(w, pl);
    st = pc_frame_step_impl(w->ctx, &pl.src, pl.budget, pl.delta_t, &dst, q, q_pos, n_q, w->scores, w->sel_idx, out, lse, stream, hooks);
    if (st != PC_OK) return st;
    window_commit(w, pl);
    if (regime) *regime = pl.left ? PC_WINDOW_SLIDE : PC_WINDOW_PACK;
    return PC_OK;
}

// A step from host memory goes up and home by a kernel each as long as it moves no more than this (queries, output, keys and values) and its
// attention is one part.  Window of six frames, eight processes a side in turn, us a call as the shortest and the middle one of their medians: the runtime's copies
// on two streams against the kernels.  24 / 8 heads, 30 tokens (0.5 MB both ways) 69 / 74 -> 56 / 58, 135 (2.2) 101 / 155 -> 93 / 100, 247 (4.0) 130 / 206
// -> 133 / 137, 360 (5.9) 168 / 279 -> 175 / 177; 8 / 8, 682 (5.6) 167 / 265 -> 170 / 171, 988 (8.1) 217 / 310 -> 224 / 225; 32 / 16, 135 (3.3) 158 / 202 -> 117 / 121,
// 247 (6.1) 171 / 208 -> 176 / 177, 360 (8.8) 219 / 259 -> 232 / 233.  What the copies take depends on the process: in its best case up to 5 % less than the
// kernels from 4 MB on, mostly a good deal more, by less the larger the step (a third below 6 MB, a tenth at 9).  What the kernels take does not.
constexpr size_t SMALL_STEP = 6 << 20;

// Runs of 16-byte chunks between pinned host memory and the device in one launch.  Bound by the link: 50 GB/s from and to pinned memory
// where the copy engine does 54, but no start-up of 3 to 9 us for every run, no hand-over from engine to kernel (5 us), and launched like any
// other kernel of the library.
constexpr int MOVE_THREADS = 256, MOVE_CHUNKS = 4, MOVE_RUNS = 5;
struct Runs {
    int n;
    const uint4 *src[MOVE_RUNS];
    uint4 *dst[MOVE_RUNS];
    long long end[MOVE_RUNS];        // chunks up to the run's end
};
__global__ void __launch_bounds__(MOVE_THREADS) k_move(const __grid_constant__ Runs R) {
    pc_grid_dep_launch();
    const long long i0 = (long long)blockIdx.x * (MOVE_THREADS * MOVE_CHUNKS) + threadIdx.x;
    pc_grid_dep_wait();
    uint4 x[MOVE_CHUNKS];
    uint4 *to[MOVE_CHUNKS];
#pragma unroll
    for (int c = 0; c < MOVE_CHUNKS; ++c) {
        const long long i = i0 + c * MOVE_THREADS;
        to[c] = nullptr;
        long long first = 0;
        for (int r = 0; r < R.n; ++r) {
            if (i >= first && i < R.end[r]) {
                x[c] = __ldcg(R.src[r] + (i - first));         // (not as constant data: a kernel that this one overlaps writes the output)
                to[c] = R.dst[r] + (i - first);
            }
            first = R.end[r];
        }
    }
#pragma unroll
    for (int c = 0; c < MOVE_CHUNKS; ++c)
        if (to[c]) *to[c] = x[c];
}
void add_run(Runs &R, const void *src, void *dst, size_t bytes) {
    R.src[R.n] = static_cast<const uint4 *>(src);
    R.dst[R.n] = static_cast<uint4 *>(dst);
    R.end[R.n] = (R.n ? R.end[R.n - 1] : 0) + (long long)(bytes / 16);
    ++R.n;
}
pc_status launch_move(const Runs &R, cudaStream_t stream) {
    const long long chunks = R.end[R.n - 1], per_block = MOVE_THREADS * MOVE_CHUNKS;
    PC_LAUNCH(k_move, dim3((unsigned)((chunks + per_block - 1) / per_block)), dim3(MOVE_THREADS), 0, stream, R);
    PC_CUDA_TRY(cudaGetLastError());
    return PC_OK;
}

// Where a kernel finds `bytes` of pinned host memory; NULL where it cannot (pageable, in part or at all, managed, or not on 16 bytes).  The
// driver says from where to where the allocation or registration around p goes: two pinned ends do not make the middle pinned.
void *device_view(const void *p, size_t bytes) {
    typedef CUresult (*AttributesFn)(unsigned, CUpointer_attribute *, void **, CUdeviceptr);
    static const AttributesFn attributes = []() -> AttributesFn {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuPointerGetAttributes", &f, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<AttributesFn>(f);
        cudaGetLastError();
        return nullptr;
    }();
    if (!attributes || !pc_aligned16(p)) return nullptr;
    unsigned type = 0, managed = 0;
    CUdeviceptr at = 0, first = 0;
    size_t size = 0;
    CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                  CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void *to[] = {&type, &managed, &at, &first, &size};
    const CUdeviceptr host = reinterpret_cast<CUdeviceptr>(p);
    if (attributes(5, what, to, host) != CUDA_SUCCESS || type != CU_MEMORYTYPE_HOST || managed) return nullptr;
    if (at != host || host < first || host - first > size || size - (host - first) < bytes) return nullptr;    // (one address on either side, as unified addressing has it)
    return const_cast<void *>(p);
}

// A part of the output is enqueued: it goes home on the side stream while the next part is computed, or (a small step, in one part) by a
// kernel behind it.  Either way ahead of the window's change of state, behind which nothing is enqueued that could fail.
struct HomeTrip {
    pc_window *w;
    const char *from;
    char *to;
    size_t row_bytes;
};

pc_status send_home(void *self, int row0, int n, cudaStream_t stream) {
    const HomeTrip &h = *static_cast<const HomeTrip *>(self);
    PC_CUDA_TRY(cudaEventRecord(h.w->main_ev, stream));
    PC_CUDA_TRY(cudaStreamWaitEvent(h.w->side, h.w->main_ev, 0));
    PC_CUDA_TRY(cudaMemcpyAsync(h.to + row0 * h.row_bytes, h.from + row0 * h.row_bytes, n * h.row_bytes, cudaMemcpyDeviceToHost, h.w->side));
    return PC_OK;
}
pc_status move_home(void *self, int row0, int n, cudaStream_t stream) {
    const HomeTrip &h = *static_cast<const HomeTrip *>(self);
    Runs home{};
    add_run(home, h.from + row0 * h.row_bytes, h.to + row0 * h.row_bytes, n * h.row_bytes);
    return launch_move(home, stream);
}

}  // namespace

extern "C" pc_status pc_window_step(pc_window *w, const void *q, const int32_t *q_pos, int32_t n_q, void *out, float *lse,
                                    int32_t *regime, void *stream) {
    if (!w) return PC_ERR_INVALID_ARG;
    return window_step(w, q, q_pos, n_q, out, lse, regime, static_cast<cudaStream_t>(stream), nullptr);
}

extern "C" pc_status pc_window_step_host(pc_window *w, const pc_host_window_step *in, const pc_window_step_workspace *ws,
                                         int32_t *regime, void *stream_) {
    if (!w || !in || !ws) return PC_ERR_INVALID_ARG;
    if (!in->q || !in->q_pos || !in->out || in->n_q <= 0 || in->n_frame < 0) return PC_ERR_INVALID_ARG;
    if (!ws->q || !ws->q_pos || !ws->out) return PC_ERR_INVALID_ARG;
    if (in->n_frame > 0 && (!in->frame_k || !in->frame_v || !in->frame_pos)) return PC_ERR_INVALID_ARG;
    if (in->n_q > w->ctx->desc.max_q) return PC_ERR_CAPACITY;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const pc_layer_desc &D = w->ctx->desc;
    const size_t row = (size_t)D.n_kv_heads * D.head_dim * w->ctx->elem_size;
    const size_t qrow = (size_t)D.n_q_heads * D.head_dim * w->ctx->elem_size;
    pc_segment &A = w->buf[w->active];
    const int n = in->n_frame;
    if (n > 0) {
        if ((int64_t)A.n_tokens + n > A.capacity || (int64_t)A.n_tokens + n > w->scratch_capacity) return PC_ERR_CAPACITY;
        if ((int)w->count.size() + 1 > PC_MAX_FRAMES) return PC_ERR_CAPACITY;
    }
    // The step is planned and checked on the window as it will be with the frame appended (host arithmetic only); if it cannot be
    // made, the window is left as it was and nothing is enqueued.
    if (n > 0) {
        A.n_tokens += n;
        w->count.push_back(n);
    }
    const auto take_back = [&]() {
        if (n > 0) {
            A.n_tokens -= n;
            w->count.pop_back();
        }
    };
    pc_status st = window_step_check(w, ws->q, ws->q_pos, in->n_q, ws->out);
    if (st != PC_OK) {
        take_back();
        return st;
    }
    // Every argument is checked: from here on work is enqueued.
    const size_t at = (size_t)(A.n_tokens - n), q_bytes = (size_t)in->n_q * qrow, kv_bytes = (size_t)n * row, q_pos_bytes = (size_t)in->n_q * 16, pos_bytes = (size_t)n * 16;
    char *const to_k = static_cast<char *>(A.k) + at * row, *const to_v = static_cast<char *>(A.v) + at * row;
    int32_t *const to_pos = A.pos + 4 * at;
    const void *const q_pos = device_view(in->q_pos, q_pos_bytes), *const pos = n > 0 ? device_view(in->frame_pos, pos_bytes) : nullptr;
    // A small step goes up and home by a kernel each, and runs as a step on the device does in between.
    const auto enqueue_small = [&](const void *q, const void *k, const void *v, void *out) -> pc_status {
        Runs up{};
        add_run(up, q, ws->q, q_bytes);
        add_run(up, q_pos, ws->q_pos, q_pos_bytes);
        if (n > 0) {
            add_run(up, k, to_k, kv_bytes);
            add_run(up, v, to_v, kv_bytes);
            add_run(up, pos, to_pos, pos_bytes);
        }
        HomeTrip trip{w, static_cast<const char *>(ws->out), static_cast<char *>(out), qrow};
        const pc_step_hooks hooks{nullptr, move_home, &trip};
        const pc_status s = launch_move(up, stream);
        return s == PC_OK ? window_step(w, ws->q, ws->q_pos, in->n_q, ws->out, nullptr, regime, stream, &hooks) : s;
    };
    // In a larger one what the scores need goes first: the queries, then the finished frame's keys, straight to the end of the active history
    // buffer, on the side stream; the positions come by a kernel beside them.  The values follow under the scoring and
    // the selection, and the output leaves in parts, under the attention of the next part.  What remains is the upload of
    // queries, keys and values (10.4 MB for a 1,008-token frame, 195 us at the copy engine's rate), the attention behind it and the
    // last part's way home: everything in a row on one stream took 508 us, with the positions as copies of their own and the values behind an event of the keys' stream 411.
    const auto enqueue = [&]() -> pc_status {
        PC_CUDA_TRY(cudaEventRecord(w->main_ev, stream));            // whatever used the buffers before
        PC_CUDA_TRY(cudaStreamWaitEvent(w->side, w->main_ev, 0));
        PC_CUDA_TRY(cudaMemcpyAsync(ws->q, in->q, q_bytes, cudaMemcpyHostToDevice, w->side));
        Runs small{};
        if (q_pos) add_run(small, q_pos, ws->q_pos, q_pos_bytes);
        else PC_CUDA_TRY(cudaMemcpyAsync(ws->q_pos, in->q_pos, q_pos_bytes, cudaMemcpyHostToDevice, w->side));
        if (pos) add_run(small, pos, to_pos, pos_bytes);
        else if (n > 0) PC_CUDA_TRY(cudaMemcpyAsync(to_pos, in->frame_pos, pos_bytes, cudaMemcpyHostToDevice, w->side));
        if (n > 0) PC_CUDA_TRY(cudaMemcpyAsync(to_k, in->frame_k, kv_bytes, cudaMemcpyHostToDevice, w->side));
        PC_CUDA_TRY(cudaEventRecord(w->keys_ev, w->side));
        if (n > 0) PC_CUDA_TRY(cudaMemcpyAsync(to_v, in->frame_v, kv_bytes, cudaMemcpyHostToDevice, w->side));
        PC_CUDA_TRY(cudaEventRecord(w->side_ev, w->side));
        if (small.n > 0) {
            const pc_status s = launch_move(small, stream);
            if (s != PC_OK) return s;
        }
        PC_CUDA_TRY(cudaStreamWaitEvent(stream, w->keys_ev, 0));
        HomeTrip trip{w, static_cast<const char *>(ws->out), static_cast<char *>(in->out), qrow};
        const pc_step_hooks hooks{w->side_ev, send_home, &trip};
        return window_step(w, ws->q, ws->q_pos, in->n_q, ws->out, nullptr, regime, stream, &hooks);
    };
    const bool small = q_pos && (n == 0 || pos) && 2 * q_bytes + 2 * kv_bytes <= SMALL_STEP && pc_attend_part_rows(w->ctx, in->n_q) >= in->n_q;
    const void *const q = small ? device_view(in->q, q_bytes) : nullptr, *const k = small && n > 0 ? device_view(in->frame_k, kv_bytes) : nullptr;
    const void *const v = k ? device_view(in->frame_v, kv_bytes) : nullptr;
    void *const out = q && (n == 0 || v) ? device_view(in->out, q_bytes) : nullptr;
    st = out ? enqueue_small(q, k, v, out) : enqueue();
    // also after an error: nothing of this call stays in flight, and the frame is not counted as appended
    const cudaError_t side = cudaStreamSynchronize(w->side), main = cudaStreamSynchronize(stream);
    if (st != PC_OK) {
        take_back();
        return st;
    }
    PC_CUDA_TRY(side);
    PC_CUDA_TRY(main);
    return PC_OK;
}

extern "C" pc_status pc_window_cache(pc_window *w, pc_cache *out) {
    if (!w || !out) return PC_ERR_INVALID_ARG;
    out->anchors = w->anchors;
    out->history = w->buf[w->active];
    out->n_frames = (int32_t)w->count.size();
    out->frame_count = w->count.data();
    return PC_OK;
}

extern "C" pc_status pc_window_state(pc_window *w, int32_t *n_frames, int32_t *counts, int64_t *t_shift, int32_t *active) {
    if (!w) return PC_ERR_INVALID_ARG;
    if (n_frames) *n_frames = (int32_t)w->count.size();
    if (counts)
        for (size_t f = 0; f < w->count.size(); ++f) counts[f] = w->count[f];
    if (t_shift) *t_shift = w->t_shift;
    if (active) *active = w->active;
    return PC_OK;
}

// Scores, per-frame selection and, for the fused step, the pack of a small history in one launch behind the query pass.
//
// A cluster of CTAs takes whole frames, so no cluster waits for another, and the stages of one are separated by cluster barriers.  A
// CTA has a run of consecutive tokens of one frame; their keys (and values) are on their way to its shared memory before the
// pooled query is there, and stay until the pack.
//   scores   as the scoring kernel has them, bit for bit (pc_rows.cuh): to global memory, and as order-preserving keys to the shared
//            memory of all CTAs of the frame.
//   select   a token is kept if fewer than budget[f] of its frame's tokens beat it (a better score, or the same and a lower index):
//            a CTA counts that for its own tokens by comparing them with all of the frame's, tells the frame's other CTAs how many it
//            keeps, and with theirs knows the ranks of its own.
//   pack     of the CTA's own kept tokens, out of shared memory.
// Bound by latency: every stage is a few hundred instructions, run once, between two barriers (0.6 us for the pooled query, 1.2 for the scores of
// one key per half warp, 0.6 for the counting, 0.4 to 0.6 for each barrier or exchange, 0.4 for the pack).  Against a launch each for
// scores and for selection and pack, a step by itself and (GPU alone, captured) in us: 135-token frames, 24 / 8 heads, 5 frames
// 25.3 (24.3) -> 24.1 (22.9), 11 frames 27.7 (26.4) -> 25.9 (25.1); 30-token frames 21.1 (19.9) -> 19.4 (16.8); 64-token fp32 frames, 4 / 2 x 64,
// 20.7 (15.6) -> 19.1 (14.5); 32 / 16 heads, 64-token frames 24.8 (24.9) -> 19.4 (18.5).
// Tried: the query pass in the same kernel, each cluster pooling all queries for itself (small bf16 step 26.7 -> 35.3) or all CTAs with a
// barrier over a cooperative grid (30.7; such a launch does not overlap the kernel before).
#include <algorithm>
#include <atomic>

#include "pc_rows.cuh"
#include "pc_select.cuh"
#include "pc_tc.cuh"

namespace {

using pc_tc::cluster_rank;
using pc_tc::cluster_sync_all;
using pc_tc::peer_addr;

constexpr int FRONT_THREADS = 512, FRONT_WARPS = FRONT_THREADS / 32;
// Clusters of eight CTAs (the portable size), as long as all of them find room beside the query pass's last blocks: with twelve and
// more the last ones start late (16 to 24 frames 5 to 15 % slower than the separate kernels).  Clusters of four from there on: 24 / 8 heads, 30 and
// 60 tokens, 12 to 24 frames, the separate kernels against eleven clusters that take several frames each, and against clusters of
// four: 24.9 -> 24.3 and 23.5 us on average; 96 tokens, 20 frames 26.6 -> 27.3 and 24.9.
constexpr int FRONT_CTAS = 8, FRONT_CLUSTERS = 11, FRONT_CTAS_MANY = 4, FRONT_CLUSTERS_MANY = 32;
constexpr int FRONT_FRAMES = FRONT_CTAS_MANY * FRONT_CLUSTERS_MANY;
static_assert(FRONT_CLUSTERS <= FRONT_FRAMES, "a cluster has at least a CTA for every frame of its own");
constexpr int FRONT_TOKENS = 48;                    // most tokens of a CTA
constexpr int FRONT_SMEM = 220 * 1024;

struct FrontParams {
    const char *k, *v;
    const int32_t *pos;
    const uint8_t *valid;
    int row_bytes, d;
    float scale;
    unsigned long long *fx;                         // the query pass's accumulator
    double fx_scale;
    float *scores;
    int32_t *sel_idx;
    char *dst_k, *dst_v, *rot_k;                    // rot_k: NULL unless rotated keys are wanted
    int32_t *dst_pos;
    int delta_t, n_frames;
    int32_t *status;
    uint32_t wait_us, extra_tx;
    int ctas, cap, at_keys, at_tok, at_rows;        // as pc_front_plan
    pc_rope_dev rope;
    int4 f[FRONT_FRAMES];                           // (first token, tokens, budget, output offset)
};

__host__ __device__ __forceinline__ int share(int n, int i, int of) { return (int)((unsigned)n * (unsigned)i / (unsigned)of); }

// the frames of a cluster and, of these, the frame of a CTA with the CTAs (first .. first + n - 1) that share it
struct FrontFrame { int frame, first, n; };
__host__ __device__ __forceinline__ FrontFrame front_frame(int n_frames, int clusters, int cluster, int rank, int ctas) {
    const int f0 = share(n_frames, cluster, clusters), nf = share(n_frames, cluster + 1, clusters) - f0, j = share(nf, rank, ctas);
    const int first = (j * ctas + nf - 1) / nf, end = ((j + 1) * ctas + nf - 1) / nf;
    return {f0 + j, first, end - first};
}

__device__ __forceinline__ void peer_st32(uint32_t a, uint32_t v) { asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }

template <typename T, int LPT /* lanes per token in scoring */, bool PACK>
__global__ void __launch_bounds__(FRONT_THREADS, 1) k_front(const __grid_constant__ FrontParams P) {
    pc_grid_dep_launch();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    constexpr int PER = Elem<T>::PER16, NP = PER / 2, SIDE = 32 / LPT;
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ __align__(8) unsigned long long bars[2];
    __shared__ int gave_up, block_kept[FRONT_WARPS], mate_kept[FRONT_CTAS];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, lt = lane % LPT, side = lane / LPT;
    const int rank = (int)cluster_rank();
    float4 *qs = reinterpret_cast<float4 *>(sm);                                  // the pooled query, as the scoring kernel has it
    uint32_t *keys = reinterpret_cast<uint32_t *>(sm + P.at_keys);                // of the whole frame
    int4 *tok_pos = reinterpret_cast<int4 *>(sm + P.at_tok);                      // of the own tokens: position, tokens that beat it, the kept ones
    int *beaten = reinterpret_cast<int *>(tok_pos + P.cap), *kept = beaten + P.cap;
    const uint32_t k_rows = pc_smem_u32(sm + P.at_rows), v_rows = k_rows + P.cap * P.row_bytes, bar0 = pc_smem_u32(bars);

    const FrontFrame own = front_frame(P.n_frames, (int)gridDim.x / P.ctas, (int)blockIdx.x / P.ctas, rank, P.ctas);
    const int4 fr = P.f[own.frame];
    const int a = share(fr.y, rank - own.first, own.n), n_tok = share(fr.y, rank - own.first + 1, own.n) - a;
    // keys, values and positions are final already: the query pass lets this kernel go after its own wait
    if (tid == 0) {
        pc_mbar_init(bar0, 1);
        pc_mbar_init(bar0 + 8, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        gave_up = 0;
        const uint32_t bytes = (uint32_t)n_tok * P.row_bytes;
        const size_t at = (size_t)(fr.x + a) * P.row_bytes;
        pc_mbar_expect_tx(bar0, bytes + P.extra_tx);
        if (bytes) pc_bulk_g2s(k_rows, P.k + at, bytes, bar0);
        if constexpr (PACK) {
            pc_mbar_expect_tx(bar0 + 8, bytes);
            if (bytes) pc_bulk_g2s(v_rows, P.v + at, bytes, bar0 + 8);
        }
    }
    for (int i = tid; i < n_tok; i += FRONT_THREADS) {
        tok_pos[i] = __ldcg(reinterpret_cast<const int4 *>(P.pos) + fr.x + a + i);
        beaten[i] = 0;
    }
    __syncthreads();
    // the first scores' table entries
    const ScoreTable<T> table(P.rope, lt, P.d);
    float2 cs[1][NP];
    auto entries = [&](int i) { table.at(P.rope, tok_pos[min(i, n_tok - 1)], cs[0], P.status); };
    if (warp * SIDE < n_tok) entries(warp * SIDE + side);
    pc_grid_dep_wait();                                                           // the pooled query comes from the kernel before

    const int n_out = P.row_bytes / (int)sizeof(T), parts = n_out / (LPT * PER);
    for (int idx = tid; idx < parts * NP * LPT; idx += FRONT_THREADS) {
        const int l = idx % LPT, u = (idx / LPT) % NP, g = idx / (LPT * NP);
        const longlong2 w = __ldcg(reinterpret_cast<const longlong2 *>(P.fx + (size_t)(g * LPT + l) * PER + 2 * u));
        const float x = (float)((double)w.x * P.fx_scale), y = (float)((double)w.y * P.fx_scale);
        qs[idx] = make_float4(x, y, y, -x);
    }
    __syncthreads();
    // as in the scoring kernel: whoever finds that all blocks have read the accumulator clears it
    unsigned long long ticket = 0;
    if (tid == 0) ticket = atomicAdd(P.fx + n_out, 1ull);

    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");                    // all CTAs run: their memory may be written
    const bool keys_here = __all_sync(0xffffffffu, pc_mbar_wait(bar0, 0, &gave_up, P.status, PC_WHERE_SCORE_WAIT, P.wait_us));
    if (keys_here)
        for (int i0 = warp * SIDE; i0 < n_tok; i0 += FRONT_WARPS * SIDE) {
            const int i = i0 + side;
            if (i0 != warp * SIDE) entries(i);
            float s[1];
            score_rows<T, LPT, 1>(k_rows + min(i, n_tok - 1) * P.row_bytes + lt * 16, 0, parts, qs + lt, cs, s);
            float v = s[0];
#pragma unroll
            for (int o = LPT / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            v *= P.scale;
            if (i < n_tok) {
                const int j = fr.x + a + i;
                if (P.valid && !P.valid[j]) v = -INFINITY;
                if (lt == 0) {
                    P.scores[j] = v;
                    if (v != v && fr.z > 0) pc_flag(P.status, PC_ERR_INVALID_ARG, PC_WHERE_SELECT_NAN);
                }
                if (lt < own.n) peer_st32(peer_addr(pc_smem_u32(keys + a + i), own.first + lt), score_key(v));
            }
        }
    cluster_sync_all();                               // the frame's keys are all here

    // Tokens that beat the own ones.  A warp takes 32 own tokens, one per lane, and a stretch of the frame.
    if (keys_here) {
        const int blocks = (n_tok + 31) / 32, stretches = max(1, FRONT_WARPS / max(1, blocks));
        for (int w = warp; w < blocks * stretches; w += FRONT_WARPS) {
            const int b = w % blocks, st = w / blocks, i = b * 32 + lane, j = a + i;
            const uint32_t key = i < n_tok ? keys[j] : 0xFFFFFFFFu;
            int n = 0;
#pragma unroll 4
            for (int x = share(fr.y, st, stretches); x < share(fr.y, st + 1, stretches); ++x) {
                const uint32_t other = keys[x];       // the same in every lane
                n += other > key || (other == key && x < j);
            }
            if (i < n_tok && n) atomicAdd(beaten + i, n);
        }
    }
    __syncthreads();
    // how many this CTA keeps, told to the frame's CTAs; the kept ones in a list
    bool mine = false;
    uint32_t kept_here = 0;
    if (warp * 32 < P.cap) {
        mine = tid < n_tok && keys_here && beaten[tid] < fr.z;
        kept_here = __ballot_sync(0xffffffffu, mine);
        if (lane == 0) block_kept[warp] = __popc(kept_here);
    }
    __syncthreads();
    const int kept_blocks = (P.cap + 31) / 32;
    int before = __popc(kept_here & ((1u << lane) - 1u)), n_kept = 0;
    for (int b = 0; b < kept_blocks; ++b) {
        before += b < warp ? block_kept[b] : 0;
        n_kept += block_kept[b];
    }
    if (mine) kept[before] = tid;
    if (tid < own.n) peer_st32(peer_addr(pc_smem_u32(mate_kept + rank - own.first), own.first + tid), (uint32_t)n_kept);
    cluster_sync_all();                               // and nobody reaches into a peer's memory any more
    int out0 = fr.w;
    for (int m = 0; m < rank - own.first; ++m) out0 += mate_kept[m];
    n_kept = max(0, min(n_kept, fr.w + fr.z - out0));  // (a CTA whose wait ran out has sent no keys)
    for (int r = tid; r < n_kept; r += FRONT_THREADS) P.sel_idx[out0 + r] = fr.x + a + kept[r];

    if constexpr (PACK) {
        const bool values_here = __all_sync(0xffffffffu, pc_mbar_wait(bar0 + 8, 0, &gave_up, P.status, PC_WHERE_SCORE_WAIT, P.wait_us));
        const int k_side = warp & 1;                                    // odd warps: keys and their rotated form; even ones: values, positions
        if (values_here)
            for (int r = warp >> 1; r < n_kept; r += FRONT_WARPS / 2) {
                const int i = kept[r];
                const size_t to = (size_t)(out0 + r) * P.row_bytes + lane * 16;
                const uint32_t from = (k_side ? k_rows : v_rows) + i * P.row_bytes + lane * 16;
                char *dst = (k_side ? P.dst_k : P.dst_v) + to;
                int4 p = tok_pos[i];
                p.x -= P.delta_t;                                       // only t moves; h, w and the tag are carried as they are
                if (!k_side || !P.rot_k) {
#pragma unroll 4
                    for (int o = 0; o < P.row_bytes; o += 512) pc_stg_stream(dst + o, pc_lds128(from + o));
                    if (!k_side && lane == 0) reinterpret_cast<int4 *>(P.dst_pos)[out0 + r] = p;
                    continue;
                }
                // 32 lanes x 8 elements span a multiple of d: all of this lane's chunks hold the same four rotary pairs
                const int pair0 = ((lane * 8) % P.d) / 2;
                float2 rc[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) rc[u] = pc_rope_cs(P.rope, pair0 + u, p.x, p.y, p.z, P.status, PC_WHERE_ROPE_POS);
                for (int o = 0; o < P.row_bytes; o += 512) {
                    const uint4 w = pc_lds128(from + o);
                    pc_stg_stream(dst + o, w);
                    const uint32_t wv[4] = {w.x, w.y, w.z, w.w};
                    uint32_t t[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float2 y = pc_rotate(pc_bf16_lo(wv[u]), pc_bf16_hi(wv[u]), rc[u]);
                        t[u] = pc_pack_bf16(y.x, y.y);
                    }
                    *reinterpret_cast<uint4 *>(P.rot_k + to + o) = make_uint4(t[0], t[1], t[2], t[3]);
                }
            }
    }
    if (warp == 0 && __shfl_sync(0xffffffffu, ticket, 0) == (unsigned long long)(gridDim.x - 1))
        for (int e = lane; e <= n_out; e += 32) P.fx[e] = 0;
    // a wait ran out: copies may be in flight that nobody waited for
    __syncthreads();
    if (tid == 0 && gave_up) pc_let_copies_land();
}

// How a call is laid out: clusters, and the shared memory of a CTA; false where it does not fit or the separate kernels are faster.  Every scoring
// call asks, so a long history is refused at once and the rest takes a division a frame at most (a walk over all CTAs took 0.5 us of host time at
// 5 frames and 1.6 at 47, twice a call).
bool lay_out(const pc_ctx *ctx, const pc_cache *src, bool pack, pc_front_plan &L) {
    const pc_layer_desc &D = ctx->desc;
    const int n_frames = src->n_frames;
    if (n_frames < 1 || n_frames > FRONT_FRAMES || src->history.n_tokens > FRONT_TOKENS * FRONT_FRAMES) return false;
    const bool many = n_frames > FRONT_CLUSTERS;
    L.ctas = many ? FRONT_CTAS_MANY : FRONT_CTAS;
    L.clusters = std::min(n_frames, FRONT_CLUSTERS_MANY);
    int longest = 1;
    for (int f = 0; f < n_frames; ++f) longest = std::max(longest, src->frame_count[f]);
    if (longest > FRONT_TOKENS * L.ctas) return false;
    int cap = (longest + L.ctas - 1) / L.ctas;      // most tokens of a CTA: a cluster to a frame, or (front_frame) a cluster's CTAs shared out over its frames
    if (n_frames > L.clusters) {
        cap = 1;
        for (int c = 0; c < L.clusters; ++c) {
            const int f0 = share(n_frames, c, L.clusters), nf = share(n_frames, c + 1, L.clusters) - f0;
            for (int j = 0, first = 0; j < nf; ++j) {
                const int end = ((j + 1) * L.ctas + nf - 1) / nf, n = end - first;
                cap = std::max(cap, (src->frame_count[f0 + j] + n - 1) / n);
                first = end;
            }
        }
    }
    const int row = D.n_kv_heads * D.head_dim, row_bytes = row * ctx->elem_size;
    const bool fp32 = D.dtype != PC_BF16;
    // Tokens of a CTA: what its warps score at once (32), or more of narrow rows, most in clusters of eight.  Steps one after the other, the separate kernels
    // against this one, us.  Clusters of eight: 2 KB, 5 frames of 257 to 288 tokens (33 to 36 a CTA) 28.9 -> 28.6, 9 frames 30.6 -> 30.2 (captured 28.4 and 28.4,
    // 29.1 and 29.2), of 296 and more 29.8 -> 30.0; 1.5 KB, 288 to 320 26.0 -> 25.6 and 28.1 -> 27.5, 352 to 384 27.6 -> 27.7 and 29.5 -> 30.3; 1 KB, 288 to 384
    // 27.5 -> 26.3 and 29.4 -> 29.0; 512 bytes, bf16, 3 and 5 frames 23.9 -> 22.5, 9 frames 24.7 -> 25.6; fp32 35.3 -> 34.0 on average of 5 and 9.
    // Clusters of four, 16 frames: 2 KB, 132 tokens (33) 26.3 -> 26.0, 144 27.9 -> 28.1; 1.5 KB, 132 to 152 27.8 -> 24.3; 1 KB 26.0 -> 24.1; 512 bytes
    // bf16 24.8 -> 22.7, fp32 30.0 -> 30.7, its rows of 1 and 1.5 KB 41.1 -> 41.7.
    const auto most = [&]() {
        if (many && (fp32 || row_bytes > 1536)) return 32;
        return row_bytes <= 1024 ? FRONT_TOKENS : (row_bytes <= 1536 ? 40 : (row_bytes <= 2048 ? 36 : 32));
    };
    // One frame and no pack, more than 256 tokens: 10.1 -> 10.7 us.  fp32 rows of 512 bytes, more than 16 frames: 24 of 100 tokens 28.8 -> 30.6, 32 of 32
    // 22.0 -> 23.9, 32 of 100 33.9 -> 35.7 (16 of 100 26.2 -> 22.9).
    if (cap > most() || (!pack && n_frames == 1 && cap > 32) || (fp32 && row_bytes <= 512 && n_frames > 16)) return false;
    L.cap = cap;
    long long at = 8LL * row;                       // the pooled query
    const auto place = [&](int &p, long long bytes) {
        at = (at + 127) / 128 * 128;
        p = (int)std::min<long long>(at, INT32_MAX);
        at += bytes;
    };
    place(L.at_keys, 4LL * longest);
    place(L.at_tok, 24LL * cap);
    place(L.at_rows, (pack ? 2LL : 1LL) * cap * row_bytes);
    L.smem = (int)std::min<long long>(at, INT32_MAX);
    return cap > 1 && at <= FRONT_SMEM;              // (a token each: a history of no more than a CTA's worth, left to the separate kernels)
}

template <typename T, int LPT, bool PACK>
pc_status launch(const pc_ctx *ctx, const FrontParams &P, const pc_front_plan &L, cudaStream_t stream) {
    static std::atomic<bool> set[PC_MAX_DEVICES];
    if (ctx->device < 0 || ctx->device >= PC_MAX_DEVICES) return PC_ERR_UNSUPPORTED;
    if (!set[ctx->device]) {
        PC_CUDA_TRY(cudaFuncSetAttribute(k_front<T, LPT, PACK>, cudaFuncAttributeMaxDynamicSharedMemorySize, FRONT_SMEM));
        set[ctx->device] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(L.clusters * L.ctas);
    cfg.blockDim = dim3(FRONT_THREADS);
    cfg.dynamicSmemBytes = L.smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = L.ctas;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    PC_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_front<T, LPT, PACK>, P));
    return PC_OK;
}

}  // namespace

bool pc_front_fits(const pc_ctx *ctx, const pc_cache *src, bool pack, pc_front_plan *plan) {
    return !ctx->timing_on && src->history.n_tokens > 0 && lay_out(ctx, src, pack, *plan);
}

pc_status pc_launch_front(pc_ctx *ctx, const pc_front_args &A, int32_t n_q, cudaStream_t stream) {
    const pc_layer_desc &D = ctx->desc;
    const pc_cache *src = A.src;
    const pc_segment *dst = A.dst;
    const pc_front_plan &L = A.plan;
    FrontParams P;
    P.ctas = L.ctas;
    P.cap = L.cap;
    P.at_keys = L.at_keys;
    P.at_tok = L.at_tok;
    P.at_rows = L.at_rows;
    P.row_bytes = D.n_kv_heads * D.head_dim * ctx->elem_size;
    P.k = static_cast<const char *>(src->history.k);
    P.v = static_cast<const char *>(src->history.v);
    P.pos = src->history.pos;
    P.valid = A.valid;
    P.d = D.head_dim;
    P.scale = (float)(1.0 / ((double)D.n_q_heads * std::sqrt((double)D.head_dim)));
    P.fx = reinterpret_cast<unsigned long long *>(ctx->qpool_fx);
    P.fx_scale = 1.0 / (4294967296.0 * (double)n_q);
    P.scores = A.scores;
    P.sel_idx = A.sel_idx;
    P.dst_k = dst ? static_cast<char *>(dst->k) : nullptr;
    P.dst_v = dst ? static_cast<char *>(dst->v) : nullptr;
    P.dst_pos = dst ? dst->pos : nullptr;
    P.rot_k = static_cast<char *>(A.k_rot_dst);
    P.delta_t = A.delta_t;
    P.n_frames = src->n_frames;
    P.status = ctx->status;
    P.wait_us = ctx->wait_limit_us;
    P.extra_tx = ctx->test_extra_tx;
    P.rope = ctx->rope;
    int first = 0, out = 0;
    for (int f = 0; f < src->n_frames; ++f) {
        P.f[f] = make_int4(first, src->frame_count[f], A.budget[f], out);
        first += src->frame_count[f];
        out += A.budget[f];
    }
    const bool wide = D.head_dim * ctx->elem_size > 256;             // fp32 heads of 128: 32 lanes a token
    if (D.dtype == PC_BF16) return dst ? launch<__nv_bfloat16, 16, true>(ctx, P, L, stream) : launch<__nv_bfloat16, 16, false>(ctx, P, L, stream);
    if (!wide) return dst ? launch<float, 16, true>(ctx, P, L, stream) : launch<float, 16, false>(ctx, P, L, stream);
    return dst ? launch<float, 32, true>(ctx, P, L, stream) : launch<float, 32, false>(ctx, P, L, stream);
}

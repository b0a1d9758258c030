// Token scoring and per-frame top-k selection (the "attention-relevant" retention of Sec. 3.4).
//
//   k_qprep  : one pass over Q: pooled query  q~[g][c] = sum_{h in group g} (1/n_q) sum_i (R(p_i) q_ih)[c]  (fixed-point
//              sums, deterministic) and, on request, the rotated bf16 queries the attention kernel reads
//   k_score  : s_j = 1/(Hq sqrt(d)) * sum_g q~_g . R(p_j) k_jg   — one pass over the history keys, HBM-bound
//   k_select : per frame the budget[f] best scores (ties to the lower index), ascending indices out
//
// The score of a key equals the mean scaled logit over all queries and heads because the logit is linear in the
// rotated query.  For one rotary pair (a, b) = elements (2i, 2i+1):
//   q_a (k_a cos - k_b sin) + q_b (k_a sin + k_b cos) = cos (q_a k_a + q_b k_b) + sin (q_b k_a - q_a k_b),
// and the angle is the same for every KV head, so the two brackets are summed over heads first and each pair costs
// one table look-up per token.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "pc_rows.cuh"
#include "pc_select.cuh"

namespace {

// ---------------------------------------------------------------------------------------------------------
// Query pass.  One read of Q serves both consumers of the rotated queries: the pooled query of the scoring pass
//   q~[g] = (1/n_q) sum_i sum_{h in g} R(p_i) q_ih
// and, for the tensor-core attention kernel, the rotated bf16 queries with log2(e)/sqrt(d) folded in (q_rot).
// A few warps share one query token: lane l of a warp reads the 16-byte chunks l, l + 32, ... of the warp's part of the
// row; 32 chunks span a multiple of d, so all of a lane's chunks hold the same rotary pairs and the lane needs PER/2 table
// entries.  A block keeps four tokens in work (as far as the row's parts leave it) and walks the tokens with a stride, the
// next token's row and position requested before the current one is turned; every thread sums its own elements over its
// tokens in registers.  At the end the sums go to one slab per token slot in shared memory; for each pooled element the threads
// add, in a fixed order, the heads and slots of QPREP_SUM_WARPS / parts tokens in fp32, turn that into a 64-bit fixed-point
// number (units of 2^-32), and go on in integers, up to the global accumulator with an integer atomic: integer addition is
// associative, so the pooled query does not depend on the order in which blocks arrive, and no fp32 sum has more terms than
// those tokens give it, however many a block works on: a thread that walks several tokens adds fewer slots, or, where it walks
// more than those tokens, keeps its own sums' roundings (all slots of a block in one fp32 sum and a thread's tokens as they
// come: scores 4 to 14 % further from a 64-bit evaluation).  The scoring kernel reads the accumulator as it is;
// nobody waits for a last block to turn it into floats.
// The kernel is bound by latency: a launch, one round trip for positions and rows, one for table entries, the sums, the
// atomics.  One block per two tokens (504 at 1,008 queries, each adding all pooled elements) and a last block that converted
// and cleared the accumulator took, with a scoring kernel of eight tokens behind it, 11.2 us at 1,008 queries of 24 heads
// (now 7.8), 23.6 at 4,032 (13.2), 9.0 at 135 (6.8), 6.1 at 64 fp32 queries of 4 heads (4.1).  Eight warps a block instead of
// sixteen 9.0 / 14.6 / 7.8; two or four copies of the accumulator 7.8 to 8.4 at 1,008.
// ---------------------------------------------------------------------------------------------------------
constexpr int QPREP_WARPS = 16;                     // most warps per block, unless one token needs more
constexpr int QPREP_SUM_WARPS = 8;                  // tokens whose elements are added in fp32, in warps
constexpr int QPREP_SLAB = 200 * 1024;              // most shared memory of a block (one token takes up to 128 KB: 32 parts of 4 x 32 chunks)
// A query row is cut into `parts` runs of CPW x 32 chunks, one warp each; a block holds `slots` tokens at a time, `run` of which
// go into one fp32 sum.
// KEEP: a thread's sums over its tokens carry what each addition rounds off into the next one (Kahan), two elements at a time.
template <typename T, int CPW /* chunks per lane of one warp's part of a query row */, int MAX_THREADS, bool KEEP>
__global__ void __launch_bounds__(MAX_THREADS, MAX_THREADS == 512 && !KEEP && CPW <= (sizeof(T) == 4 ? 3 : 2) ? 2 : 1) k_qprep(const T *__restrict__ q, const int32_t *__restrict__ q_pos, int n_q,
                                                int n_q_heads, int group, int d, int parts, int run, pc_rope_dev rope,
                                                float out_scale, T *__restrict__ q_rot, unsigned long long *fx,
                                                int32_t *status) {
    pc_grid_dep_wait();
    pc_grid_dep_launch();   // after the wait: the scoring kernel reads keys and positions ahead of its own
    constexpr int PER = Elem<T>::PER16, NP = PER / 2;
    extern __shared__ __align__(16) float slab[];                     // [slots][Hq*d]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int slots = (blockDim.x >> 5) / parts;
    const int row_len = n_q_heads * d, row_chunks = row_len / PER;
    const int slot = warp / parts, part = warp - slot * parts;
    const int chunk0 = part * CPW * 32 + lane, pair0 = ((lane * PER) % d) / 2, stride = gridDim.x * slots;
    const uint4 *src = reinterpret_cast<const uint4 *>(q) + chunk0;
    uint4 *dst = q_rot ? reinterpret_cast<uint4 *>(q_rot) + chunk0 : nullptr;
    int i = blockIdx.x * slots + slot;
    int4 pp = make_int4(0, 0, 0, 0);
    uint4 raw[CPW];
    float2 acc[CPW][NP], off[KEEP ? CPW : 1][KEEP ? NP : 1];
#pragma unroll
    for (int c = 0; c < CPW; ++c)
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            acc[c][u] = make_float2(0.f, 0.f);
            if constexpr (KEEP) off[c][u] = make_float2(0.f, 0.f);
        }
    if (i < n_q) {
        pp = __ldg(reinterpret_cast<const int4 *>(q_pos) + i);
#pragma unroll
        for (int c = 0; c < CPW; ++c) raw[c] = pc_ldg_stream(src + (size_t)i * row_chunks + c * 32);
    }
    while (i < n_q) {
        const int at = i;
        float2 cs[NP];
#pragma unroll
        for (int u = 0; u < NP; ++u) cs[u] = pc_rope_cs(rope, pair0 + u, pp.x, pp.y, pp.z, status, PC_WHERE_QPOOL_POS);
        i += stride;
        const bool more = i < n_q;
        if (more) pp = __ldg(reinterpret_cast<const int4 *>(q_pos) + i);
#pragma unroll
        for (int c = 0; c < CPW; ++c) {
            const uint4 cur = raw[c];
            if (more) raw[c] = pc_ldg_stream(src + (size_t)i * row_chunks + c * 32);
            float x[PER], r[PER];
            Elem<T>::unpack(cur, x);
#pragma unroll
            for (int u = 0; u < NP; ++u) {
                const float2 y = pc_rotate(x[2 * u], x[2 * u + 1], cs[u]);
                r[2 * u] = y.x;
                r[2 * u + 1] = y.y;
            }
#pragma unroll
            for (int u = 0; u < NP; ++u) {
                const float2 y = make_float2(r[2 * u], r[2 * u + 1]);
                if constexpr (KEEP) {
                    const float2 m1 = make_float2(-1.f, -1.f);
                    const float2 z = __ffma2_rn(off[c][u], m1, y), t = __fadd2_rn(acc[c][u], z);
                    off[c][u] = __ffma2_rn(z, m1, __ffma2_rn(acc[c][u], m1, t));
                    acc[c][u] = t;
                } else {
                    acc[c][u] = __fadd2_rn(acc[c][u], y);
                }
            }
            if (dst) {                                                  // the attention kernel's queries carry its scale
#pragma unroll
                for (int k = 0; k < PER; ++k) r[k] = __fmul_rn(r[k], out_scale);
                dst[(size_t)at * row_chunks + c * 32] = Elem<T>::pack(r);
            }
        }
    }
    if constexpr (KEEP)
#pragma unroll
        for (int c = 0; c < CPW; ++c)
#pragma unroll
            for (int u = 0; u < NP; ++u) acc[c][u] = __ffma2_rn(off[c][u], make_float2(-1.f, -1.f), acc[c][u]);
    float *mine = slab + (size_t)slot * row_len + (size_t)chunk0 * PER;
#pragma unroll
    for (int c = 0; c < CPW; ++c) {
        float4 *s4 = reinterpret_cast<float4 *>(mine + (size_t)c * 32 * PER);
#pragma unroll
        for (int k = 0; k < PER / 4; ++k) s4[k] = make_float4(acc[c][2 * k].x, acc[c][2 * k].y, acc[c][2 * k + 1].x, acc[c][2 * k + 1].y);
    }
    __syncthreads();
    const int n_out = (n_q_heads / group) * d;
    const int used = min(slots, n_q - (int)blockIdx.x * slots);        // slots that had a token
    // the sums of N elements over the slots w0 .. w0 + run - 1, token by token, head by head: chains of reads and additions, so
    // two elements go side by side where a thread has more than one
    auto add_up = [&](auto n, const float *const (&s)[2], int w0, long long (&total)[2]) {
        constexpr int N = decltype(n)::value;
        int at = w0 * row_len;
        float sum[2] = {0.f, 0.f};
        for (int left = (min(w0 + run, used) - w0) * group, h = group; left > 0; left -= 4) {
            float x[2][4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
#pragma unroll
                for (int i = 0; i < N; ++i) x[i][k] = k < left ? s[i][at] : 0.f;
                at += d;
                if (--h == 0) { h = group; at += row_len - group * d; }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int i = 0; i < N; ++i) sum[i] += x[i][k];
        }
#pragma unroll
        for (int i = 0; i < N; ++i) total[i] += __float2ll_rn(sum[i] * FX_ONE);
    };
    auto at_element = [&](int e) { return slab + (size_t)(e / d) * group * d + e % d; };
    int e = threadIdx.x;
    for (; e + (int)blockDim.x < n_out; e += 2 * blockDim.x) {
        const float *const s[2] = {at_element(e), at_element(e + blockDim.x)};
        long long total[2] = {0, 0};
        for (int w0 = 0; w0 < used; w0 += run) add_up(std::integral_constant<int, 2>{}, s, w0, total);
        atomicAdd(fx + e, (unsigned long long)total[0]);
        atomicAdd(fx + e + blockDim.x, (unsigned long long)total[1]);
    }
    if (e < n_out) {
        const float *const s[2] = {at_element(e), nullptr};
        long long total[2] = {0, 0};
        for (int w0 = 0; w0 < used; w0 += run) add_up(std::integral_constant<int, 1>{}, s, w0, total);
        atomicAdd(fx + e, (unsigned long long)total[0]);
    }
}

// ---------------------------------------------------------------------------------------------------------
// Score.  A warp takes a group of consecutive history tokens at a time: LPT lanes share a token's row, 16 bytes at a time,
// so 32 / LPT tokens lie side by side in the warp, TPL of them one after the other in a lane.  LPT chunks span a multiple of
// d, so all of a lane's chunks cover the same PER/2 rotary pairs (of different heads): it sums the two brackets over its
// chunks and needs PER/2 table look-ups per token.  For a pair (a, b) the two brackets are two-lane products of the pair as
// it comes out of the unpacking, (k_a, k_b), with (q_a, q_b) and with (q_b, -q_a): two two-lane fp32 multiply-adds per pair,
// no register shuffling.  The pooled query sits in shared memory in that form; one 16-byte read serves a lane's TPL tokens.
//
// The rows come by bulk copies (a group's rows are one run of memory) into a ring of stages that belongs to the warp: up to
// 200 KB an SM in flight while the warps compute.  Rows held in registers (two of a warp, sixteen warps an SM) put 64 KB in
// flight, and none of it while the row before was worked on.  A warp's first copies go out ahead of its wait for the pooled
// query: the query pass lets this kernel start only when everything before that pass has completed, so keys and positions
// are final.  Bound by DRAM at long histories (97 MB at 47 frames), by latency at short ones.  Steps of 24 / 8 heads, rows in
// registers against this: 12 frames 84.2 -> 81.4 us, 47 frames 150.4 -> 147.2, masked update of 24 frames 141.3 -> 136.5,
// 135-token frames 28.3 -> 27.4; 32 / 16 heads: 12 frames 115.7 -> 111.6, 47 frames 220.6 -> 209.8.  Eight warps 148.5 at 47
// frames; warps held to 80 registers and 8 of them, to be resident beside the query pass, 152.0 to 153.8.  A group's table look-ups are
// made a group ahead, the first ones ahead of the wait for the pooled query, so no sum waits for them: 11 frames of 420 tokens, 24 / 12 heads,
// 47.7 -> 46.9 us, 7 of 459, 24 / 8, 33.1 -> 32.8, 12 of 1,008 74.5 -> 74.2, longer ones level (both chains side by side in 157
// registers, or two chunk rows a turn: level as well).
// ---------------------------------------------------------------------------------------------------------
constexpr int SCORE_WARPS = 12;                      // most warps per block (fewer where two stages of each would not fit)
constexpr int SCORE_STAGES = 8;                     // most stages of a warp's ring
constexpr int SCORE_RING = 200 * 1024;              // bytes of a block's rings

template <typename T, int LPT /* lanes per token */, int TPL /* tokens per lane */>
__global__ void __launch_bounds__(SCORE_WARPS * 32, 1) k_score(const T *__restrict__ k, const int32_t *__restrict__ k_pos,
                                                               const uint8_t *__restrict__ valid, int n_src, int d, int parts, int stages, float scale,
                                                               pc_rope_dev rope, unsigned long long *fx, double fx_scale,
                                                               float *__restrict__ scores, int32_t *status, uint32_t wait_us, uint32_t extra_tx) {
    pc_grid_dep_launch();
    constexpr int PER = Elem<T>::PER16, NP = PER / 2, SIDE = 32 / LPT, TOK = SIDE * TPL;
    extern __shared__ __align__(128) unsigned char score_smem[];
    __shared__ __align__(8) unsigned long long bars[SCORE_WARPS * SCORE_STAGES];
    __shared__ int gave_up;
    float4 *qs = reinterpret_cast<float4 *>(score_smem);              // (q_a, q_b, q_b, -q_a) of (head, pair, lane of the token)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, lt = lane % LPT, side = lane / LPT, n_warps = blockDim.x >> 5;
    const int row_bytes = parts * LPT * 16, stage_bytes = TOK * row_bytes;
    const int n_groups = (n_src + TOK - 1) / TOK, step = gridDim.x * n_warps;
    const uint32_t ring = pc_smem_u32(score_smem) + parts * NP * LPT * 16 + warp * stages * stage_bytes;
    const uint32_t bar0 = pc_smem_u32(bars) + warp * SCORE_STAGES * 8;
    int grp = warp * gridDim.x + blockIdx.x;                          // small calls spread over the blocks first

    auto fill = [&](int stage, int group, uint32_t extra = 0) {       // one lane
        const uint32_t bytes = (uint32_t)(min(TOK, n_src - group * TOK) * row_bytes);
        pc_mbar_expect_tx(bar0 + 8 * stage, bytes + extra);
        pc_bulk_g2s(ring + stage * stage_bytes, reinterpret_cast<const char *>(k) + (size_t)group * stage_bytes, bytes, bar0 + 8 * stage);
    };
    if (lane == 0) {
        for (int s = 0; s < stages; ++s) pc_mbar_init(bar0 + 8 * s, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        for (int s = 0; s < stages && grp + s * step < n_groups; ++s) fill(s, grp + s * step, s == 0 ? extra_tx : 0u);
    }
    if (threadIdx.x == 0) gave_up = 0;
    int4 p[TPL];
    auto positions = [&](int group) {
#pragma unroll
        for (int i = 0; i < TPL; ++i) p[i] = __ldcg(reinterpret_cast<const int4 *>(k_pos) + min(group * TOK + i * SIDE + side, n_src - 1));
    };
    const ScoreTable<T> table(rope, lt, d);
    float2 cs[TPL][NP];
    auto look_up = [&]() {
#pragma unroll
        for (int i = 0; i < TPL; ++i) table.at(rope, p[i], cs[i], status);
    };
    if (grp < n_groups) {
        positions(grp);
        look_up();
        if (grp + step < n_groups) positions(grp + step);
    }
    pc_grid_dep_wait();                                               // the pooled query comes from the kernel before

    // the pooled query: the accumulator, scaled
    const int n_out = parts * LPT * PER;
    for (int idx = threadIdx.x; idx < parts * NP * LPT; idx += blockDim.x) {
        const int l = idx % LPT, u = (idx / LPT) % NP, g = idx / (LPT * NP);
        const longlong2 w = __ldcg(reinterpret_cast<const longlong2 *>(fx + (size_t)(g * LPT + l) * PER + 2 * u));
        const float a = (float)((double)w.x * fx_scale), b = (float)((double)w.y * fx_scale);
        qs[idx] = make_float4(a, b, b, -a);
    }
    __syncthreads();
    // Every block takes a ticket once it has read the accumulator; whoever finds that all others have read it, too, clears
    // it for the next call when its tokens are done.  Nobody waits for anybody, and nothing of this lives on the host, so a
    // captured graph replays it unchanged.
    unsigned long long ticket = 0;
    if (threadIdx.x == 0) ticket = atomicAdd(fx + n_out, 1ull);

    int stage = 0, phase = 0;
    for (; grp < n_groups; grp += step) {
        if (!__all_sync(0xffffffffu, pc_mbar_wait(bar0 + 8 * stage, phase, &gave_up, status, PC_WHERE_SCORE_WAIT, wait_us))) break;
        float s[TPL];
        score_rows<T, LPT, TPL>(ring + stage * stage_bytes + side * row_bytes + lt * 16, SIDE * row_bytes, parts, qs + lt, cs, s);
        __syncwarp();                                                 // every lane has read the stage
        if (lane == 0 && grp + stages * step < n_groups) fill(stage, grp + stages * step);
        if (grp + step < n_groups) {
            look_up();
            if (grp + 2 * step < n_groups) positions(grp + 2 * step);
        }
        if (++stage == stages) { stage = 0; phase ^= 1; }
        // a token's lanes are added up; with two tokens in a lane its lower lanes carry on with the first, the upper ones with the second
        float sum = s[0];
        int o = LPT / 2, i_out = 0;
        if constexpr (TPL == 2) {
            i_out = lt >= LPT / 2;
            sum = i_out ? s[1] : s[0];
            sum += __shfl_xor_sync(0xffffffffu, i_out ? s[0] : s[1], LPT / 2);
            o = LPT / 4;
        }
#pragma unroll
        for (; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lt % (LPT / TPL) == 0) {
            const int j = grp * TOK + i_out * SIDE + side;
            if (j < n_src) {
                float r = sum * scale;
                if (valid && !valid[j]) r = -INFINITY;
                scores[j] = r;
            }
        }
    }
    // a wait ran out: copies are in flight that this warp no longer waits for
    if (grp < n_groups && lane == 0) pc_let_copies_land();
    if (warp == 0 && __shfl_sync(0xffffffffu, ticket, 0) == (unsigned long long)(gridDim.x - 1)) {
        for (int e = lane; e < n_out; e += 32) fx[e] = 0;
        if (lane == 0) fx[n_out] = 0;
    }
}

// ---------------------------------------------------------------------------------------------------------
// Select.  One block per frame runs the block-level selection of pc_select.cuh and writes the kept tokens' indices in
// ascending order.
// ---------------------------------------------------------------------------------------------------------
template <int THREADS>
__global__ void __launch_bounds__(THREADS) k_select(const float *__restrict__ scores, const __grid_constant__ FrameTab tab,
                                                    int32_t *__restrict__ sel_idx, int32_t *status) {
    pc_grid_dep_launch();
    pc_grid_dep_wait();
    __shared__ SelectShared<THREADS> sm;
    const int4 fr = tab.f[blockIdx.x];
    if (fr.z <= 0 || fr.y <= 0) return;
    const int out0 = fr.w;
    frame_select<THREADS>(scores + fr.x, fr, sm, status, [&](int at, int idx) { sel_idx[out0 + at] = idx; });
}

// Enqueue the query pass and the scoring kernel on caller-given scratch (a context's, or the library's fixed array).
// fx: the fixed-point accumulator (Hkv*d sums and one ticket word), all zero on entry, filled by the
// query pass, read by the scoring kernel and zero again when that has run;
// q_rot / q_scale: where the rotated queries go as well and the factor folded into them.
template <typename T>
pc_status enqueue_score(const pc_layer_desc &D, int sm_count, const pc_rope_dev &rope, long long *fx, int32_t *status, const void *hist_k, const int32_t *hist_pos, int n_src, const void *q,
                        const int32_t *q_pos, int32_t n_q, const uint8_t *valid, float *scores, void *q_rot, float q_scale,
                        cudaStream_t stream, pc_ctx *ctx /* whose marks and wait limit; NULL: none */,
                        const pc_front_args *front = nullptr /* scores, selection and pack in one launch */) {
    constexpr int PER = Elem<T>::PER16;
    const int row = D.n_kv_heads * D.head_dim;
    const int group = D.n_q_heads / D.n_kv_heads;
    const int q_row = D.n_q_heads * D.head_dim;
    const int q_chunks = q_row / PER, chunks = row / PER;            // 16-byte chunks per query row / key row
    if (chunks % 32 || q_chunks % 32 || (32 * PER) % D.head_dim) return PC_ERR_UNSUPPORTED;
    const double fx_scale = 1.0 / (4294967296.0 * (double)n_q);
    // a row's chunk rows are dealt to `parts` warps of 1-4 chunk rows each
    const int qcpl = q_chunks / 32;
    int cpw = 0, parts = 0, slots = 0, summed = 0, q_smem = 0, q_threads = 0;
    const auto cut = [&](int chunk_rows) {
        cpw = chunk_rows;
        parts = qcpl / cpw;
        slots = std::max(1, QPREP_WARPS / parts);
        slots = std::max(1, std::min<int>(slots, (int)(QPREP_SLAB / ((size_t)q_row * sizeof(float)))));
        summed = std::min(slots, std::max(1, QPREP_SUM_WARPS / parts));
        q_smem = slots * q_row * (int)sizeof(float);
        q_threads = slots * parts * 32;
    };
    cut(qcpl % 3 == 0 ? 3 : (qcpl % 4 == 0 ? 4 : (qcpl % 2 == 0 ? 2 : 1)));
    if (parts > 32) return PC_ERR_UNSUPPORTED;
    int dev_id = 0;
    PC_CUDA_TRY(cudaGetDevice(&dev_id));
    if (dev_id < 0 || dev_id >= PC_MAX_DEVICES) return PC_ERR_UNSUPPORTED;
    if (ctx) pc_mark(ctx, PC_MARK_SCORE0, stream);
    // Blocks: as many as are resident at once, each walking over its share of the tokens.  Where a thread then adds up more tokens
    // than QPREP_SUM_WARPS gives one fp32 sum, it keeps the roundings (blocks of more than 512 threads have no registers for that
    // and come in more rounds instead).
    int q_blocks = 0, walked = 0;
#define PC_QPREP_LAUNCH(KERNEL, RUN)                                                                                 \
    {                                                                                                               \
        /* one limit for all sizes: the attribute is the kernel's, whichever thread and context calls */            \
        static std::atomic<bool> set[PC_MAX_DEVICES];                                                               \
        if (!set[dev_id]) {                                                                                         \
            PC_CUDA_TRY(cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, QPREP_SLAB));     \
            set[dev_id] = true;                                                                                     \
        }                                                                                                           \
        PC_LAUNCH((KERNEL), dim3(q_blocks), dim3(q_threads), q_smem, stream, static_cast<const T *>(q), q_pos, n_q, D.n_q_heads, group, \
                  D.head_dim, parts, RUN, rope, q_scale, static_cast<T *>(q_rot), reinterpret_cast<unsigned long long *>(fx), status); \
    }
#define PC_QPREP_CASE(CPW)                                                                                           \
    {                                                                                                               \
        /* resident blocks and the size they were looked up for, in one word: no reader sees half of a pair */      \
        static std::atomic<uint64_t> occ_of[PC_MAX_DEVICES];                                                        \
        const uint64_t key = (uint64_t)(q_smem + q_threads) << 32, known = occ_of[dev_id];                          \
        int occ = (known ^ key) >> 32 ? 0 : (int)known;                                                             \
        if (occ == 0) {                                                                                             \
            PC_CUDA_TRY(q_threads <= 512 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_qprep<T, CPW, 512, false>, q_threads, q_smem) \
                                         : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_qprep<T, CPW, 1024, false>, q_threads, q_smem)); \
            occ = std::max(1, occ);                                                                                 \
            occ_of[dev_id] = key | (uint32_t)occ;                                                                   \
        }                                                                                                           \
        q_blocks = std::min((n_q + slots - 1) / slots, sm_count * occ);                                             \
        if (q_threads > 512) q_blocks = std::max(q_blocks, (n_q + slots * summed - 1) / (slots * summed));          \
        walked = (n_q + q_blocks * slots - 1) / (q_blocks * slots);                                                 \
        if (q_threads > 512) PC_QPREP_LAUNCH((k_qprep<T, CPW, 1024, false>), std::max(1, summed / walked))          \
        else if (walked <= summed) PC_QPREP_LAUNCH((k_qprep<T, CPW, 512, false>), summed / walked)                  \
        else if (CPW == 4) { cut(2); continue; }                    /* no registers for both */                    \
        else PC_QPREP_LAUNCH((k_qprep<T, CPW == 4 ? 3 : CPW, 512, true>), std::max(1, summed / 2))                  \
    }
    for (;;) {
        switch (cpw) {
        case 3: PC_QPREP_CASE(3) break;        // 24 query heads x 128 bf16: four warps per token
        case 4: PC_QPREP_CASE(4) break;
        case 2: PC_QPREP_CASE(2) break;
        default: PC_QPREP_CASE(1) break;
        }
        break;
    }
#undef PC_QPREP_CASE
#undef PC_QPREP_LAUNCH
    PC_CUDA_TRY(cudaGetLastError());
    if (ctx) pc_mark(ctx, PC_MARK_QPOOL, stream);
    if (front) return pc_launch_front(ctx, *front, n_q, stream);
    const float scale = (float)(1.0 / ((double)D.n_q_heads * std::sqrt((double)D.head_dim)));
    const T *k = static_cast<const T *>(hist_k);
    const int lpt = std::max(16, D.head_dim / PER), row_bytes = row * (int)sizeof(T);
    // Two tokens per lane share each read of the pooled query, where every warp gets two stages of them.  Wider rows leave
    // fewer warps two stages, which pays once there are groups for all warps: 3 KB rows, 44,000 tokens 38.2 (one token) against
    // 32.6 us, 675 tokens 7.9 against 9.1; 4 KB rows 46.2 against 43.2, 8.8 against 10.9.
    const int room = SCORE_RING / (4 * (32 / lpt) * row_bytes);      // warps with two stages of two tokens per lane
    const bool two = room >= SCORE_WARPS || (room >= SCORE_WARPS / 2 && n_src > sm_count * SCORE_WARPS * (32 / lpt));
    const int tok = (two ? 2 : 1) * (32 / lpt), stage_bytes = tok * row_bytes, n_groups = (n_src + tok - 1) / tok;
    const int blocks = std::max(1, std::min(n_groups, sm_count)), need = (n_groups + blocks - 1) / blocks;
    // Short histories: as many warps as it takes to stage the pooled query quickly, and no more: one for every 40 of its elements.
    // Query pass, scores and selection of 675 tokens with 4 / 8 / 12 warps: 128 elements 8.7 / 7.8 / 7.9 us, 256 (bf16) 9.9 / 9.7 /
    // 9.9, 512 10.4 / 10.1 / 9.7, 1,024 10.9 / 10.2 / 10.0, 2,048 12.3 / 11.8 / 11.3; of 1,500 tokens: 128 elements 7.8 / 7.9 / 9.0,
    // 256 (fp32, 4 / 6 / 12 warps) 8.6 / 8.5 / 9.5, 1,024 10.6 / 11.0 / 10.9.
    const int warps = std::min({SCORE_WARPS, SCORE_RING / (2 * stage_bytes), std::max({4, need, row / 40})});
    const int stages = std::max(1, std::min({SCORE_STAGES, SCORE_RING / (warps * stage_bytes), (n_groups + blocks * warps - 1) / (blocks * warps)}));
    const int smem = row * 8 + warps * stages * stage_bytes;
#define PC_SCORE_CASE(LPT, TPL)                                                                                      \
    {                                                                                                               \
        static bool set[PC_MAX_DEVICES] = {};                                                                       \
        if (!set[dev_id]) {                                                                                         \
            PC_CUDA_TRY(cudaFuncSetAttribute(k_score<T, LPT, TPL>, cudaFuncAttributeMaxDynamicSharedMemorySize, SCORE_RING + 16 * 1024)); \
            set[dev_id] = true;                                                                                     \
        }                                                                                                           \
        PC_LAUNCH((k_score<T, LPT, TPL>), dim3(blocks), dim3(warps * 32), smem, stream, k, hist_pos, valid, n_src, D.head_dim, row_bytes / (lpt * 16), stages, scale, \
                  rope, reinterpret_cast<unsigned long long *>(fx), fx_scale, scores, status,                        \
                  ctx ? ctx->wait_limit_us : 0u, ctx ? ctx->test_extra_tx : 0u);                            \
    }
    if (lpt == 16) {
        if (two) PC_SCORE_CASE(16, 2) else PC_SCORE_CASE(16, 1)
    } else if constexpr (sizeof(T) == 4) {           // fp32 heads of 128
        if (two) PC_SCORE_CASE(32, 2) else PC_SCORE_CASE(32, 1)
    }
#undef PC_SCORE_CASE
    PC_CUDA_TRY(cudaGetLastError());
    if (ctx) pc_mark(ctx, PC_MARK_SCORE, stream);
    return PC_OK;
}

}  // namespace

// The shapes the query pass and the scoring kernel are built for: a key row of 512, 1024, 1536, 2048, 3072 or 4096 bytes
// over all KV heads, a query row that is a multiple of 512 bytes and splits into at most 32 warps' parts.
bool pc_score_supports(const pc_layer_desc &D) {
    const int elem = D.dtype == PC_BF16 ? 2 : 4, per = 16 / elem;
    const int row = D.n_kv_heads * D.head_dim, q_row = D.n_q_heads * D.head_dim;
    if (row % (32 * per) || q_row % (32 * per) || (32 * per) % D.head_dim) return false;
    const int cpl = row / per / 32, qcpl = q_row / per / 32;
    if (cpl != 1 && cpl != 2 && cpl != 3 && cpl != 4 && cpl != 6 && cpl != 8) return false;
    const int cpw = qcpl % 3 == 0 ? 3 : (qcpl % 4 == 0 ? 4 : (qcpl % 2 == 0 ? 2 : 1));
    return qcpl / cpw <= 32;
}

// Every host-side check of a scoring call, nothing enqueued.
pc_status pc_score_check(const pc_ctx *ctx, const pc_cache *src, const void *q, const int32_t *q_pos, int32_t n_q, const int32_t *budget,
                         const float *scores_override, const float *scores, const int32_t *sel_idx) {
    if (!ctx || !src || !budget) return PC_ERR_INVALID_ARG;
    const int n_frames = src->n_frames;
    if (n_frames < 0 || (n_frames > 0 && !src->frame_count)) return PC_ERR_INVALID_ARG;
    if (n_frames > PC_MAX_FRAMES) return PC_ERR_CAPACITY;
    pc_status st = pc_check_segment(&src->history, true);
    if (st != PC_OK) return st;
    const int n_src = src->history.n_tokens;
    if (n_src > ctx->desc.max_keys) return PC_ERR_CAPACITY;
    int64_t first = 0, out = 0;
    for (int f = 0; f < n_frames; ++f) {
        const int n = src->frame_count[f], b = budget[f];
        if (n < 0 || b < 0) return PC_ERR_INVALID_ARG;
        if (b > n) return PC_ERR_BUDGET;
        first += n;
        out += b;
    }
    if (first != n_src) return PC_ERR_INVALID_ARG;
    if (out > 0 && (!sel_idx || !pc_aligned16(sel_idx))) return PC_ERR_INVALID_ARG;
    if (scores_override) return reinterpret_cast<uintptr_t>(scores_override) & 3 ? PC_ERR_INVALID_ARG : PC_OK;   // read element by element: any float address will do
    if (n_src == 0) return PC_OK;
    if (!q || !q_pos || n_q <= 0 || !scores) return PC_ERR_INVALID_ARG;
    if (!pc_aligned16(q) || !pc_aligned16(q_pos) || !pc_aligned16(scores)) return PC_ERR_INVALID_ARG;
    if (n_q > ctx->desc.max_q) return PC_ERR_CAPACITY;
    return pc_score_supports(ctx->desc) ? PC_OK : PC_ERR_UNSUPPORTED;
}

pc_status pc_score_impl(pc_ctx *ctx, const pc_cache *src, const void *q, const int32_t *q_pos, int32_t n_q, const int32_t *budget,
                        const uint8_t *valid, const float *scores_override, float *scores, int32_t *sel_idx, void *q_rot_out,
                        cudaStream_t stream, bool select, const pc_front_args *front) {
    pc_status st = pc_score_check(ctx, src, q, q_pos, n_q, budget, scores_override, scores, sel_idx);
    if (st != PC_OK) return st;
    const int n_frames = src->n_frames, n_src = src->history.n_tokens;
    FrameTab tab;
    int first = 0, out = 0, longest = 0;
    for (int f = 0; f < n_frames; ++f) {
        const int n = src->frame_count[f], b = budget[f];
        longest = std::max(longest, n);
        tab.f[f] = make_int4(first, n, b, out);
        first += n;
        out += b;
    }
    const float *select_on = scores_override;
    pc_front_args here{src, budget, valid, scores, sel_idx, 0, nullptr, nullptr, {}};
    if (!scores_override) {
        if (n_src > 0) {
            const size_t row = (size_t)ctx->desc.n_kv_heads * ctx->desc.head_dim;
            if (ctx->qpool_dirty) {          // an earlier call stopped between the query pass and the scoring kernel
                PC_CUDA_TRY(cudaMemsetAsync(ctx->qpool_fx, 0, (row + 1) * sizeof(long long), stream));
                ctx->qpool_dirty = 0;
            }
            ctx->qpool_dirty = 1;
            if (!front && select && out > 0 && pc_front_fits(ctx, src, false, &here.plan)) front = &here;
            const float q_scale = pc_q_rot_scale(ctx->desc.head_dim);
            st = ctx->desc.dtype == PC_BF16
                     ? enqueue_score<__nv_bfloat16>(ctx->desc, ctx->sm_count, ctx->rope, ctx->qpool_fx, ctx->status, src->history.k,
                                                    src->history.pos, n_src, q, q_pos, n_q, valid, scores, q_rot_out, q_scale, stream, ctx, front)
                     : enqueue_score<float>(ctx->desc, ctx->sm_count, ctx->rope, ctx->qpool_fx, ctx->status, src->history.k,
                                            src->history.pos, n_src, q, q_pos, n_q, valid, scores, nullptr, 1.0f, stream, ctx, front);
            if (st != PC_OK) return st;
            ctx->qpool_dirty = 0;
            if (q_rot_out) ctx->q_rot_n = n_q;
        }
        select_on = scores;
    }
    if (!front && select && n_frames > 0 && out > 0) {
        if (scores_override) pc_mark(ctx, PC_MARK_SCORE, stream);
        // a thread per key, as far as a block goes: frames of 64 and 135 tokens take 2.4 and 2.5 us with 256
        // threads, 2.7 and 2.8 with 1,024; frames of 1,008 and 4,032 tokens 3.6 and 8.0 with 1,024, 3.8 and 8.9 with 512
        if (longest <= 256)
            PC_LAUNCH(k_select<256>, dim3(n_frames), dim3(256), 0, stream, select_on, tab, sel_idx, ctx->status);
        else
            PC_LAUNCH(k_select<1024>, dim3(n_frames), dim3(1024), 0, stream, select_on, tab, sel_idx, ctx->status);
        PC_CUDA_TRY(cudaGetLastError());
        pc_mark(ctx, PC_MARK_SELECT, stream);
    }
    return PC_OK;
}

extern "C" pc_status pc_score(pc_ctx *ctx, const pc_cache *src, const void *q, const int32_t *q_pos, int32_t n_q,
                              const int32_t *budget, const uint8_t *valid, const float *scores_override, float *scores,
                              int32_t *sel_idx, void *stream_) {
    return pc_score_impl(ctx, src, q, q_pos, n_q, budget, valid, scores_override, scores, sel_idx, nullptr,
                         static_cast<cudaStream_t>(stream_));
}

// ---------------------------------------------------------------------------------------------------------
// Scoring without a context and without any allocation.
//
// Meant for hosts that cannot call cudaMalloc at the point where they need scores: a process whose device memory
// was handed to its own arena at start-up and whose policy forbids driver allocations afterwards, or a
// latency-critical thread that cannot take the device-wide synchronisation a cudaMalloc / cudaFree implies.  Such
// callers cannot create a pc_ctx (pc_create allocates), so everything a context would hold for scoring — the rotary
// table and the fixed-point accumulator of the pooled query — lives in one file-scope device array of fixed size
// that every GPU loading this library carries until the process exits.
//
// In host code the array's name is only a handle; the device address is obtained once per device with
// cudaGetSymbolAddress while that device is current, and that pointer (never the symbol) is what kernels receive.
// ---------------------------------------------------------------------------------------------------------
namespace {

constexpr int STATIC_MAX_ROW = 1024;          // n_kv_heads * head_dim
constexpr int STATIC_MAX_ROPE = 32768;        // rotary table entries: sum over axes of max_pos * pairs on that axis
constexpr int STATIC_MAX_QROW = 12288;        // n_q_heads * head_dim: one row of the query pass's shared-memory slab
constexpr int STATIC_MAX_DEVICES = PC_MAX_DEVICES;

constexpr size_t STATIC_OFF_FX = 256;  /* first 256 bytes unused */       // long long [STATIC_MAX_ROW + 1 counter word]
constexpr size_t STATIC_OFF_ROPE = STATIC_OFF_FX + (size_t)STATIC_MAX_ROW * sizeof(long long) + 256;   // float2 [STATIC_MAX_ROPE]
constexpr size_t STATIC_BYTES = STATIC_OFF_ROPE + (size_t)STATIC_MAX_ROPE * sizeof(float2);    // 270,848 bytes

static __device__ __align__(256) unsigned char g_static_scratch[STATIC_BYTES];

// Rotary table in fp64, stored as fp32 (cos, sin): entry (axis a, position p, column m) = p * base^(-m / n_axis[a]).
// The first `clear` 64-bit words of `fx` are set to zero as well (the accumulator of the pooled query).
__global__ void __launch_bounds__(256) k_rope_table(float2 *__restrict__ tab, pc_rope_dev rope, double base, int total,
                                                    long long *__restrict__ fx, int clear) {
    pc_grid_dep_launch();
    pc_grid_dep_wait();
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < clear) fx[e] = 0;
    if (e >= total) return;
    const int a = e >= rope.off[2] ? 2 : (e >= rope.off[1] ? 1 : 0);
    const int na = rope.n_axis[a], local = e - rope.off[a];
    const int p = local / na, m = local % na;
    const double ang = (double)p * pow(base, -(double)m / (double)na);
    tab[e] = make_float2((float)cos(ang), (float)sin(ang));
}

// Device address of the static scratch on the current device; looked up on the first call per device.
pc_status static_scratch_base(unsigned char **base) {
    static unsigned char *addr[STATIC_MAX_DEVICES] = {};
    int dev = -1;
    PC_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= STATIC_MAX_DEVICES) return PC_ERR_UNSUPPORTED;
    unsigned char *p = __atomic_load_n(&addr[dev], __ATOMIC_ACQUIRE);
    if (!p) {
        void *sym = nullptr;
        PC_CUDA_TRY(cudaGetSymbolAddress(&sym, g_static_scratch));
        if (!sym) return PC_ERR_CUDA;
        p = static_cast<unsigned char *>(sym);
        __atomic_store_n(&addr[dev], p, __ATOMIC_RELEASE);   // every thread resolves the same address
    }
    *base = p;
    return PC_OK;
}

template <typename T>
pc_status launch_score_static(const pc_layer_desc &D, unsigned char *base, const void *hist_k, const int32_t *hist_pos,
                              int32_t n_src, const void *q, const int32_t *q_pos, int32_t n_q, const uint8_t *valid,
                              float *scores, int32_t *status, cudaStream_t stream) {
    long long *fx = reinterpret_cast<long long *>(base + STATIC_OFF_FX);
    float2 *tab = reinterpret_cast<float2 *>(base + STATIC_OFF_ROPE);

    pc_rope_dev rope;
    int total = 0;
    for (int a = 0; a < 3; ++a) {
        rope.n_axis[a] = (D.head_dim / 2 - a + 2) / 3;
        rope.max_pos[a] = D.max_pos[a];
        rope.off[a] = total;
        total += D.max_pos[a] * rope.n_axis[a];
    }
    rope.tab = tab;
    // the array keeps whatever the last call left: the table is rewritten before it is read, and the accumulator of the
    // pooled query, which must start at zero, is cleared by the same kernel
    const int row = D.n_kv_heads * D.head_dim;
    const int fx_words = row + 1;
    PC_LAUNCH(k_rope_table, dim3((std::max(total, fx_words) + 255) / 256), dim3(256), 0, stream, tab, rope, D.rope_base, total, fx,
              fx_words);
    PC_CUDA_TRY(cudaGetLastError());

    int sm_count = 0, dev = 0;
    PC_CUDA_TRY(cudaGetDevice(&dev));
    PC_CUDA_TRY(cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev));
    return enqueue_score<T>(D, sm_count, rope, fx, status, hist_k, hist_pos, n_src, q, q_pos, n_q, valid, scores, nullptr,
                            1.0f, stream, nullptr);
}

}  // namespace

extern "C" pc_status pc_score_tokens_static(const pc_layer_desc *desc, const void *hist_k, const int32_t *hist_pos,
                                            int32_t n_src, const void *q, const int32_t *q_pos, int32_t n_q,
                                            const uint8_t *valid, float *scores, int32_t *status, void *stream_) {
    if (!desc || !hist_k || !hist_pos || !q || !q_pos || !scores || !status || n_src <= 0 || n_q <= 0)
        return PC_ERR_INVALID_ARG;
    if (!pc_aligned16(hist_k) || !pc_aligned16(hist_pos) || !pc_aligned16(q) || !pc_aligned16(q_pos) ||
        !pc_aligned16(scores) || (reinterpret_cast<uintptr_t>(status) & 7u))
        return PC_ERR_INVALID_ARG;
    const pc_layer_desc &D = *desc;
    if (D.head_dim != 64 && D.head_dim != 128) return PC_ERR_UNSUPPORTED;
    if (D.dtype != PC_F32 && D.dtype != PC_BF16) return PC_ERR_UNSUPPORTED;
    if (D.n_q_heads <= 0 || D.n_kv_heads <= 0 || D.n_q_heads % D.n_kv_heads) return PC_ERR_UNSUPPORTED;
    if (!(D.rope_base > 1.0)) return PC_ERR_INVALID_ARG;
    const int row = D.n_kv_heads * D.head_dim;
    if (!pc_score_supports(D)) return PC_ERR_UNSUPPORTED;                      // before anything is enqueued
    int64_t rope_entries = 0;
    for (int a = 0; a < 3; ++a) {
        if (D.max_pos[a] <= 0 || D.max_pos[a] > (1 << 20)) return PC_ERR_INVALID_ARG;
        rope_entries += (int64_t)D.max_pos[a] * ((D.head_dim / 2 - a + 2) / 3);
    }
    if (row > STATIC_MAX_ROW || rope_entries > STATIC_MAX_ROPE || D.n_q_heads * D.head_dim > STATIC_MAX_QROW) {
        fprintf(stderr,
                "packcache: pc_score_tokens_static: shape exceeds the fixed scratch (n_kv_heads*head_dim %d > %d, or "
                "rotary table %lld > %d entries, or n_q_heads*head_dim > %d)\n",
                row, STATIC_MAX_ROW, (long long)rope_entries, STATIC_MAX_ROPE, STATIC_MAX_QROW);
        return PC_ERR_CAPACITY;
    }
    unsigned char *base = nullptr;
    pc_status st = static_scratch_base(&base);
    if (st != PC_OK) return st;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    return D.dtype == PC_BF16
               ? launch_score_static<__nv_bfloat16>(D, base, hist_k, hist_pos, n_src, q, q_pos, n_q, valid, scores, status, stream)
               : launch_score_static<float>(D, base, hist_k, hist_pos, n_src, q, q_pos, n_q, valid, scores, status, stream);
}

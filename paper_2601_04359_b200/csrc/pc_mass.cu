// Attention mass of every cached key on tcgen05 tensor cores (Sec. 3.4: retention guided by the attention a token
// receives):  mass_j = 1/(n_q Hq) * sum over query rows (i, h) of softmax_j((R q_ih).(R k_j,g(h))/sqrt(d)).
//
// The call follows an attention call on the same context and reuses what that call left behind: the rotated keys and
// the rotated, pre-scaled queries (base-2 logits) in the context's scratch, and the log-sum-exp of every query row that
// the attention kernel wrote.  With the normaliser of every row known, a key's mass is a plain column sum of
// 2^(s_ij - lse2_i), so no running maximum and no second operand are needed:
//
//   k_mass_tc      a unit = two 128-key tiles of one KV head, which stay in shared memory while the query tiles of the
//                  head's group stream through a four-stage TMA ring, each stage feeding both key tiles (a unit of a
//                  single key tile reads every query tile twice as often from L2 for no gain).  Persistent CTAs, one per
//                  SM, share the line of (unit, query tile) steps evenly: a CTA's run usually crosses from one unit into
//                  the next, and a unit's sums come in up to MASS_PARTS pieces.  (A CTA per unit left SMs idle in its last
//                  wave, as many as 38 %: 24 / 8 heads, 1,008 queries
//                  x 5,168 keys 70.7 us against 43.7, 9,200 72.9 / 70.5, 12,980 106.3 / 95.6; 16 / 16, 300 x 1,200 10.1 / 9.9;
//                  8 / 8, 1,500 x 4,000, a unit per CTA either way, 21.8 / 22.1.)  The step's
//                  normalisers go into an eight-slot ring beside it, fetched by the warp that issues the copies (laid out by a kernel of its own for a bulk
//                  copy first: guided steps of 28 to 294 tokens 2 to 10 % longer, of 1,008 0.8 % at 12 frames).  S^T = K Q^T (keys on the TMEM lanes,
//                  queries on the columns) goes to one of two TMEM buffers per key tile.  Sixteen warps turn scores
//                  into sums: per key tile and column half one warp per TMEM lane quadrant, one key per thread, 64
//                  columns per step: 2^(s + (-lse2)) added up in registers.  Four such warps share each scheduler, so
//                  the waits of one hide behind the exponentials of the others; with two warps per scheduler (128
//                  columns per thread) and a per-step meeting of the warps to stage the normalisers, a third of
//                  every step was dead time.  The kernel is bound by the exponentials.
//   k_mass_reduce  adds the partial sums of the KV heads, column halves and pieces in a fixed order, divides by n_q Hq and drops the padding rows
//                  between segments.
// Every wait is bounded as in the attention kernel.
#include <algorithm>

#include "pc_tc.cuh"

namespace {

using namespace pc_tc;

constexpr int MASS_PARTS = 4;              // most pieces of a unit
constexpr int MASS_THREADS = 640;          // warp 0 TMA + TMEM owner, warp 1 MMA issuer, warps 4-19 column sums
constexpr int Q_STAGES = 4;
constexpr int L_SLOTS = 8;                 // normaliser ring: deeper than query stages + score buffers, see the producer

constexpr int SM_K = 0;                                  // 2 key tiles
constexpr int SM_Q = SM_K + 2 * TILE_BYTES;              // Q_STAGES query tiles
constexpr int SM_BAR = SM_Q + Q_STAGES * TILE_BYTES;
constexpr int SM_LSE = SM_BAR + 256;                     // [L_SLOTS][128] fp32: minus the base-2 normaliser of each query row
constexpr int SM_TOTAL = SM_LSE + L_SLOTS * TILE * 4;
constexpr int SM_ALLOC = SM_TOTAL + 1024;

enum { BAR_K = 0, BAR_QFULL = 1, BAR_QEMPTY = BAR_QFULL + Q_STAGES, BAR_SFULL = BAR_QEMPTY + Q_STAGES /* [tile][buffer] */,
       BAR_SEMPTY = BAR_SFULL + 4, BAR_LFULL = BAR_SEMPTY + 4, BAR_DONE = BAR_LFULL + L_SLOTS,
       BAR_KFREE = BAR_DONE + 1, N_BARS = BAR_KFREE + 1 };
static_assert(N_BARS * 8 + 16 <= 256, "barrier area");

struct MassParams {
    int n_q, n_q_heads, group, n_tb, n_kv_tiles, pairs;    // pairs = key-tile pairs per KV head
    const float *lse;      // [n_q][Hq] natural log
    // Partial sums, [slot][2 key tiles][2 column halves][128].  A piece's slot is its unit's number plus its CTA's: along the line of
    // steps one or both of them grow at every change, so no two pieces share a slot and there are at most units + n_cta of them.
    float *part;
    int32_t *status;
    int n_cta, n_steps;    // persistent CTAs; steps (query tiles of the head's group) of a unit
    int run, longer;       // steps of a CTA's run; the first `longer` CTAs take one more
    uint32_t wait_us;      // limit of every bounded wait in microseconds (0 = about one second)
    uint32_t extra_tx;     // test hook: bytes the first barrier expects beyond what is sent (0 = off)
};
__host__ __device__ __forceinline__ int run_start(const MassParams &P, int c) { return c * P.run + min(c, P.longer); }
// the CTA whose run holds step x
__host__ __device__ __forceinline__ int cta_of_step(const MassParams &P, int x) {
    const int head = P.longer * (P.run + 1);
    return x < head ? x / (P.run + 1) : P.longer + (x - head) / P.run;
}

// WHOLE: every CTA has one unit and all of it (n_cta = units), which needs none of what a change of unit takes in the loops.  The
// three launches, 24 / 8 heads, 400 queries x 3,344 keys: 23.8 -> 23.3 us, and 22.5 with the divisions of the first unit and of the
// reduction ahead of their waits; 8 / 8, 64 x 20: 6.9 -> 6.1 -> 5.6.
template <bool WHOLE>
__global__ void __launch_bounds__(MASS_THREADS, 1)
k_mass_tc(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
          const __grid_constant__ MassParams P) {
    pc_grid_dep_launch();
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *gen = smem_raw + (base - smem_u32(smem_raw));
    volatile int *abort_flag = reinterpret_cast<volatile int *>(gen + SM_BAR + N_BARS * 8);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(gen + SM_BAR + N_BARS * 8 + 8);
    const uint32_t bar0 = base + SM_BAR;
    auto bar = [&](int i) { return bar0 + 8u * i; };

    // from one lane: known to be uniform, addresses and descriptors stay in uniform registers (guided step of 12 frames 130.8 -> 130.2 us)
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int G0 = run_start(P, blockIdx.x), G1 = run_start(P, blockIdx.x + 1);     // never empty
    const int unit0 = WHOLE ? (int)blockIdx.x : G0 / P.n_steps, g0 = unit0 / P.pairs, pair0 = unit0 - g0 * P.pairs;
    const int n_t = WHOLE ? min(2, P.n_kv_tiles - 2 * pair0) : 2;

    if (threadIdx.x == 0) {
        mbar_init(bar(BAR_K), 1);
        for (int s = 0; s < Q_STAGES; ++s) {
            mbar_init(bar(BAR_QFULL + s), 1);
            mbar_init(bar(BAR_QEMPTY + s), 1);
        }
        for (int i = 0; i < 4; ++i) {
            mbar_init(bar(BAR_SFULL + i), 1);
            mbar_init(bar(BAR_SEMPTY + i), 256);
        }
        for (int i = 0; i < L_SLOTS; ++i) mbar_init(bar(BAR_LFULL + i), 1);
        mbar_init(bar(BAR_DONE), 1);
        mbar_init(bar(BAR_KFREE), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 0) {   // two score buffers of 128 columns per key tile
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    pc_grid_dep_wait();   // from here on the rotated K / Q of the attention call and the normalisers are read

    if (warp == 0) {
        // ---------------------------------------------------------------- TMA producer
        // Ring stages, score buffers and normaliser slots follow the step count of the whole run (gs).  One lane issues the copies; all of them fetch
        // the step's normalisers (a query's values of all heads lie side by side, so a step's are one word of every row), ahead of the wait
        // for the stage.
        bool alive = true;
        int gs = 0, un = 0, unit = unit0, g = g0, pair = pair0;
        auto wait = [&](int b, int parity) {
            return __all_sync(0xffffffffu, mbar_wait(bar(b), parity, abort_flag, P.status, PC_WHERE_MASS_WAIT, P.wait_us));
        };
        float *const norms = reinterpret_cast<float *>(gen + SM_LSE);
        for (int x = G0; x < G1 && alive; ++un) {
            if (un > 0) {
                ++unit;
                if (++pair == P.pairs) { pair = 0; ++g; }
            }
            const int s0 = x - unit * P.n_steps, n = min(P.n_steps - s0, G1 - x), jt0 = 2 * pair;
            x += n;
            if (!WHOLE && un > 0) alive = wait(BAR_KFREE, (un - 1) & 1);
            if (!alive) break;
            if (lane == 0) {
                mbar_expect_tx(bar(BAR_K), n_t * TILE_BYTES + (un == 0 ? P.extra_tx : 0u));
                for (int t = 0; t < n_t; ++t) {
                    const int jt = min(jt0 + t, P.n_kv_tiles - 1);       // an odd tile count: the last tile twice, one copy dropped
                    tma_load_2d(base + SM_K + t * TILE_BYTES, &map_k, g * TILE, jt * TILE, bar(BAR_K));
                    tma_load_2d(base + SM_K + t * TILE_BYTES + HALF_BYTES, &map_k, g * TILE + 64, jt * TILE, bar(BAR_K));
                }
            }
            for (int s = s0; s < s0 + n && alive; ++s, ++gs) {
                const int st = gs % Q_STAGES, use = gs / Q_STAGES;
                const int tb = s / P.group, h = g * P.group + s % P.group;
                float lse[TILE / 32];
#pragma unroll
                for (int k = 0; k < TILE / 32; ++k) {
                    const int row = tb * TILE + k * 32 + lane;
                    lse[k] = row < P.n_q ? -1.4426950408889634f * __ldcg(P.lse + (size_t)row * P.n_q_heads + h) : -INFINITY;
                }
                if (use > 0) alive = wait(BAR_QEMPTY + st, (use - 1) & 1);
                if (!alive) break;
                if (lane == 0) {
                    mbar_expect_tx(bar(BAR_QFULL + st), TILE_BYTES);
                    tma_load_2d(base + SM_Q + st * TILE_BYTES, &map_q, h * TILE, tb * TILE, bar(BAR_QFULL + st));
                    tma_load_2d(base + SM_Q + st * TILE_BYTES + HALF_BYTES, &map_q, h * TILE + 64, tb * TILE, bar(BAR_QFULL + st));
                }
                // The step's normalisers go to slot gs mod 8.  Its previous tenant, step gs - 8, is out of use: this point
                // is reached after the products of step gs - 4 completed, those needed the score buffers of step gs - 6
                // released, and a buffer is released only after the step before it was summed up.
                const int slot = gs % L_SLOTS;
#pragma unroll
                for (int k = 0; k < TILE / 32; ++k) norms[slot * TILE + k * 32 + lane] = lse[k];
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(BAR_LFULL + slot));
            }
            if constexpr (WHOLE) break;
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------------- MMA issuer (converged warp, one elected lane)
        const bool lead = elect_one();
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
        bool alive = true;
        int gs = 0, un = 0;
        for (int x = G0, end = (unit0 + 1) * P.n_steps; x < G1 && alive; ++un, end += P.n_steps) {
            const int n = min(end, G1) - x;
            x += n;
            alive = mbar_wait(bar(BAR_K), un & 1, abort_flag, P.status, PC_WHERE_MASS_WAIT, P.wait_us);
            for (int s = 0; s < n && alive; ++s, ++gs) {
                const int st = gs % Q_STAGES, quse = gs / Q_STAGES, b = gs & 1, use = gs >> 1;
                alive = mbar_wait(bar(BAR_QFULL + st), quse & 1, abort_flag, P.status, PC_WHERE_MASS_WAIT, P.wait_us);
                for (int t = 0; t < n_t && alive; ++t) {
                    if (use > 0) alive = mbar_wait(bar(BAR_SEMPTY + 2 * t + b), (use - 1) & 1, abort_flag, P.status, PC_WHERE_MASS_WAIT, P.wait_us);
                    if (!alive) break;
                    tc_fence_after();
                    const uint32_t ka = base + SM_K + t * TILE_BYTES, qa = base + SM_Q + st * TILE_BYTES;
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks) {
                        const uint32_t off = (ks >> 2) * HALF_BYTES + (ks & 3) * 32;
                        if (lead) mma_ss(tm + (2 * t + b) * TILE, desc_kmajor(ka + off), desc_kmajor(qa + off), IDESC_QK, ks > 0);
                    }
                    if (lead) tc_commit(bar(BAR_SFULL + 2 * t + b));
                }
                if (alive && lead) tc_commit(bar(BAR_QEMPTY + st));
            }
            if constexpr (WHOLE) break;
            if (alive && lead) tc_commit(bar(BAR_KFREE));       // the unit's key tiles may be overwritten
        }
        // nothing of ours may still be running on the tensor core when TMEM is freed
        if (lead) tc_commit(bar(BAR_DONE));
        __syncwarp();
        pc_mbar_drain(bar(BAR_DONE), 0, P.status, PC_WHERE_MASS_WAIT);
    } else if (warp >= 4 && (warp - 4) >> 3 < n_t) {
        // ---------------------------------------------------------------- column sums: one key and 64 query columns per thread
        const int cw = warp - 4;
        const int t = cw >> 3, hf = (cw >> 2) & 1;        // key tile and column half of this warp
        const int quad = warp & 3;                        // TMEM lane quadrant this warp may touch
        const int r = quad * 32 + lane;                   // key row of the tile
        const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
        const float *lse_s = reinterpret_cast<const float *>(gen + SM_LSE) + hf * 64;
        float2 acc0 = make_float2(0.f, 0.f), acc1 = make_float2(0.f, 0.f);
        bool alive = true;
        int unit = unit0;
        auto put = [&]() { P.part[(((size_t)unit + blockIdx.x) * 4 + 2 * t + hf) * TILE + r] = (acc0.x + acc0.y) + (acc1.x + acc1.y); };
        int unit_left = min((unit + 1) * P.n_steps, G1) - G0;    // steps of the run that are left in the unit
        for (int s = 0; s < G1 - G0 && alive; ++s) {
            const int b = s & 1, use = s >> 1, slot = s % L_SLOTS;
            alive = __all_sync(0xffffffffu, mbar_wait(bar(BAR_SFULL + 2 * t + b), use & 1, abort_flag, P.status, PC_WHERE_MASS_WAIT, P.wait_us) &&
                                                mbar_wait(bar(BAR_LFULL + slot), (s / L_SLOTS) & 1, abort_flag, P.status, PC_WHERE_MASS_WAIT, P.wait_us));
            if (!alive) break;
            tc_fence_after();
            uint32_t sv[64];
            const uint32_t s_addr = tmem + lane_addr + (2 * t + b) * TILE + hf * 64;
            tmem_ld32(s_addr, sv);
            tmem_ld32(s_addr + 32, sv + 32);
            tmem_wait_ld();
            tc_fence_before();
            mbar_arrive(bar(BAR_SEMPTY + 2 * t + b));     // the buffer may take the scores of step s + 2
            const float4 *nl = reinterpret_cast<const float4 *>(lse_s + slot * TILE);
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                const float4 m = nl[c];                   // the same address in every lane: a broadcast
                float2 x = add2(make_float2(__uint_as_float(sv[4 * c]), __uint_as_float(sv[4 * c + 1])), make_float2(m.x, m.y));
                float2 y = add2(make_float2(__uint_as_float(sv[4 * c + 2]), __uint_as_float(sv[4 * c + 3])), make_float2(m.z, m.w));
                x.x = fast_exp2(x.x); x.y = fast_exp2(x.y);
                y.x = fast_exp2(y.x); y.y = fast_exp2(y.y);
                acc0 = add2(acc0, x);
                acc1 = add2(acc1, y);
            }
            if (!WHOLE && --unit_left == 0) {                // the unit, or this CTA's piece of it, is done
                put();
                acc0 = acc1 = make_float2(0.f, 0.f);
                ++unit;
                unit_left = min(P.n_steps, G1 - unit * P.n_steps);
            }
        }
        if (WHOLE && alive) put();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
    // every thread has done with its waits: the flag is final, and copies may be in flight that nobody waited for
    if (threadIdx.x == 0 && *abort_flag) pc_let_copies_land();
}

struct ReduceParams {
    int n_seg, n_kv_heads;
    int seg_first[PC_MAX_SEGMENTS + 1];     // first key of each segment in the output order; [n_seg] = all keys
    int seg_tile0[PC_MAX_SEGMENTS];         // first tile of each segment in the rotated-key scratch
    float inv_rows;                         // 1 / (n_q Hq)
};

// One block per key tile, a thread per key and MASS_ROWS rows of threads that share out the KV heads, so that the pieces of
// different heads are read at the same time; the rows' sums are added in a fixed order.
constexpr int MASS_ROWS = 8;

__global__ void __launch_bounds__(TILE * MASS_ROWS) k_mass_reduce(const __grid_constant__ ReduceParams R, const __grid_constant__ MassParams P,
                                                                  float *__restrict__ mass) {
    __shared__ float rows[MASS_ROWS][TILE];
    pc_grid_dep_launch();
    const int jt = blockIdx.x, key = threadIdx.x % TILE, y = threadIdx.x / TILE;
    int s = 0;
    while (s + 1 < R.n_seg && jt >= R.seg_tile0[s + 1]) ++s;
    const int j = R.seg_first[s] + (jt - R.seg_tile0[s]) * TILE + key;             // key number; past the segment: padding rows
    int pieces = 0;
    auto pieces_of = [&](int g) {                  // the first piece's sums of KV head g, and how many pieces follow one another
        const int unit = g * P.pairs + jt / 2, x = unit * P.n_steps, first = cta_of_step(P, x);
        pieces = cta_of_step(P, x + P.n_steps - 1) - first + 1;
        return P.part + (((size_t)unit + first) * 4 + 2 * (jt & 1)) * TILE + key;
    };
    const float *p = pieces_of(y);                 // the divisions run under the tail of the kernel before
    pc_grid_dep_wait();
    float sum = 0.f;
    for (int g = y; g < R.n_kv_heads;) {
        float a = __ldcg(p), b = __ldcg(p + TILE);                     // the first piece's two column halves
        for (int piece = 1; piece < pieces; ++piece) {
            p += 4 * TILE;
            a += __ldcg(p);
            b += __ldcg(p + TILE);
        }
        sum += a + b;
        if ((g += MASS_ROWS) < R.n_kv_heads) p = pieces_of(g);
    }
    rows[y][key] = sum;
    __syncthreads();
    if (y > 0 || j >= R.seg_first[s + 1]) return;
#pragma unroll
    for (int k = 1; k < MASS_ROWS; ++k) sum += rows[k][key];
    mass[j] = sum * R.inv_rows;
}

// Number of persistent CTAs: the fewest steps of the longest run, a change of unit reckoned as three of them (the products and
// sums drain, the next key tiles load).  One CTA per SM, or a number that gives every CTA whole units or cuts every unit
// into equal pieces.  The shortest run is at least a unit's steps over MASS_PARTS - 1, so no unit has more than MASS_PARTS pieces.
int choose_mass_ctas(int units, int n_steps, int sm_count) {
    const int steps = units * n_steps, shortest = (n_steps + MASS_PARTS - 2) / (MASS_PARTS - 1);
    const int most = std::min(sm_count, steps / shortest);
    int best = most;
    long long best_cost = -1;
    for (int n = most; n >= 1 && n >= most / 2; --n) {
        const bool even = units % n == 0 || (n % units == 0 && n_steps % (n / units) == 0);
        if (!even && n != most) continue;
        const long long run = (steps + n - 1) / n;
        const long long cost = run + 3 * (even ? std::max(units / n, 1) - 1 : (run - 1) / n_steps + 1);
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best = n;
        }
    }
    return best;
}

}  // namespace

size_t pc_mass_part_floats(const pc_layer_desc *d, int sm_count, size_t k_rot_rows) {
    const size_t units = (size_t)d->n_kv_heads * ((k_rot_rows / TILE + 1) / 2);
    return (units + sm_count) * 4 * TILE;
}

extern "C" pc_status pc_attend_mass(pc_ctx *ctx, const float *lse, float *mass, int32_t n_keys, void *stream_) {
    if (!ctx || !lse || !mass) return PC_ERR_INVALID_ARG;
    if (!pc_aligned16(lse) || !pc_aligned16(mass)) return PC_ERR_INVALID_ARG;
    const pc_layer_desc &D = ctx->desc;
    if (!pc_tensor_core_shape(ctx) || ctx->attend_impl == 1) return PC_ERR_UNSUPPORTED;
    if (ctx->last_n_q <= 0 || ctx->last_n_seg <= 0) return PC_ERR_INVALID_ARG;   // no tensor-core attention call precedes
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);

    MassParams P{};
    ReduceParams R{};
    int tiles = 0, keys = 0;
    for (int s = 0; s < ctx->last_n_seg; ++s) {
        R.seg_first[s] = keys;
        R.seg_tile0[s] = tiles;
        keys += ctx->last_seg_n[s];
        tiles += (ctx->last_seg_n[s] + TILE - 1) / TILE;
    }
    R.seg_first[ctx->last_n_seg] = keys;
    if (n_keys != keys) return PC_ERR_INVALID_ARG;
    if ((size_t)tiles * TILE > ctx->k_rot_rows) return PC_ERR_CAPACITY;
    R.n_seg = ctx->last_n_seg;
    R.n_kv_heads = D.n_kv_heads;
    R.inv_rows = (float)(1.0 / ((double)ctx->last_n_q * D.n_q_heads));
    P.n_q = ctx->last_n_q;
    P.n_q_heads = D.n_q_heads;
    P.group = ctx->group;
    P.n_tb = (P.n_q + TILE - 1) / TILE;
    P.n_kv_tiles = tiles;
    P.pairs = (tiles + 1) / 2;
    P.n_steps = P.group * P.n_tb;
    const int units = D.n_kv_heads * P.pairs;
    if ((long long)units * P.n_steps > INT32_MAX) return PC_ERR_CAPACITY;
    P.n_cta = choose_mass_ctas(units, P.n_steps, ctx->sm_count);
    P.run = units * P.n_steps / P.n_cta;
    P.longer = units * P.n_steps % P.n_cta;
    P.lse = lse;
    P.part = ctx->mass_part;
    P.status = ctx->status;
    P.wait_us = ctx->wait_limit_us;
    P.extra_tx = ctx->test_extra_tx;

    CUtensorMap mq, mk;
    if (!make_map(&mq, ctx->q_rot, (uint64_t)P.n_q, (uint64_t)D.n_q_heads * D.head_dim) ||
        !make_map(&mk, ctx->k_rot, (uint64_t)tiles * TILE, (uint64_t)D.n_kv_heads * D.head_dim)) {
        fprintf(stderr, "packcache: cuTensorMapEncodeTiled failed\n");
        return PC_ERR_CUDA;
    }
    static bool attr_set[PC_MAX_DEVICES] = {};      // the attribute belongs to the device, not to the process
    if (ctx->device < 0 || ctx->device >= PC_MAX_DEVICES) return PC_ERR_UNSUPPORTED;
    if (!attr_set[ctx->device]) {
        PC_CUDA_TRY(cudaFuncSetAttribute(k_mass_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SM_ALLOC));
        PC_CUDA_TRY(cudaFuncSetAttribute(k_mass_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SM_ALLOC));
        attr_set[ctx->device] = true;
    }
    pc_mark(ctx, PC_MARK_MASS0, stream);
    if (P.n_cta == units) PC_LAUNCH(k_mass_tc<true>, dim3(P.n_cta), dim3(MASS_THREADS), SM_ALLOC, stream, mq, mk, P);
    else PC_LAUNCH(k_mass_tc<false>, dim3(P.n_cta), dim3(MASS_THREADS), SM_ALLOC, stream, mq, mk, P);
    PC_CUDA_TRY(cudaGetLastError());
    PC_LAUNCH(k_mass_reduce, dim3(tiles), dim3(TILE * MASS_ROWS), 0, stream, R, P, mass);
    PC_CUDA_TRY(cudaGetLastError());
    pc_mark(ctx, PC_MARK_MASS, stream);
    return PC_OK;
}

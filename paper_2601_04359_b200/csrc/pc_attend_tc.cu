// bf16 attention of one frame's queries over the compacted cache on tcgen05 tensor cores (Eq. 2, all keys visible).
//
// Launch sequence of pc_launch_attend_tc:
//   k_rope_rows   rotates K of every segment (3D rotary tables, from the stored positions) into a bf16 scratch whose
//                 segments start on 128-row boundaries, and rotates Q with log2(e)/sqrt(d) folded in.
//   k_attend_tc   persistent CTAs (one per SM) share the line of (item, key tile) steps evenly; an item = two 128-row
//                 query tiles that share a KV head (grouped-query packing).
//                 Warp 0 lane 0 drives TMA (K and V tiles, 128B swizzle, two stages each), warps 1 and 2 issue
//                 tcgen05.mma S = Q_t K^T of tile 0 and 1 (both operands K-major in shared memory) into TMEM, and warp 3
//                 O_t += P_t V of both with P_t read from TMEM and V MN-major in shared memory.  Warps 4-7 / 8-11 are the
//                 softmax groups of tile 0 / 1: tcgen05.ld the S row into registers, running max and sum in fp32 (base 2),
//                 write bf16 P beside it (handed over in two halves of 64 keys), and rescale O in TMEM only when
//                 the running max moved by more than 2^8.
//                 While one tile's softmax runs, the tensor core works on the other tile.
//                 An item that two CTAs share, as most are where runs cross items, is merged by the one with its first keys, at the end of its run.
//   k_combine     merges the (max, sum, O) partials of the other items that several CTAs worked on.  On request (pc_set_cluster_merge) the
//                 key ranges of one item are launched as a thread-block cluster instead and merge through distributed shared
//                 memory at the end of k_attend_tc.
//
// TMEM columns: S 0-127 (both tiles in turn), P0 128-191, P1 192-255, O0 256-383, O1 384-511 (128 lanes = the tile's rows).
// A score row stays in TMEM only until it is in its thread's registers, so one S serves both tiles, and P has columns of its own:
// a tile's next Q K^T waits for the other tile's scores to be read and no longer for its own P V, which wrote P over S and made
// softmax -> P V -> Q K^T one chain (3,030 cycles per 128 keys of both tiles, of which the tensor core, the exponentials and
// shared memory need 2,050 each).  What it took to get something from that, all on the critical path before: a wait
// whose phase is complete costs 75 cycles instead of 155 with the first question outside the bounded loop; one commit behind a
// group of multiply-adds (a second one in a row waits until the group has run: stages and query tiles are
// released by the softmax warps); Q K^T and P V from different warps (in one, the tensor core's queue of about two
// multiply-adds ran dry at every change); Q K^T of the two tiles from warps of two schedulers (the softmax warps beside
// an issuer of Q K^T take 1,600 instead of 1,400 cycles for a row's exponentials); sums held to their chunk of exponentials; a warp's
// number that the compiler knows to be uniform.  2,560 cycles now, bound by the softmax warps (the exponentials of a tile's 128 rows take
// 1,024 at 16 a clock, twice).
// That form -> this one, a call: the step at 12 frames 81.8 -> 78.8 us, at 47 157.8 -> 150.2, of 4,032-token frames 635 -> 588; the
// whole cache of 47 frames 618 -> 568 (1.15 PFLOP/s without the rotary pre-pass), five passes over 7,184 keys 486 -> 452; since the
// bounded wait lost its loop of questions 77.2, 148.5, 586, 569 and 450; with the merge in this kernel and the way out for a part that
// does not come, both sides in turn on one box, the step at 12 frames 75.5 -> 74.9, at 47 149.0 -> 147.3, of 4,032-token frames 589 -> 582, five passes
// 452 -> 445, the whole cache level.
// Every wait is bounded: a wait that runs out records PC_ERR_TIMEOUT and raises a CTA-wide abort flag; every later wait whose
// phase is not complete gives up within some ten microseconds, and the CTA still drains its multiply-adds and copies, frees TMEM and exits.
#include <algorithm>
#include <numeric>

#include "pc_tc.cuh"

namespace {

using namespace pc_tc;

constexpr int TC_THREADS = 384;
// Registers a thread: as launched (all that one CTA of this size can have), then of warps 0-3 and of the softmax warps 4-11, which hold
// a whole score row.  setmaxnreg.inc waits without a limit for registers that are not there, so the split may not exceed what the
// block was launched with; that the compiler gave it as many is checked before the first launch.
constexpr int REGS_LAUNCH = 65536 / TC_THREADS / 8 * 8, REGS_ISSUE = 72, REGS_SOFTMAX = 216;
constexpr int REGS_SPLIT = 128 * REGS_ISSUE + 256 * REGS_SOFTMAX;
static_assert(REGS_SPLIT <= TC_THREADS * REGS_LAUNCH && REGS_ISSUE % 8 == 0 && REGS_SOFTMAX % 8 == 0, "more registers than the block has");
constexpr int KV_STAGES = 2;
constexpr int MAX_SPLITS = 8;             // most parts of an item
constexpr int BOUNDARY_STEPS = 2;         // what a CTA's crossing into the next item costs, in steps
constexpr int MAX_FIXED_SPLITS = 4;       // most key ranges a caller can fix, and most of the cluster merge
constexpr float RESCALE_THRESHOLD = 8.0f;

// shared memory map (dynamic, 1024-byte aligned)
constexpr int SM_Q = 0;                                   // 2 tiles
constexpr int SM_K = SM_Q + 2 * TILE_BYTES;               // KV_STAGES tiles
constexpr int SM_V = SM_K + KV_STAGES * TILE_BYTES;       // KV_STAGES tiles
constexpr int SM_BAR = SM_V + KV_STAGES * TILE_BYTES;     // barriers etc.
constexpr int SM_ML = SM_BAR + 256;                       // (max, sum) of both tiles' rows for the cluster merge: 2 KB
constexpr int SM_TOTAL = SM_ML + 2 * TILE * 8;
constexpr int SM_ALLOC = SM_TOTAL + 1024;                 // slack for manual alignment

enum { BAR_Q = 0 /* [tile] */, BAR_QFREE = 2 /* [tile] */, BAR_VFULL = 4 /* [stage] */, BAR_EMPTY = 6 /* [step & 1] */, BAR_SFULL = 8 /* [tile] */,
       BAR_SFREE = 10 /* [tile] */, BAR_PHALF = 12 /* [tile][half] */, BAR_PVDONE = 16 /* [tile] */, BAR_DONE = 18, BAR_PART = 19, N_BARS = 20 };
static_assert(N_BARS * 8 + 12 <= 256, "barriers, abort flag and TMEM address share 256 bytes");

constexpr int SYNC_PARTS = 2, LEFT_PER_ITEM = 8;          // words of TcParams::sync
// How long a CTA with a first part looks for the second one before it leaves both to the last CTA
constexpr uint64_t PART_NS = 100000;

// TMEM columns
constexpr int TM_S = 0, TM_P = TILE, TM_O = 2 * TILE;     // scores; P of tile t at TM_P + 64 t; O of tile t at TM_O + 128 t

struct TcParams {
    int n_q, n_q_heads, group, n_tb, tiles_per_g, pairs_per_g, n_splits, n_kv_tiles;
    int n_items;      // (KV head, pair of query tiles)
    int persistent;   // 1: n_cta CTAs share the line of (item, key tile) steps evenly; 0: CTA (item, s) takes one of n_splits ranges
    int n_cta;
    int gap;          // steps an item boundary is reckoned as when the line is shared out (persistent form)
    int part_stride;  // partial slots reserved per item (most parts any item has)
    int n_seg;
    int cluster;      // 1: the KV ranges of one item form a thread-block cluster and merge through shared memory
    uint32_t wait_us; // limit of every bounded wait in microseconds (0 = about one second)
    uint32_t extra_tx; // test hook: bytes the first barrier expects beyond what is sent, so that its wait runs out (0 = off)
    int seg_tile_end[PC_MAX_SEGMENTS];
    int seg_n[PC_MAX_SEGMENTS];
    __nv_bfloat16 *out;
    float *lse;
    float *part_o;    // [item*S + s][2] tiles of 128 x 128 fp32, 16-byte unit (c4, r) at c4*128 + r
    float *part_ml;   // [item*S + s][2][128][2]
    // Merge: [0] number of the call, [1] tickets of CTAs that are done and, in the upper half, how many of them left a merge to the last one;
    // from SYNC_PARTS on, per item, the number of the call that left the second part; behind those, per item, tile and quarter, that of the
    // call that left the merge.
    uint32_t *sync;
    int leave_parts;  // test hook: every merge is left to the last CTA
    int32_t *status;
};

// ------------------------------------------------------------------------------------------------ rotary pre-pass
struct RopeJob {
    const __nv_bfloat16 *src;
    const int32_t *pos;
    __nv_bfloat16 *dst;
    int first_warp;    // one warp per slice
    int slices;        // consecutive slices that make a row and share its position record
    float scale;
};
struct RopeJobs { RopeJob job[PC_MAX_SEGMENTS + 1]; int n_jobs, total_warps; };

// One warp per slice of CPL x 32 16-byte chunks; key and query rows are cut into slices of one width (a query row is a whole number
// of key rows), so all warps of a launch carry the same load.  32 lanes x 8 elements = 256 is a multiple of d, so all of a lane's
// chunks (lane, lane + 32, ...) hold the same four rotary pairs: four table entries per lane serve them; the output scale (1
// for keys) is applied after the rotation, exactly as the query pass of the scoring stage does, so both give the same bits.  A
// slice's chunks are requested together with its position, before the table entries that wait for it.
// Bound by memory, so warps in flight count: a kernel per width, with the registers that this width needs (40 up to three
// chunks a lane, six blocks an SM).  One kernel for every width (64 registers, four blocks), rows of 3, 5, 6 and 7 chunks a lane
// taken chunk by chunk, against this, 7,184 keys: 8 KV heads 5.5 -> 5.6 us, 4 4.6 -> 4.4, 6 8.3 -> 4.9, 10 13.3 -> 6.2, 12 15.2 ->
// 7.7, 14 18.7 -> 7.9, 16 9.0 -> 9.0; 48,000 keys: 8 34.9 -> 33.3 (5.9 TB/s), 4 22.0 -> 17.9, 6 50.6 -> 23.6, 12 93 -> 47.
constexpr int rope_blocks(int cpl) { return cpl <= 3 ? 6 : (cpl <= 7 ? 4 : 2); }
template <int CPL /* chunks per lane */>
__global__ void __launch_bounds__(256, rope_blocks(CPL)) k_rope_rows(const __grid_constant__ RopeJobs jobs, pc_rope_dev rope, int d, int32_t *status) {
    pc_grid_dep_launch();
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int ji = 0;
    while (ji + 1 < jobs.n_jobs && warp >= jobs.job[ji + 1].first_warp) ++ji;
    const RopeJob &J = jobs.job[ji];
    const int slice = warp - J.first_warp, pair0 = ((lane * 8) % d) / 2;
    pc_grid_dep_wait();
    if (warp >= jobs.total_warps) return;
    const size_t at = (size_t)slice * (CPL * 32) + lane;
    const uint4 *src = reinterpret_cast<const uint4 *>(J.src) + at;
    uint4 *dst = reinterpret_cast<uint4 *>(J.dst) + at;
    const float scale = J.scale;
    uint4 v[CPL];
#pragma unroll
    for (int c = 0; c < CPL; ++c) v[c] = pc_ldg_stream(src + c * 32);
    const int4 pp = __ldg(reinterpret_cast<const int4 *>(J.pos) + slice / J.slices);
    bool bad = false;
    float2 cs[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) cs[u] = pc_rope_cs_clamped(rope, pair0 + u, pp.x, pp.y, pp.z, bad);
    if (bad) pc_flag(status, PC_ERR_INVALID_ARG, PC_WHERE_ROPE_POS);
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
        const uint32_t w[4] = {v[c].x, v[c].y, v[c].z, v[c].w};
        uint32_t o[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float2 y = pc_rotate(pc_bf16_lo(w[u]), pc_bf16_hi(w[u]), cs[u]);
            o[u] = pc_pack_bf16(__fmul_rn(y.x, scale), __fmul_rn(y.y, scale));
        }
        dst[c * 32] = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

// ------------------------------------------------------------------------------------------------ main kernel
__device__ __forceinline__ void kv_tile_info(const TcParams &P, int jt, int &seg, int &local, int &n_valid) {
    seg = 0;
    int start = 0;
    while (seg + 1 < P.n_seg && jt >= P.seg_tile_end[seg]) { start = P.seg_tile_end[seg]; ++seg; }
    local = jt - start;
    n_valid = min(TILE, P.seg_n[seg] - local * TILE);
}

// ---- work decomposition.  The (item, key tile) pairs of a call form one line of n_items * n_kv_tiles steps, item-major.
// A CTA takes a contiguous run of it.  Persistent form: n_cta CTAs (one per SM) share the line evenly, so a CTA's run
// usually crosses from one item into the next; set-up (barriers, tensor memory) is paid once per CTA, the next item's
// queries and first keys arrive under the current item's last steps, and all SMs finish together.  Split form: CTA
// (item, s) takes the s-th of n_splits equal ranges of one item (used when the caller fixes the number of key ranges, and
// by the cluster merge).  The part of an item one CTA works on is a "unit"; an item's units are numbered by "part".
//
// A CTA that crosses from one item into the next spends the time of two to three steps on the boundary (the last PV drains, O
// is read out, the tensor core waits for the next item's first probabilities).  So the line is shared out with `gap` further
// places behind every item, on which no step lies.
__host__ __device__ __forceinline__ long long line_length(const TcParams &P) { return (long long)P.n_items * (P.n_kv_tiles + P.gap); }
__device__ __forceinline__ long long line_cut(const TcParams &P, int c) {        // first step of CTA c (persistent form)
    const int pitch = P.n_kv_tiles + P.gap;
    const long long v = line_length(P) * c / P.n_cta, item = v / pitch;
    return item * P.n_kv_tiles + min((int)(v - item * pitch), P.n_kv_tiles);
}
__device__ __forceinline__ void cta_run(const TcParams &P, int c, long long &g0, long long &g1) {
    if (P.persistent) {
        g0 = line_cut(P, c);
        g1 = line_cut(P, c + 1);
    } else {
        const int item = c / P.n_splits, s = c % P.n_splits;
        g0 = (long long)item * P.n_kv_tiles + (long long)P.n_kv_tiles * s / P.n_splits;
        g1 = (long long)item * P.n_kv_tiles + (long long)P.n_kv_tiles * (s + 1) / P.n_splits;
    }
}
// persistent form: the CTA whose run holds key tile j of an item
__host__ __device__ __forceinline__ int cta_of_step(const TcParams &P, int item, int j) {
    const long long L = line_length(P), v = (long long)item * (P.n_kv_tiles + P.gap) + j;
    return (int)(((v + 1) * P.n_cta + L - 1) / L) - 1;
}
// number of parts of an item, and the part the unit of CTA c is
__device__ __forceinline__ void item_parts(const TcParams &P, int item, int c, int &part, int &parts) {
    if (P.persistent) {
        const int first = cta_of_step(P, item, 0);
        const int last = cta_of_step(P, item, P.n_kv_tiles - 1);
        part = c - first;
        parts = last - first + 1;
    } else {
        part = c % P.n_splits;
        parts = P.n_splits;
    }
}
struct Unit { int item, jb, n_j; };   // key tiles jb .. jb + n_j - 1 of an item
__device__ __forceinline__ Unit unit_at(const TcParams &P, long long g, long long g1) {
    Unit u;
    u.item = (int)(g / P.n_kv_tiles);
    u.jb = (int)(g - (long long)u.item * P.n_kv_tiles);
    u.n_j = (int)min((long long)(P.n_kv_tiles - u.jb), g1 - g);
    return u;
}

// arrival without a branch around it
__device__ __forceinline__ void arrive_if(bool who, uint32_t bar) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %1, 0;\n\t@p mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}" ::"r"(bar), "r"((uint32_t)who) : "memory");
}
// Wait of a whole warp.  The first question stands alone: a phase that is complete is seen in 75 to 85 cycles; through the loop
// that the bounded wait began with once it took 155.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int32_t *status, uint32_t limit_us) {
    if (__builtin_expect(__all_sync(0xffffffffu, pc_mbar_try(bar, parity)), 1)) return true;
    return __all_sync(0xffffffffu, pc_mbar_wait(bar, parity, abort_flag, status, PC_WHERE_ATTN_WAIT, limit_us));
}

// Merges that were left, a warp of the last CTA per (item, tile, quarter), with the merge kernel's order and arithmetic: 32 rows, one a lane.
// A function of its own: as part of the kernel's code it made every call 0.3 us longer (the step at 12 frames 70.7 against 71.0 us, 70.5 without it).
__device__ __noinline__ void merge_left(const TcParams &P, uint32_t call, int w, int lane) {
    for (int e = w; e < P.n_items * LEFT_PER_ITEM; e += (TC_THREADS - 128) / 32) {
        if (__ldcg(P.sync + SYNC_PARTS + P.n_items + e) != call) continue;
        const int item = e / LEFT_PER_ITEM, t = (e >> 2) & 1, r = (e & 3) * 32 + lane;
        const int T = 2 * (item % P.pairs_per_g) + t, h = item / P.pairs_per_g * P.group + T % P.group, row = T / P.group * TILE + r;
        if (row >= P.n_q) continue;
        const size_t slot = (size_t)item * P.part_stride * 2 + t;
        const float2 a = __ldcg(reinterpret_cast<const float2 *>(P.part_ml) + slot * TILE + r), b = __ldcg(reinterpret_cast<const float2 *>(P.part_ml) + (slot + 2) * TILE + r);
        const float m = fmaxf(a.x, b.x), sc0 = exp2f(a.x - m), sc1 = exp2f(b.x - m), l = fmaf(b.y, sc1, a.y * sc0), inv = 1.f / l;
        const float4 *po = reinterpret_cast<const float4 *>(P.part_o) + slot * (TILE * TILE / 4) + r;
        uint2 *orow = reinterpret_cast<uint2 *>(P.out + ((size_t)row * P.n_q_heads + h) * TILE);
#pragma unroll 4
        for (int c = 0; c < TILE / 4; ++c) {
            const float4 x = __ldcg(po + c * TILE), y = __ldcg(po + TILE * TILE / 2 + c * TILE);
            orow[c] = make_uint2(pc_pack_bf16(fmaf(y.x, sc1, x.x * sc0) * inv, fmaf(y.y, sc1, x.y * sc0) * inv),
                                 pc_pack_bf16(fmaf(y.z, sc1, x.z * sc0) * inv, fmaf(y.w, sc1, x.w * sc0) * inv));
        }
        if (P.lse) P.lse[(size_t)row * P.n_q_heads + h] = (m + log2f(l)) * 0.6931471805599453f;
    }
}

// MERGE: items in two parts are merged by the CTA that has the first one.  A kernel of its own: with what that takes in its code, calls
// that merge nothing took 0.3 us longer.
template <bool MERGE>
__global__ void __launch_bounds__(TC_THREADS, 1)
k_attend_tc(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
            const __grid_constant__ CUtensorMap map_v0, const __grid_constant__ CUtensorMap map_v1,
            const __grid_constant__ CUtensorMap map_v2, const __grid_constant__ TcParams P) {
    pc_grid_dep_launch();
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *gen = smem_raw + (base - smem_u32(smem_raw));
    volatile int *abort_flag = reinterpret_cast<volatile int *>(gen + SM_BAR + N_BARS * 8);
    volatile int *left_here = abort_flag + 1;            // a warp of this CTA left a merge
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(gen + SM_BAR + N_BARS * 8 + 8);
    const uint32_t bar0 = base + SM_BAR;
    auto bar = [&](int i) { return bar0 + 8u * i; };

    // from one lane, so that the compiler knows a warp's number, and with it barrier and tensor-memory addresses and descriptors, to be
    // the same in all lanes and keeps them in uniform registers
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    long long G0, G1;
    cta_run(P, (int)blockIdx.x, G0, G1);           // this CTA's run of steps (never empty: the host sizes the grid so)

    if (threadIdx.x == 0) {
        for (int s = 0; s < KV_STAGES; ++s) {
            mbar_init(bar(BAR_VFULL + s), 1);
            mbar_init(bar(BAR_EMPTY + s), 4);
        }
        for (int t = 0; t < 2; ++t) {
            mbar_init(bar(BAR_Q + t), 1);
            mbar_init(bar(BAR_QFREE + t), 4);
            mbar_init(bar(BAR_SFULL + t), 1);
            mbar_init(bar(BAR_SFREE + t), 4);
            mbar_init(bar(BAR_PVDONE + t), 1);
            mbar_init(bar(BAR_PHALF + 2 * t), 4);
            mbar_init(bar(BAR_PHALF + 2 * t + 1), 4);
        }
        mbar_init(bar(BAR_DONE), 3);
        mbar_init(bar(BAR_PART), 8);
        *abort_flag = 0;
        *left_here = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 2) {   // TMEM: all 512 columns
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    pc_grid_dep_wait();   // barriers and TMEM are set up; from here on the rotated K / Q are read

    // Steps are counted through the whole run (gs): ring stages and barrier phases follow gs, so a unit boundary is an
    // ordinary step for the key / value pipeline.  Both query tiles always run; a unit whose head group has an odd tile
    // count loads its one tile twice and the second copy's result is dropped.
    // registers move from warps 0-3 to warps 4-11
    if (warp == 0) {
        // ---------------------------------------------------------------- TMA producer
        reg_dealloc<REGS_ISSUE>();
        if (lane == 0) {
            // A unit's query tile t arrives on BAR_Q + t once the tile's last QK^T of the unit before has completed (BAR_QFREE + t);
            // the run's first K tile rides with tile 0's first queries.  After that V(step) and K(step + 1) always travel together:
            // they are needed at about the same time and their stages are released together, so one full / empty
            // barrier pair serves both.  K(step + 1) may be the first tile of the next unit.
            bool alive = true;
            int gs = 0, un = 0;
            // The second part of a two-part item is the first unit of its CTA.  Once the softmax warps have stored it (BAR_PART) this thread, which
            // has time to spare, says so to the CTA with the first part: the fence would hold up a softmax warp.
            int first_part = 0, first_parts = 1;
            if constexpr (MERGE) item_parts(P, (int)(G0 / P.n_kv_tiles), (int)blockIdx.x, first_part, first_parts);
            bool owes = MERGE && first_part == 1;
            const auto pass_on = [&]() {
                __threadfence();
                asm volatile("st.release.gpu.u32 [%0], %1;" ::"l"(P.sync + SYNC_PARTS + (int)(G0 / P.n_kv_tiles)), "r"(__ldcg(P.sync)) : "memory");
                owes = false;
            };
            for (long long g = G0; g < G1 && alive; ++un) {
                const Unit U = unit_at(P, g, G1);
                g += U.n_j;
                const int kvh = U.item / P.pairs_per_g, pair = U.item % P.pairs_per_g;
                const int n_tiles_q = min(2, P.tiles_per_g - 2 * pair);
                for (int t = 0; t < 2 && alive; ++t) {
                    if (un > 0) alive = mbar_wait(bar(BAR_QFREE + t), (un - 1) & 1, abort_flag, P.status, PC_WHERE_ATTN_WAIT, P.wait_us);
                    if (!alive) break;
                    const bool first = un == 0 && t == 0;
                    mbar_expect_tx(bar(BAR_Q + t), (first ? 2 : 1) * TILE_BYTES + (first ? P.extra_tx : 0u));
                    const int T = 2 * pair + min(t, n_tiles_q - 1), tb = T / P.group, h = kvh * P.group + T % P.group;
                    tma_load_2d(base + SM_Q + t * TILE_BYTES, &map_q, h * TILE, tb * TILE, bar(BAR_Q + t));
                    tma_load_2d(base + SM_Q + t * TILE_BYTES + HALF_BYTES, &map_q, h * TILE + 64, tb * TILE, bar(BAR_Q + t));
                    if (first) {
                        tma_load_2d(base + SM_K, &map_k, kvh * TILE, U.jb * TILE, bar(BAR_Q));
                        tma_load_2d(base + SM_K + HALF_BYTES, &map_k, kvh * TILE + 64, U.jb * TILE, bar(BAR_Q));
                    }
                }
                if (!alive) break;
                for (int j = 0; j < U.n_j && alive; ++j, ++gs) {
                    const int st = gs % KV_STAGES, kst = (gs + 1) % KV_STAGES;
                    int seg, local, n_valid;
                    kv_tile_info(P, U.jb + j, seg, local, n_valid);
                    const CUtensorMap *mv = seg == 0 ? &map_v0 : (seg == 1 ? &map_v1 : &map_v2);
                    // PV(step - 2) and QK^T(step - 1) have read what lies where V(step) and K(step + 1) go
                    if (gs > 0) alive = mbar_wait(bar(BAR_EMPTY + ((gs - 1) & 1)), ((gs - 1) >> 1) & 1, abort_flag, P.status, PC_WHERE_ATTN_WAIT, P.wait_us);
                    if (!alive) break;
                    const bool in_unit = j + 1 < U.n_j, more = in_unit || g < G1;
                    mbar_expect_tx(bar(BAR_VFULL + st), (more ? 2 : 1) * TILE_BYTES);
                    tma_load_2d(base + SM_V + st * TILE_BYTES, mv, kvh * TILE, local * TILE, bar(BAR_VFULL + st));
                    tma_load_2d(base + SM_V + st * TILE_BYTES + HALF_BYTES, mv, kvh * TILE + 64, local * TILE, bar(BAR_VFULL + st));
                    if (more) {
                        // the next step's keys: the next tile of this item, or the first tile of the next item
                        const int nk = in_unit ? kvh : (U.item + 1) / P.pairs_per_g, nj = in_unit ? U.jb + j + 1 : 0;
                        tma_load_2d(base + SM_K + kst * TILE_BYTES, &map_k, nk * TILE, nj * TILE, bar(BAR_VFULL + st));
                        tma_load_2d(base + SM_K + kst * TILE_BYTES + HALF_BYTES, &map_k, nk * TILE + 64, nj * TILE, bar(BAR_VFULL + st));
                    }
                    if (owes && un > 0 && pc_mbar_test(bar(BAR_PART), 0)) pass_on();
                }
            }
            if (owes && alive && mbar_wait(bar(BAR_PART), 0, abort_flag, P.status, PC_WHERE_ATTN_WAIT, P.wait_us)) pass_on();
        }
    } else if (warp < 4) {
        // ---------------------------------------------------------------- MMA issuers: warps 1 and 2 S = Q_t K^T, warp 3 O += P V
        // A warp stays converged (every lane takes the waits) and only the tcgen05 instructions are predicated on
        // one elected lane: issuing a multiply-add then costs about 12 cycles instead of about 60.
        reg_dealloc<REGS_ISSUE>();
        const bool lead = elect_one();
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
        const int n_steps = (int)(G1 - G0);
        auto wait = [&](int b, int parity) {
            const bool ok = warp_wait(bar(b), parity, abort_flag, P.status, P.wait_us);
            tc_fence_after();
            return ok;
        };
        bool alive = true;
        if (warp < 3) {
            const int t = warp - 1;
            const uint64_t dq0 = desc_kmajor(base + SM_Q + t * TILE_BYTES), dk0 = desc_kmajor(base + SM_K);
            long long g = G0;
            int un = -1, left = 0;                           // this unit, and its steps left
#pragma unroll 1
            for (int gs = 0; gs < n_steps; ++gs) {
                if (left == 0) {
                    left = unit_at(P, g, G1).n_j;
                    g += left;
                    ++un;
                    alive = wait(BAR_Q + t, un & 1);
                    if (!alive) break;
                }
                --left;
                if (gs > 0) alive = wait(BAR_VFULL + (gs - 1) % KV_STAGES, ((gs - 1) / KV_STAGES) & 1);      // K(step) came with V(step - 1)
                if (alive && gs + t > 0) alive = wait(BAR_SFREE + (t ^ 1), (gs + t + 1) & 1);      // the other tile's scores have left the columns
                if (!alive) break;
                uint64_t dq = dq0, dk = dk0 + (gs % KV_STAGES) * (TILE_BYTES >> 4);
#pragma unroll 1
                for (int half = 0; half < 2; ++half) {
#pragma unroll
                    for (int k4 = 0; k4 < 4; ++k4)
                        if (lead) mma_ss(tm + TM_S, dq + k4 * 2, dk + k4 * 2, IDESC_QK, (half > 0 || k4 > 0));
                    dq += HALF_BYTES >> 4;
                    dk += HALF_BYTES >> 4;
                }
                if (lead) tc_commit(bar(BAR_SFULL + t));
            }
        } else {
            const uint64_t dv0 = desc_mnmajor(base + SM_V);
            int at = (int)(G0 % P.n_kv_tiles);               // key tile of the step
#pragma unroll 1
            for (int gs = 0; gs < n_steps && alive; ++gs) {
                const int st = gs % KV_STAGES;
                const bool first = gs == 0 || at == 0;       // of its unit
                alive = wait(BAR_VFULL + st, (gs / KV_STAGES) & 1);
                // the cluster merge stages O_0 where both query tiles lie: tile 1's last QK^T has read them before O_0 is final
                if (P.cluster && gs + 1 == n_steps) alive = alive && wait(BAR_SFULL + 1, gs & 1);
#pragma unroll 1
                for (int t = 0; t < 2 && alive; ++t) {
                    // P arrives in two halves of 64 keys: the first PV steps run while the rest is exponentiated
                    uint64_t dv = dv0 + st * (TILE_BYTES >> 4);
                    uint32_t pa = tm + TM_P + t * (TILE / 2);
                    const uint32_t oa = tm + TM_O + t * TILE;
#pragma unroll 1
                    for (int hf = 0; hf < 2; ++hf) {
                        alive = wait(BAR_PHALF + 2 * t + hf, gs & 1);
                        if (!alive) break;
#pragma unroll
                        for (int k4 = 0; k4 < 4; ++k4)     // 16 keys per step: P columns advance by 8 (two bf16 per column)
                            if (lead) mma_ts(oa, pa + k4 * 8, dv + k4 * (2048 >> 4), IDESC_PV, (!first || hf > 0 || k4 > 0));
                        dv += 8192 >> 4;
                        pa += 32;
                    }
                    if (alive && lead) tc_commit(bar(BAR_PVDONE + t));            // P_t may be overwritten, O_t read
                }
                if (++at == P.n_kv_tiles) at = 0;
            }
        }
        // make sure nothing of ours is still running on the tensor core before TMEM is freed
        if (lead) tc_commit(bar(BAR_DONE));
        __syncwarp();
        pc_mbar_drain(bar(BAR_DONE), 0, P.status, PC_WHERE_ATTN_WAIT);
    } else {
        // ---------------------------------------------------------------- softmax + correction + epilogue
        reg_alloc<REGS_SOFTMAX>();
        const int t = (warp - 4) >> 2;
        const int quad = warp & 3;                       // TMEM lane quadrant this warp may touch
        const int r = quad * 32 + lane;                  // row of the tile
        const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
        const uint32_t s_addr = tmem + lane_addr + TM_S;
        const uint32_t p_addr = tmem + lane_addr + TM_P + t * (TILE / 2);
        const uint32_t o_addr = tmem + lane_addr + TM_O + t * TILE;
        bool alive = true;
        const bool lead = elect_one();
        const int n_steps = (int)(G1 - G0);
        Unit U = unit_at(P, G0, G1);
        long long g = G0 + U.n_j;                        // end of the unit
        float m_used = -INFINITY, l = 0.f;
        int j = 0;
        auto next_end = [&](int jt) {                    // last tile of the segment that tile jt is in
            int seg = 0;
            while (seg + 1 < P.n_seg && jt >= P.seg_tile_end[seg]) ++seg;
            return P.seg_tile_end[seg] - 1;
        };
        int ragged = next_end(U.jb);
        // A unit's output leaves O_t in the turn behind its last step, after the next unit's first probabilities are computed and before they
        // are handed over (the first PV of a unit overwrites O_t): the stores run under the tensor core's next work.  Reading and storing O_t first left the tensor core idle meanwhile: the step at
        // 12 frames 88.1 against 86.4 us, 47 frames 167.4 against 165.5, 4,032-token frames 663.9 against 656.3.  The run's last unit leaves
        // in one more turn, or behind the loop where that may take a merge.  The kernel without merges has its read-out in the loop and written out
        // by itself: behind the loop, or through the functions that the other one uses, calls of a few steps took 0.2 to 0.6 us longer.
        const auto read_out = [&](uint32_t (&v)[128]) {  // the thread's whole O row leaves TMEM in one pass (four loads in flight, one wait)
            tmem_ld32(o_addr, v);
            tmem_ld32(o_addr + 32, v + 32);
            tmem_ld32(o_addr + 64, v + 64);
            tmem_ld32(o_addr + 96, v + 96);
            tmem_wait_ld();
        };
        struct Place { int h, row, part, parts, slot; bool there; };
        const auto place_of = [&](int item) {
            Place p;
            const int kvh = item / P.pairs_per_g, pair = item % P.pairs_per_g, T = 2 * pair + t, tb = T / P.group;
            p.there = t < min(2, P.tiles_per_g - 2 * pair);        // not the second copy of a single query tile, which is dropped
            p.h = kvh * P.group + T % P.group;
            p.row = tb * TILE + r;
            item_parts(P, item, (int)blockIdx.x, p.part, p.parts);
            p.slot = (item * P.part_stride + p.part) * 2 + t;
            return p;
        };
        const auto write_whole = [&](const Place &p, const uint32_t (&v)[128], float m_e, float l_e) {
            const float inv = 1.f / l_e;
            __nv_bfloat16 *orow = P.out + ((size_t)p.row * P.n_q_heads + p.h) * TILE;
            if (p.row < P.n_q) {
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    uint4 w;
                    w.x = pc_pack_bf16(__uint_as_float(v[8 * i + 0]) * inv, __uint_as_float(v[8 * i + 1]) * inv);
                    w.y = pc_pack_bf16(__uint_as_float(v[8 * i + 2]) * inv, __uint_as_float(v[8 * i + 3]) * inv);
                    w.z = pc_pack_bf16(__uint_as_float(v[8 * i + 4]) * inv, __uint_as_float(v[8 * i + 5]) * inv);
                    w.w = pc_pack_bf16(__uint_as_float(v[8 * i + 6]) * inv, __uint_as_float(v[8 * i + 7]) * inv);
                    *reinterpret_cast<uint4 *>(orow + i * 8) = w;
                }
            }
            if (P.lse && p.row < P.n_q) P.lse[(size_t)p.row * P.n_q_heads + p.h] = (m_e + log2f(l_e)) * 0.6931471805599453f;
        };
        // Partial tile layout: 16-byte unit (c4, r) = columns 4*c4..4*c4+3 of row r at unit c4*128 + r, so the 32 rows
        // of a warp store 512 contiguous bytes per instruction (a row-major tile would touch 32 lines per store).
        const auto write_part = [&](const Place &p, const uint32_t (&v)[128], float m_e, float l_e) {
            uint4 *ptile = reinterpret_cast<uint4 *>(P.part_o) + (size_t)p.slot * (TILE * TILE / 4) + r;
#pragma unroll
            for (int i = 0; i < 32; ++i) ptile[i * TILE] = make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            *reinterpret_cast<float2 *>(P.part_ml + ((size_t)p.slot * TILE + r) * 2) = make_float2(m_e, l_e);
        };
        for (int gs = 0; alive && (!MERGE || gs < n_steps); ++gs) {
            const bool end = !MERGE && gs == n_steps, flush = end || j == U.n_j;
            const int e_item = U.item;                   // the unit to flush
            const float m_e = m_used, l_e = l;
            if (flush && !end) {
                U = unit_at(P, g, G1);
                g += U.n_j;
                j = 0;
                m_used = -INFINITY;
                l = 0.f;
                ragged = next_end(0);
            }
            if (!end) {
                alive = warp_wait(bar(BAR_SFULL + t), gs & 1, abort_flag, P.status, P.wait_us);
                if (!alive) break;
                tc_fence_after();
                if (__builtin_expect(U.jb + j == ragged, 0)) {      // last tile of a segment: keys past its end score -inf
                    int seg, local, n_valid;
                    kv_tile_info(P, ragged, seg, local, n_valid);
                    ragged = P.seg_tile_end[min(seg + 1, P.n_seg - 1)] - 1;
                    int i = n_valid;
#pragma unroll 1
                    for (; i & 7; ++i) tmem_st1(s_addr + i, 0xFF800000u);
#pragma unroll 1
                    for (; i < TILE; i += 8) tmem_st8(s_addr + i, 0xFF800000u);
                    tmem_wait_st();
                }
                // the whole score row of this thread: one TMEM pass
                uint32_t sv[128];
                tmem_ld32(s_addr, sv);
                tmem_ld32(s_addr + 32, sv + 32);
                tmem_ld32(s_addr + 64, sv + 64);
                tmem_ld32(s_addr + 96, sv + 96);
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                arrive_if(lead, bar(BAR_SFREE + t));         // the columns are the other tile's
                if (j + 1 == U.n_j) arrive_if(lead, bar(BAR_QFREE + t));      // that was the unit's last QK^T of this tile
                // the PV of the step before: its P columns are written again below, and O_t may be rescaled
                const bool pv_done = gs == 0 || pc_mbar_test(bar(BAR_PVDONE + t), (gs - 1) & 1);
                float mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY, mx3 = -INFINITY;
#pragma unroll
                for (int i = 0; i < TILE; i += 4) {
                    mx0 = fmaxf(mx0, __uint_as_float(sv[i]));
                    mx1 = fmaxf(mx1, __uint_as_float(sv[i + 1]));
                    mx2 = fmaxf(mx2, __uint_as_float(sv[i + 2]));
                    mx3 = fmaxf(mx3, __uint_as_float(sv[i + 3]));
                }
                const float mx = fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3));
                // lazy rescale: move the reference maximum only when it grew by more than the threshold
                const bool grow = mx > m_used + RESCALE_THRESHOLD;
                if (__builtin_expect(!__all_sync(0xffffffffu, pv_done), 0)) {
                    alive = warp_wait(bar(BAR_PVDONE + t), (gs - 1) & 1, abort_flag, P.status, P.wait_us);
                    if (!alive) break;
                }
                tc_fence_after();
                // tile 1 comes last: QK^T(step) and PV(step - 1) have read their keys and values
                if (t == 1) arrive_if(lead, bar(BAR_EMPTY + (gs & 1)));
                if (__builtin_expect(__any_sync(0xffffffffu, grow), 0)) {
                    const float m_new = fmaxf(m_used, mx);
                    const float corr = fast_exp2(m_used - m_new);       // 0 on the first tile (m_used = -inf)
                    l *= corr;
                    if (j > 0) {
                        uint32_t v[32];
#pragma unroll 1
                        for (int c = 0; c < 4; ++c) {
                            tmem_ld32(o_addr + c * 32, v);
                            tmem_wait_ld();
#pragma unroll
                            for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * corr);
                            tmem_st32(o_addr + c * 32, v);
                        }
                    }
                    m_used = m_new;
                }
                // p = 2^(s - m) as bf16 pairs; the row sum runs on two-lane adds
                const float2 neg_m = make_float2(-m_used, -m_used);
                float2 la = make_float2(0.f, 0.f), lb = make_float2(0.f, 0.f);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    uint32_t pk[16];
#pragma unroll
                    for (int i = 0; i < 16; i += 2) {
                        float2 x = add2(make_float2(__uint_as_float(sv[c * 32 + 2 * i]), __uint_as_float(sv[c * 32 + 2 * i + 1])), neg_m);
                        float2 y = add2(make_float2(__uint_as_float(sv[c * 32 + 2 * i + 2]), __uint_as_float(sv[c * 32 + 2 * i + 3])), neg_m);
                        x.x = fast_exp2(x.x); x.y = fast_exp2(x.y);
                        y.x = fast_exp2(y.x); y.y = fast_exp2(y.y);
                        la = add2(la, x);
                        lb = add2(lb, y);
                        pk[i] = pc_pack_bf16(x.x, x.y);
                        pk[i + 1] = pc_pack_bf16(y.x, y.y);
                    }
                    // the sums belong in the gaps of this chunk's exponentials, not behind the hand-over
                    asm volatile("" : "+f"(la.x), "+f"(la.y), "+f"(lb.x), "+f"(lb.y));
                    tmem_st16(p_addr + c * 16, pk);
                    if (c & 1) {                               // keys 0-63, then 64-127, handed to the tensor core
                        tmem_wait_st();
                        tc_fence_before();
                        __syncwarp();
                        arrive_if(lead && !flush, bar(BAR_PHALF + 2 * t + (c >> 1)));
                    }
                }
                l += (la.x + la.y) + (lb.x + lb.y);
            }
            if (end) {
                alive = warp_wait(bar(BAR_PVDONE + t), (gs - 1) & 1, abort_flag, P.status, P.wait_us);
                if (!alive) break;
                tc_fence_after();
            }
            if (__builtin_expect(flush, 0)) {
                if constexpr (MERGE) {
                    uint32_t v[128];
                    read_out(v);
                    tc_fence_before();
                    __syncwarp();
                    arrive_if(lead, bar(BAR_PHALF + 2 * t));
                    arrive_if(lead, bar(BAR_PHALF + 2 * t + 1));
                    const Place p = place_of(e_item);
                    if (p.there) {
                        if (p.parts == 1) write_whole(p, v, m_e, l_e);
                        else write_part(p, v, m_e, l_e);
                    }
                    if (p.part == 1) {
                        __syncwarp();
                        arrive_if(lead, bar(BAR_PART));
                    }
                } else {
                    // the thread's whole O row leaves TMEM in one pass (four loads in flight, one wait)
                    uint32_t v[128];
                    tmem_ld32(o_addr, v);
                    tmem_ld32(o_addr + 32, v + 32);
                    tmem_ld32(o_addr + 64, v + 64);
                    tmem_ld32(o_addr + 96, v + 96);
                    tmem_wait_ld();
                    if (!end) {
                        tc_fence_before();
                        __syncwarp();
                        arrive_if(lead, bar(BAR_PHALF + 2 * t));
                        arrive_if(lead, bar(BAR_PHALF + 2 * t + 1));
                    }
                    const int kvh = e_item / P.pairs_per_g, pair = e_item % P.pairs_per_g;
                    const int n_tiles_q = min(2, P.tiles_per_g - 2 * pair);
                    int part, parts;
                    item_parts(P, e_item, (int)blockIdx.x, part, parts);
                    const int T = 2 * pair + t, tb = T / P.group, h = kvh * P.group + T % P.group;
                    const int row = tb * TILE + r;
                    if (t >= n_tiles_q) {
                        // the second copy of a single query tile: dropped
                    } else if (parts == 1) {
                        const float inv = 1.f / l_e;
                        __nv_bfloat16 *orow = P.out + ((size_t)row * P.n_q_heads + h) * TILE;
                        if (row < P.n_q) {
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                uint4 w;
                                w.x = pc_pack_bf16(__uint_as_float(v[8 * i + 0]) * inv, __uint_as_float(v[8 * i + 1]) * inv);
                                w.y = pc_pack_bf16(__uint_as_float(v[8 * i + 2]) * inv, __uint_as_float(v[8 * i + 3]) * inv);
                                w.z = pc_pack_bf16(__uint_as_float(v[8 * i + 4]) * inv, __uint_as_float(v[8 * i + 5]) * inv);
                                w.w = pc_pack_bf16(__uint_as_float(v[8 * i + 6]) * inv, __uint_as_float(v[8 * i + 7]) * inv);
                                *reinterpret_cast<uint4 *>(orow + i * 8) = w;
                            }
                        }
                        if (P.lse && row < P.n_q) P.lse[(size_t)row * P.n_q_heads + h] = (m_e + log2f(l_e)) * 0.6931471805599453f;
                    } else if (P.cluster) {
                        // (split form, one unit per CTA) Stage O (un-normalised, fp32) and (max, sum) in shared memory that no
                        // multiply-add reads any more: tile 0 over both query tiles (every QK^T has completed once this tile's
                        // last PV has, which was issued behind the other tile's last QK^T), tile 1 over the key stages (its own last PV is the last multiply-add of the CTA).
                        const uint32_t stage = base + (t == 0 ? SM_Q : SM_K);
#pragma unroll
                        for (int i = 0; i < 32; ++i) sts128(stage + stage_off(i, r), v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                        *reinterpret_cast<float2 *>(gen + SM_ML + (t * TILE + r) * 8) = make_float2(m_e, l_e);
                    } else {
                        // Partial tile layout: 16-byte unit (c4, r) = columns 4*c4..4*c4+3 of row r at unit c4*128 + r, so the 32 rows
                        // of a warp store 512 contiguous bytes per instruction (a row-major tile would touch 32 lines per store).
                        const size_t tile_slot = ((size_t)e_item * P.part_stride + part) * 2 + t;
                        uint4 *ptile = reinterpret_cast<uint4 *>(P.part_o) + tile_slot * (TILE * TILE / 4) + r;
#pragma unroll
                        for (int i = 0; i < 32; ++i) ptile[i * TILE] = make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                        *reinterpret_cast<float2 *>(P.part_ml + (tile_slot * TILE + r) * 2) = make_float2(m_e, l_e);
                    }
                }
            }
            if (end) break;
            ++j;
        }
        // ---- the run's last unit.  If it is the first part of an item in two parts, the second one lies in the scratch, stored by the same warp of the
        // next CTA at the start of its run: it is fetched under the last PV and added here, in the order of the
        // merge kernel and with its arithmetic.  That CTA may not have had an SM yet (somebody else's kernel holds it), and this one's SM may be what it is waiting
        // for, so a part that does not come is no error: the first one is stored as well, and the last CTA merges them.
        if constexpr (MERGE) {
            const Place p = place_of(U.item);
            const bool head = p.parts == 2 && p.part == 0 && p.there;
            bool merge = false;
            uint4 x[32];
            float2 ml = make_float2(-INFINITY, 0.f);
            if (__builtin_expect(head && alive && !P.leave_parts, 0)) {
                const uint32_t *flag = P.sync + SYNC_PARTS + U.item;
                const uint32_t call = __ldcg(P.sync);
                const uint64_t t0 = pc_global_ns();
                for (;;) {
                    uint32_t seen;
                    asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(seen) : "l"(flag) : "memory");
                    merge = __all_sync(0xffffffffu, seen == call);
                    if (merge || __any_sync(0xffffffffu, *abort_flag || pc_global_ns() - t0 > PART_NS)) break;
                }
                if (merge) {
                    const size_t slot = p.slot + 2;
                    const uint4 *ptile = reinterpret_cast<const uint4 *>(P.part_o) + slot * (TILE * TILE / 4) + r;
                    ml = __ldcg(reinterpret_cast<const float2 *>(P.part_ml) + slot * TILE + r);
#pragma unroll
                    for (int i = 0; i < 32; ++i) x[i] = __ldcg(ptile + i * TILE);
                }
            }
            if (alive) alive = warp_wait(bar(BAR_PVDONE + t), (n_steps - 1) & 1, abort_flag, P.status, P.wait_us);
            if (alive) {
                tc_fence_after();
                if (!merge) {
                    uint32_t v[128];
                    read_out(v);
                    if (p.there) {
                        if (p.parts == 1) write_whole(p, v, m_used, l); else write_part(p, v, m_used, l);
                    }
                    if (p.part == 1) {
                        __syncwarp();
                        arrive_if(lead, bar(BAR_PART));
                    } else if (head && lead) {
                        P.sync[SYNC_PARTS + P.n_items + U.item * LEFT_PER_ITEM + t * 4 + quad] = __ldcg(P.sync);
                        *left_here = 1;
                    }
                } else {
                    // Rows leave through shared memory, over the queries of this tile (its last QK^T has been seen): a warp's store then covers two whole rows
                    // of 256 bytes instead of 16 bytes of each of 32.  16-byte unit c of row r at r * 256 + (c ^ (r & 15)) * 16: no bank twice.
                    const float m = fmaxf(m_used, ml.x), sc0 = exp2f(m_used - m), sc1 = exp2f(ml.x - m);
                    const float lsum = fmaf(ml.y, sc1, l * sc0), inv = 1.f / lsum;
                    const uint32_t stage = base + SM_Q + t * TILE_BYTES + quad * (32 * 256);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        uint32_t v[32];
                        tmem_ld32(o_addr + c * 32, v);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const uint4 y = x[8 * c + i];
                            v[4 * i + 0] = __float_as_uint(fmaf(__uint_as_float(y.x), sc1, __uint_as_float(v[4 * i + 0]) * sc0));
                            v[4 * i + 1] = __float_as_uint(fmaf(__uint_as_float(y.y), sc1, __uint_as_float(v[4 * i + 1]) * sc0));
                            v[4 * i + 2] = __float_as_uint(fmaf(__uint_as_float(y.z), sc1, __uint_as_float(v[4 * i + 2]) * sc0));
                            v[4 * i + 3] = __float_as_uint(fmaf(__uint_as_float(y.w), sc1, __uint_as_float(v[4 * i + 3]) * sc0));
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            uint32_t w[4];
#pragma unroll
                            for (int k = 0; k < 4; ++k) w[k] = pc_pack_bf16(__uint_as_float(v[8 * i + 2 * k]) * inv, __uint_as_float(v[8 * i + 2 * k + 1]) * inv);
                            sts128(stage + lane * 256 + (((4 * c + i) ^ (lane & 15)) << 4), w[0], w[1], w[2], w[3]);
                        }
                    }
                    __syncwarp();
                    const int row0 = p.row - lane;
#pragma unroll 4
                    for (int i = 0; i < 16; ++i) {
                        const int rr = 2 * i + (lane >> 4), c = lane & 15;
                        const uint4 w = pc_lds128(stage + rr * 256 + ((c ^ (rr & 15)) << 4));
                        if (row0 + rr < P.n_q) *reinterpret_cast<uint4 *>(P.out + ((size_t)(row0 + rr) * P.n_q_heads + p.h) * TILE + c * 8) = w;
                    }
                    if (P.lse && p.row < P.n_q) P.lse[(size_t)p.row * P.n_q_heads + p.h] = (m + log2f(lsum)) * 0.6931471805599453f;
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
    // every thread has done with its waits: the flag is final, and copies may be in flight that nobody waited for
    if (threadIdx.x == 0 && *abort_flag) pc_let_copies_land();
    if constexpr (MERGE) {
        // The last CTA to come here moves the call's number on: what this call left in the flags means nothing to the next one, also if
        // some of it was given up, and a captured call replays unchanged.  It also merges what was left: every part of the call is
        // stored and fenced ahead of its CTA's ticket (a second part by pass_on, which this thread ran).
        // That something was left travels with the ticket: a look behind it (a fence and a load) made every call 1.2 us longer.
        volatile uint32_t *last = reinterpret_cast<volatile uint32_t *>(gen + SM_BAR + N_BARS * 8 + 4);   // (left_here and tmem_slot, read already) anything left, number of the call
        if (threadIdx.x == 0) {
            const uint32_t mine = *left_here ? 0x10000u : 0u;
            uint32_t left = 0;
            if (mine) __threadfence();
            const uint32_t ticket = atomicAdd(P.sync + 1, 1u + mine);
            if ((ticket & 0xFFFFu) == (uint32_t)gridDim.x - 1) {
                left = (ticket >> 16) + mine;
                if (left) {
                    __threadfence();
                    last[1] = __ldcg(P.sync);
                }
                P.sync[1] = 0;
                atomicAdd(P.sync, 1u);
            }
            last[0] = left;
        }
        __syncthreads();
        if (__builtin_expect(last[0] != 0 && warp >= 4, 0)) merge_left(P, last[1], warp - 4, lane);
    }
    if (!MERGE && P.cluster && P.n_splits > 1) {
        // Merge the KV ranges of this item across the cluster: CTA `rank` finishes every n_splits-th row of the two
        // tiles, reading each peer's staged O and (max, sum) through distributed shared memory.  Sixteen threads share
        // a row (two 16-byte units each), so a row's 256 output bytes leave as two 128-byte runs.
        const int item = (int)blockIdx.x / P.n_splits;
        const int kvh = item / P.pairs_per_g, pair = item % P.pairs_per_g;
        const int n_tiles_q = min(2, P.tiles_per_g - 2 * pair);
        cluster_sync_all();                        // every CTA's staging is complete and visible
        if (warp >= 4) {
            const int S = P.n_splits, my = (int)cluster_rank();
            const int id = threadIdx.x - 128, sub = id & 15, slot = id >> 4;
            uint32_t peer_base[MAX_SPLITS];
#pragma unroll
            for (int k = 0; k < MAX_SPLITS; ++k) peer_base[k] = peer_addr(base, k < S ? k : 0);
            for (int R = my + slot * S; R < 2 * TILE; R += 16 * S) {
                const int t = R >> 7, r = R & (TILE - 1);
                if (t >= n_tiles_q) break;
                const int T = 2 * pair + t, tb = T / P.group, h = kvh * P.group + T % P.group;
                const int row = tb * TILE + r;
                if (row >= P.n_q) continue;
                float mk[MAX_SPLITS], lk[MAX_SPLITS], m = -INFINITY;
#pragma unroll
                for (int k = 0; k < MAX_SPLITS; ++k)
                    if (k < S) {
                        const float2 ml = peer_ld64(peer_base[k] + SM_ML + (t * TILE + r) * 8);
                        mk[k] = ml.x; lk[k] = ml.y;
                        m = fmaxf(m, ml.x);
                    }
                float lsum = 0.f;
                float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
                const uint32_t stage = (t == 0 ? SM_Q : SM_K);
#pragma unroll
                for (int k = 0; k < MAX_SPLITS; ++k)
                    if (k < S) {
                        const float sc = exp2f(mk[k] - m);
                        lsum = fmaf(lk[k], sc, lsum);
                        const float4 x = peer_ld128(peer_base[k] + stage + stage_off(sub, r));
                        const float4 y = peer_ld128(peer_base[k] + stage + stage_off(sub + 16, r));
                        a.x = fmaf(x.x, sc, a.x); a.y = fmaf(x.y, sc, a.y); a.z = fmaf(x.z, sc, a.z); a.w = fmaf(x.w, sc, a.w);
                        b.x = fmaf(y.x, sc, b.x); b.y = fmaf(y.y, sc, b.y); b.z = fmaf(y.z, sc, b.z); b.w = fmaf(y.w, sc, b.w);
                    }
                const float inv = 1.f / lsum;
                __nv_bfloat16 *orow = P.out + ((size_t)row * P.n_q_heads + h) * TILE;
                *reinterpret_cast<uint2 *>(orow + 4 * sub) = make_uint2(pc_pack_bf16(a.x * inv, a.y * inv), pc_pack_bf16(a.z * inv, a.w * inv));
                *reinterpret_cast<uint2 *>(orow + 64 + 4 * sub) = make_uint2(pc_pack_bf16(b.x * inv, b.y * inv), pc_pack_bf16(b.z * inv, b.w * inv));
                if (P.lse && sub == 0) P.lse[(size_t)row * P.n_q_heads + h] = (m + log2f(lsum)) * 0.6931471805599453f;
            }
        }
        cluster_sync_all();                        // nobody leaves while a peer may still read its shared memory
    }
}

// ------------------------------------------------------------------------------------------------ combine
// Merge of the KV ranges' partials.  One block per (query tile of one head, 32-row quadrant); its eight warps take four
// 16-byte column units each, lanes are consecutive rows, so every load of the partial tiles is a 512-byte run.  Up to four
// parts' loads of a thread are issued before any is used.  Bound by L2 and its latency, so loads in flight count: for items in
// two parts (which the attention kernel leaves to this one where they end together) the kernel is built with 48 registers instead of 108 and four
// blocks an SM instead of two.  The step at 12 frames 80.6 -> 79.1 us, 47 frames 147.0 -> 145.4; six blocks an SM 79.9 and 146.0.
template <int PARTS /* most parts of an item */, int BLOCKS /* resident on an SM */>
__global__ void __launch_bounds__(256, BLOCKS) k_combine(const TcParams P) {
    pc_grid_dep_launch();
    const int lane = threadIdx.x & 31, cg = threadIdx.x >> 5;                   // cg: units 4*cg .. 4*cg+3
    const int quad = blockIdx.x & 3, tile = blockIdx.x >> 2;
    const int h = tile % P.n_q_heads, tb = tile / P.n_q_heads;
    const int g = h / P.group, T = tb * P.group + h % P.group;
    const int item = g * P.pairs_per_g + (T >> 1), t = T & 1;
    const int r = quad * 32 + lane, row = tb * TILE + r;
    if (row >= P.n_q) return;
    int part0, n_parts;
    item_parts(P, item, 0, part0, n_parts);
    pc_grid_dep_wait();                           // the divisions above run under the attention kernel's tail
    if (n_parts < 2) return;                      // the one CTA that had the whole item wrote its output itself
    constexpr int WAY = PARTS < 4 ? PARTS : 4;      // parts in flight
    float2 ml[PARTS];
    float4 o[WAY][4];
    const float2 *pml = reinterpret_cast<const float2 *>(P.part_ml);
    const float4 *po = reinterpret_cast<const float4 *>(P.part_o);
    auto load4 = [&](int s0) {                     // the O units of parts s0 .. s0 + 3
#pragma unroll
        for (int s = 0; s < WAY; ++s)
            if (s0 + s < n_parts) {
                const float4 *pt = po + (((size_t)item * P.part_stride + s0 + s) * 2 + t) * (TILE * TILE / 4) + r;
#pragma unroll
                for (int u = 0; u < 4; ++u) o[s][u] = __ldcg(pt + (cg * 4 + u) * TILE);
            }
    };
#pragma unroll
    for (int s = 0; s < PARTS; ++s)
        if (s < n_parts) ml[s] = __ldcg(pml + (((size_t)item * P.part_stride + s) * 2 + t) * TILE + r);
    load4(0);
    float m = -INFINITY;
#pragma unroll
    for (int s = 0; s < PARTS; ++s)
        if (s < n_parts) m = fmaxf(m, ml[s].x);
    float l = 0.f;
    float4 acc[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int s = 0; s < PARTS; ++s) {
        if (PARTS > 4 && s == 4 && n_parts > 4) load4(4);
        if (s < n_parts) {
            const float sc = exp2f(ml[s].x - m);
            l = fmaf(ml[s].y, sc, l);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                acc[u].x = fmaf(o[s % WAY][u].x, sc, acc[u].x); acc[u].y = fmaf(o[s % WAY][u].y, sc, acc[u].y);
                acc[u].z = fmaf(o[s % WAY][u].z, sc, acc[u].z); acc[u].w = fmaf(o[s % WAY][u].w, sc, acc[u].w);
            }
        }
    }
    const float inv = 1.f / l;
    // this thread's 16 columns of its row: 32 contiguous bytes
    uint4 w0, w1;
    w0.x = pc_pack_bf16(acc[0].x * inv, acc[0].y * inv); w0.y = pc_pack_bf16(acc[0].z * inv, acc[0].w * inv);
    w0.z = pc_pack_bf16(acc[1].x * inv, acc[1].y * inv); w0.w = pc_pack_bf16(acc[1].z * inv, acc[1].w * inv);
    w1.x = pc_pack_bf16(acc[2].x * inv, acc[2].y * inv); w1.y = pc_pack_bf16(acc[2].z * inv, acc[2].w * inv);
    w1.z = pc_pack_bf16(acc[3].x * inv, acc[3].y * inv); w1.w = pc_pack_bf16(acc[3].z * inv, acc[3].w * inv);
    uint4 *orow = reinterpret_cast<uint4 *>(P.out + ((size_t)row * P.n_q_heads + h) * TILE + cg * 16);
    orow[0] = w0;
    orow[1] = w1;
    if (P.lse && cg == 0) P.lse[(size_t)row * P.n_q_heads + h] = (m + log2f(l)) * 0.6931471805599453f;
}

// ------------------------------------------------------------------------------------------------ host side
int div_up(int a, int b) { return (a + b - 1) / b; }

// number of KV ranges of the cluster merge: fewest waves of CTAs, a fixed cost per CTA standing in for prologue and epilogue
int choose_splits(int n_items, int n_kv_tiles, int sm_count) {
    int best = 1;
    long best_cost = -1;
    for (int s = 1; s <= MAX_FIXED_SPLITS && s <= n_kv_tiles; ++s) {
        const long waves = div_up(n_items * s, sm_count);
        const long cost = waves * (div_up(n_kv_tiles, s) + 3) + (s > 1 ? 2 : 0);
        if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = s; }
    }
    return best;
}

// Number of persistent CTAs.  CTAs that start at the same place inside their items run through the same key tiles at the
// same time: of n CTAs over `items` equal items there are n / gcd(n, items) different starting places, and every one of
// them is a stream of K and V of its own through L2.  With a cache larger than L2 the many streams of one CTA per SM read
// everything again for each item (47 whole frames, 96 items on 148 SMs: 37 streams per KV head, 2.36 GB from DRAM for
// 203 MB of K and V); 144 CTAs have three, and their runs are two thirds of an item, so no item is cut into more than two
// parts.  So up to 1/32 of the SMs is given up for the fewest starting places, as long as the longest run grows by no more
// than that (a run counts whole steps), where that makes streams that CTAs share: at least two CTAs of a KV head to a starting place,
// and runs so much shorter than an item (items fewer than 3/4 of the CTAs) that neighbours stay in step.  Measured, one CTA per SM
// against this rule: attention over 47 whole frames 677 -> 571 us a call, five passes over 7,184 keys 461 -> 452, the step at 47
// frames 151.0 -> 149.7, at 12 79.5 -> 77.9.  With the loop before this one (probabilities over the scores): 144 CTAs without the two
// conditions, against 148 (rotated keys, sides in turn): 16 / 16 heads, 1,008 queries x 30,000 keys (9 places, 9 CTAs a head)
// 232 -> 243 us, 32 / 8, 1,008 x 30,000 (128 items) 464 -> 471, 64 / 8, 1,008 x 30,000 (256) 976 -> 999, 24 / 8, 2,000 x 30,000
// (192) 691 -> 702, 24 / 8, 4,032 x 7,184 (384) 326 -> 330; where they hold: 8 / 8, 1,008 x 48,000 (32) 189 -> 178, 24 / 12,
// 1,008 x 30,000 (96) 352 -> 327, 24 / 8, 400 x 30,000 (48) 157 -> 156.
int choose_ctas(int n_items, int n_kv_heads, long long steps, int most) {
    if (4 * n_items >= 3 * most) return most;
    int best = most, best_starts = most / std::gcd(most, n_items);
    const long long longest = (steps + most - 1) / most;
    for (int n = most - 1; n >= most - most / 32; --n) {
        const int starts = n / std::gcd(n, n_items);
        if (starts < best_starts && 2 * starts * n_kv_heads <= n && 32 * ((steps + n - 1) / n) <= 33 * longest) {
            best = n;
            best_starts = starts;
        }
    }
    return best;
}

// Divides the line of (item, key tile) steps over CTAs: fills P.persistent, n_cta, n_splits, part_stride.
//
// What a division costs, in quarters of a step (a step is about 1.4 us): its longest run (boundaries reckoned in, or 16 for
// them where runs are too short or too long for that), 8 for a merge (in the attention kernel as well, where it takes less).  The persistent form takes an even share of the line per CTA; the
// split form cuts every item into s equal ranges, one CTA each, as long as all are resident at once: no boundary, and with one
// range no merge.  Measured on rotated keys (query rotation + attention + merge), the persistent form against the one chosen
// here: 16 / 4 heads, 556 queries x 1,549 keys 29.1 -> 21.9 us, 74 x 4,767 20.9 -> 18.4; 24 / 8, 300 x 305 17.8 -> 17.2 (two ranges,
// which 7 for a merge took, 18.7), 355 x 2,818 27.5 -> 26.4; 32 / 8, 237 x 1,040 20.3 -> 18.8, 1,040 x 3,629 75.1 -> 65.2; 32 / 16,
// 500 x 2,000 29.1 -> 28.1.  Over 274 calls of 20 to 2,500 queries and 100 to 14,000 keys (10 to 260 us) the choice takes 2.0 % more
// than the best form of each, in the geometric mean; most where the reckoning is level, more than four parts are merged and the
// persistent form stands: 32 / 8, 48 x 1,033 17.2 against 14.7 in five ranges.  (Merging the ranges of an item in a cluster instead:
// 24 / 8, 135 x 472 in three 24.1 against 15.9, 1,008 x 9,200 in two 143 against 133.)
void choose_division(const pc_ctx *ctx, int n_items, int tiles, TcParams &P) {
    const long long T = (long long)n_items * tiles;
    P.persistent = 0;
    if (ctx->kv_splits > 0 || ctx->cluster_merge) {
        P.n_splits = ctx->kv_splits > 0 ? std::min(ctx->kv_splits, tiles) : choose_splits(n_items, tiles, ctx->sm_count);
    } else {
        const int n = choose_ctas(n_items, ctx->desc.n_kv_heads, T, (int)std::min<long long>(std::min<long long>(ctx->sm_count, (long long)n_items * (MAX_SPLITS - 1)), T));
        const bool crossing = n % n_items != 0;
        P.n_cta = n;
        // Shorter runs than six times the boundary could end up empty; in longer ones than 64 steps it shows little.
        // Boundaries reckoned in against an even share of the steps, a pass: 4,160 keys (runs of 22) 56.8 -> 54.6 us, 7,184 (38) 88.7 ->
        // 85.6, 9,200 (48) 108.1 -> 105.7; in runs of 75 to 127 166.2 -> 165.0, 187.3 -> 181.4, 266.0 -> 263.0, of 131 to 343 within
        // 1 % either way but for 721.9 -> 736.3 (305), and 154.4 -> 157.8 (69, 71 key tiles an item).
        P.gap = crossing && T >= 6LL * BOUNDARY_STEPS * n && T <= 64LL * n ? BOUNDARY_STEPS : 0;
        int most = 1;
        for (int i = 0; i < n_items / std::gcd(n, n_items); ++i)        // the cuts repeat
            most = std::max(most, cta_of_step(P, i, tiles - 1) - cta_of_step(P, i, 0) + 1);
        long long best = 4 * ((line_length(P) + n - 1) / n) + (crossing && P.gap == 0 ? 16 : 0) + (most > 1 ? 8 : 0);
        P.persistent = 1;
        P.n_splits = P.part_stride = most;
        for (int s = 1; s <= MAX_SPLITS && s <= tiles && n_items * s <= ctx->sm_count; ++s) {
            const long long cost = 4 * div_up(tiles, s) + (s > 1 ? 8 : 0);
            if (cost < best) {
                best = cost;
                P.persistent = 0;
                P.n_splits = s;
            }
        }
        if (P.persistent) return;
    }
    P.n_cta = n_items * P.n_splits;
    P.part_stride = P.n_splits;
}

}  // namespace

pc_status pc_attend_tc_scratch(const pc_layer_desc *d, int sm_count, size_t *k_rot_rows, size_t *part_o_floats,
                               size_t *part_ml_floats, size_t *part_sync_words) {
    // every segment starts on a tile boundary; the query rows follow the keys in the same scratch
    *k_rot_rows = (size_t)(div_up(d->max_keys, TILE) + PC_MAX_SEGMENTS) * TILE;
    const int group = d->n_q_heads / d->n_kv_heads;
    const int n_items = d->n_kv_heads * div_up(group * div_up(d->max_q, TILE), 2);
    // slots: a fixed number of ranges per item, or the parts of the persistent form (every CTA and every item boundary makes
    // one at most, and an item has room for its longest row of them)
    const size_t slots = std::max((size_t)n_items * MAX_FIXED_SPLITS, (size_t)sm_count + 2 * (size_t)n_items);
    *part_o_floats = slots * 2 * TILE * TILE;
    *part_ml_floats = slots * 2 * TILE * 2;
    *part_sync_words = SYNC_PARTS + (size_t)n_items * (1 + LEFT_PER_ITEM);
    return PC_OK;
}

// A part has enough row tiles for a CTA on (nearly) every SM: an item is cut into at most MAX_SPLITS parts, so fewer items
// would leave SMs idle.  At most four parts: each costs a launch, a prologue and an epilogue of its own.
int pc_attend_part_rows(const pc_ctx *ctx, int n_q) {
    const int tiles = div_up(n_q, TILE);
    int least = 1;
    while (least < tiles && ctx->desc.n_kv_heads * div_up(ctx->group * least, 2) * (MAX_SPLITS - 1) < ctx->sm_count - ctx->sm_count / 32) ++least;
    const int parts = std::max(1, std::min(4, tiles / least));
    return div_up(tiles, parts) * TILE;
}

// what: PC_TC_ROPE_K rotates the segments' keys into the context scratch, PC_TC_ROPE_Q rotates the queries,
// PC_TC_ATTEND runs attention (and the merge) on the rotated data.
pc_status pc_launch_attend_tc(pc_ctx *ctx, int n_seg, const pc_segment *segs, const void *q, const int32_t *q_pos,
                              int32_t n_q, void *out, float *lse, cudaStream_t stream, int what, int q_row0) {
    const pc_layer_desc &D = ctx->desc;
    if (D.head_dim != TILE || D.dtype != PC_BF16) return PC_ERR_UNSUPPORTED;
    const int row_elems = D.n_kv_heads * D.head_dim;
    __nv_bfloat16 *k_rot = static_cast<__nv_bfloat16 *>(ctx->k_rot);

    TcParams P{};
    RopeJobs jobs{};
    const int k_chunks = row_elems / 8, q_chunks = D.n_q_heads * D.head_dim / 8;
    if (k_chunks % 32 || q_chunks % 32) return PC_ERR_UNSUPPORTED;
    // chunks per lane: the widest of these that key rows (and with them query rows) are a multiple of; rows have at most 16
    const int k_cpl = k_chunks / 32;
    int cpl = 1;
    for (int m : {2, 13, 11, 7, 5, 3, 4})
        if (k_cpl % m == 0) cpl = m;
    int tiles = 0, warps = 0, n_jobs = 0;
    const auto add_job = [&](const void *src, const int32_t *pos, __nv_bfloat16 *dst, int rows, int chunks, float scale) {
        const int slices = chunks / 32 / cpl;
        jobs.job[n_jobs++] = RopeJob{static_cast<const __nv_bfloat16 *>(src), pos, dst, warps, slices, scale};
        warps += rows * slices;
    };
    for (int s = 0; s < n_seg; ++s) {
        if ((what & PC_TC_ROPE_K) || (s == 0 && (what & PC_TC_ROPE_K0)))
            add_job(segs[s].k, segs[s].pos, k_rot + (size_t)tiles * TILE * row_elems, segs[s].n_tokens, k_chunks, 1.0f);
        tiles += div_up(segs[s].n_tokens, TILE);
        P.seg_tile_end[s] = tiles;
        P.seg_n[s] = segs[s].n_tokens;
    }
    if ((size_t)tiles * TILE > ctx->k_rot_rows) return PC_ERR_CAPACITY;
    __nv_bfloat16 *q_rot = static_cast<__nv_bfloat16 *>(ctx->q_rot);
    if (what & PC_TC_ROPE_Q) add_job(q, q_pos, q_rot, n_q, q_chunks, pc_q_rot_scale(D.head_dim));
    jobs.n_jobs = n_jobs;
    jobs.total_warps = warps;
    if (!(what & PC_TC_GOES_ON)) {
        ctx->ev_mask &= ~((1u << PC_MARK_ATT0) | (1u << PC_MARK_ROPE) | (1u << PC_MARK_ATTEND) | (1u << PC_MARK_COMBINE));
        pc_mark(ctx, PC_MARK_ATT0, stream);
    }
    if (n_jobs > 0) {
#define PC_ROPE_CASE(CPL)                                                                                              \
    case CPL: PC_LAUNCH(k_rope_rows<CPL>, dim3(div_up(warps, 8)), dim3(256), 0, stream, jobs, ctx->rope, D.head_dim, ctx->status); break;
        switch (cpl) {
            PC_ROPE_CASE(1) PC_ROPE_CASE(2) PC_ROPE_CASE(3) PC_ROPE_CASE(4) PC_ROPE_CASE(5) PC_ROPE_CASE(7) PC_ROPE_CASE(11) PC_ROPE_CASE(13)
        }
#undef PC_ROPE_CASE
        PC_CUDA_TRY(cudaGetLastError());
        pc_mark(ctx, PC_MARK_ROPE, stream);          // no pre-pass (a fused frame step with cached anchors): no mark
    }
    if (!(what & PC_TC_ATTEND)) return PC_OK;

    P.n_q = n_q;
    P.n_q_heads = D.n_q_heads;
    P.group = ctx->group;
    P.n_tb = div_up(n_q, TILE);
    P.tiles_per_g = P.group * P.n_tb;
    P.pairs_per_g = div_up(P.tiles_per_g, 2);
    P.n_kv_tiles = tiles;
    P.n_seg = n_seg;
    const int n_items = D.n_kv_heads * P.pairs_per_g;
    P.n_items = n_items;
    P.out = static_cast<__nv_bfloat16 *>(out);
    P.lse = lse;
    P.part_o = ctx->part_o;
    P.part_ml = ctx->part_ml;
    P.status = ctx->status;
    P.wait_us = ctx->wait_limit_us;
    P.extra_tx = ctx->test_extra_tx;
    choose_division(ctx, n_items, tiles, P);
    P.cluster = (!P.persistent && P.n_splits > 1 && ctx->cluster_merge) ? 1 : 0;
    // Merged in the kernel: items in two parts where runs cross items.  The second part of an item is then the first unit of its CTA and lies there long
    // before it is asked for, or it is that CTA's whole run and ends a step or two ahead of the first (three CTAs to two items, as 96 items on 144 CTAs:
    // every second item); both kinds together still gain (96 items: the step at 12 frames 75.5 -> 74.5 us).  Where all pairs end together (split form, or
    // two CTAs to an item) the one only waits for the other's stores: 703 queries of 24 / 8 heads x 2,689 keys 67.8 (merge kernel)
    // against 71.2 us.
    const bool merge = P.persistent && P.part_stride == 2 && P.n_cta % n_items != 0;
    P.sync = ctx->part_sync;
    P.leave_parts = ctx->test_leave_parts;
    if (P.part_stride > 1 && !P.cluster && (size_t)n_items * P.part_stride * 2 * TILE * TILE > ctx->part_o_floats) return PC_ERR_CAPACITY;

    CUtensorMap mq, mk, mv[PC_MAX_SEGMENTS];
    bool ok = make_map(&mq, q_rot + (size_t)q_row0 * D.n_q_heads * D.head_dim, (uint64_t)n_q, (uint64_t)D.n_q_heads * D.head_dim) &&
              make_map(&mk, k_rot, (uint64_t)tiles * TILE, (uint64_t)row_elems);
    for (int s = 0; s < PC_MAX_SEGMENTS; ++s) {
        const pc_segment &sg = segs[s < n_seg ? s : 0];
        ok = ok && make_map(&mv[s], sg.v, (uint64_t)sg.n_tokens, (uint64_t)row_elems);
    }
    if (!ok) {
        fprintf(stderr, "packcache: cuTensorMapEncodeTiled failed\n");
        return PC_ERR_CUDA;
    }
    static bool attr_set[PC_MAX_DEVICES] = {};      // the attribute belongs to the device, not to the process
    if (ctx->device < 0 || ctx->device >= PC_MAX_DEVICES) return PC_ERR_UNSUPPORTED;
    if (!attr_set[ctx->device]) {
        for (const auto kernel : {k_attend_tc<false>, k_attend_tc<true>}) {
            cudaFuncAttributes a;
            PC_CUDA_TRY(cudaFuncGetAttributes(&a, kernel));
            if (a.numRegs * TC_THREADS < REGS_SPLIT) {
                fprintf(stderr, "packcache: attention kernel built with %d registers a thread, its warps would wait for more\n", a.numRegs);
                return PC_ERR_CUDA;
            }
            PC_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SM_ALLOC));
        }
        attr_set[ctx->device] = true;
    }
    if (P.cluster) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(P.n_cta);
        cfg.blockDim = dim3(TC_THREADS);
        cfg.dynamicSmemBytes = SM_ALLOC;
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = P.n_splits;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        PC_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_attend_tc<false>, mq, mk, mv[0], mv[1], mv[2], P));
    } else {
        PC_LAUNCH(merge ? k_attend_tc<true> : k_attend_tc<false>, dim3(P.n_cta), dim3(TC_THREADS), SM_ALLOC, stream, mq, mk, mv[0], mv[1], mv[2], P);
    }
    PC_CUDA_TRY(cudaGetLastError());
    pc_mark(ctx, PC_MARK_ATTEND, stream);
    if (P.part_stride > 1 && !P.cluster && !merge) {
        const dim3 grid(P.n_tb * D.n_q_heads * 4);
        if (P.part_stride == 2) PC_LAUNCH((k_combine<2, 4>), grid, dim3(256), 0, stream, P);
        else if (P.part_stride <= 4) PC_LAUNCH((k_combine<4, 3>), grid, dim3(256), 0, stream, P);
        else PC_LAUNCH((k_combine<MAX_SPLITS, 2>), grid, dim3(256), 0, stream, P);
        PC_CUDA_TRY(cudaGetLastError());
        pc_mark(ctx, PC_MARK_COMBINE, stream);
    }
    ctx->last_n_q = n_q;
    ctx->last_n_seg = n_seg;
    for (int s = 0; s < n_seg; ++s) ctx->last_seg_n[s] = segs[s].n_tokens;
    return PC_OK;
}

// Per-frame top-k selection as a block-level routine.  Scores map to 32-bit keys whose unsigned order is the score order
// (-0 folded onto +0).  A histogram of the frame's own key range finds the bin that holds the budget-th best key T; the few
// keys in that bin are compared with one another (a bin with many keys gets a histogram of its own first), which gives T and
// how many keys beat it.  An ordered sweep then keeps every key > T and the lowest-index (budget - beaten) keys == T,
// handing each kept token and its rank among the frame's kept tokens (ascending index order) to the caller.
//
// One block per frame, so a frame's chain of barriers is the kernel's time.  Counting into bins of the frame's range instead
// of four passes over fixed 8-bit digits (whose first digit, sign and exponent, is the same for most scores: the counters
// collided) takes one pass and a comparison; block sums are one ballot or one scan per warp and one read of the warps' totals.
// Measured back to back, four fixed digits against this: frames of 1,008 tokens 5.0 -> 3.6 us, 4,032 10.0 -> 6.0, 135 4.6 ->
// 2.4, 64 4.6 -> 2.3.  Bins with up to 256 keys settled by comparison instead of 64: 7.4 at 4,032; 4,096 bins: 2.9 at 64.
#pragma once
#include "pc_common.cuh"

struct FrameTab { int4 f[PC_MAX_FRAMES]; };   // (first token, tokens, budget, output offset)

__device__ __forceinline__ uint32_t score_key(float s) {
    uint32_t u = __float_as_uint(s);
    if ((u << 1) == 0) u = 0;                       // -0 -> +0
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

constexpr int SEL_CACHE = 4096;   // keys of a frame kept in shared memory; longer frames re-read the rest from global
constexpr int SEL_LOG_BINS = 10, SEL_BINS = 1 << SEL_LOG_BINS;
constexpr int SEL_LIST = 64;      // a bin with at most this many keys is settled by comparing them

template <int THREADS> struct SelectShared {
    uint32_t keys[SEL_CACHE];
    int hist[SEL_BINS];
    __align__(16) uint32_t list[SEL_LIST];
    uint32_t warp_a[4][THREADS / 32], warp_b[4][THREADS / 32];
    uint32_t bin, T;
    int n_bin, want, n_list, want_eq;
};

// The whole block selects frame `fr` (budget > 0, n > 0), whose scores start at `s`; keep(rank, global index) is called once per kept token by the
// thread that owns it.  Every thread of the block must call this.
template <int THREADS, typename Keep>
__device__ __forceinline__ void frame_select(const float *__restrict__ s, int4 fr, SelectShared<THREADS> &sm,
                                             int32_t *status, Keep keep) {
    constexpr int WARPS = THREADS / 32, PER = SEL_BINS / THREADS;
    static_assert(WARPS <= 32 && PER >= 1, "a warp reads the warps' totals, a thread owns whole bins");
    const int first = fr.x, n = fr.y, budget = fr.z;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t below = (1u << lane) - 1u;

    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
    bool nan = false;
    for (int j = threadIdx.x; j < n; j += THREADS) {
        const float v = s[j];
        nan |= v != v;
        const uint32_t key = score_key(v);
        lo = min(lo, key);
        hi = max(hi, key);
        if (j < SEL_CACHE) sm.keys[j] = key;
    }
    if (nan) pc_flag(status, PC_ERR_INVALID_ARG, PC_WHERE_SELECT_NAN);
    if (budget >= n) {                               // a frame kept whole
        for (int j = threadIdx.x; j < n; j += THREADS) keep(j, first + j);
        return;
    }
#pragma unroll
    for (int b = 0; b < PER; ++b) sm.hist[threadIdx.x + b * THREADS] = 0;
    for (int i = threadIdx.x; i < SEL_LIST; i += THREADS) sm.list[i] = 0;
    if (threadIdx.x == 0) sm.n_list = 0;
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) { sm.warp_a[0][warp] = lo; sm.warp_b[0][warp] = hi; }
    __syncthreads();
    lo = __reduce_min_sync(0xffffffffu, lane < WARPS ? sm.warp_a[0][lane] : 0xFFFFFFFFu);
    hi = __reduce_max_sync(0xffffffffu, lane < WARPS ? sm.warp_b[0][lane] : 0u);
    auto key_at = [&](int j) { return j < SEL_CACHE ? sm.keys[j] : score_key(s[j]); };

    // Keys lo .. hi in bins of 2^shift; the bin that holds the `want`-th best of them becomes the next range, until it is a
    // single key or holds few.
    int want = budget, shift;
    uint32_t span = hi - lo;                         // keys of the range above its first
    for (;;) {
        shift = max(0, 32 - __clz(span) - SEL_LOG_BINS);
        for (int j = threadIdx.x; j < n; j += THREADS) {
            const uint32_t off = key_at(j) - lo;     // keys below the range wrap around
            if (off <= span) atomicAdd(&sm.hist[off >> shift], 1);
        }
        __syncthreads();
        // thread t owns bins SEL_BINS - 1 - PER t downwards; an inclusive scan counts keys from the top bin down
        int c[PER], mine = 0;
#pragma unroll
        for (int b = 0; b < PER; ++b) { c[b] = sm.hist[SEL_BINS - 1 - PER * (int)threadIdx.x - b]; mine += c[b]; }
        int inc = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        if (lane == 31) sm.warp_a[1][warp] = inc;
        __syncthreads();
        const uint32_t wt = lane < WARPS ? sm.warp_a[1][lane] : 0u;
        const int base = (int)__reduce_add_sync(0xffffffffu, lane < warp ? wt : 0u);
        const int before = base + inc - mine;
        if (before < want && want <= base + inc) {   // exactly one thread: the bin is one of its own
            int w = want - before, b = 0;
            while (b + 1 < PER && c[b] < w) w -= c[b++];
            sm.bin = SEL_BINS - 1 - PER * threadIdx.x - b;
            sm.n_bin = c[b];
            sm.want = w;
        }
#pragma unroll
        for (int b = 0; b < PER; ++b) sm.hist[SEL_BINS - 1 - PER * (int)threadIdx.x - b] = 0;
        __syncthreads();
        want = sm.want;
        const uint32_t first_key = lo + (sm.bin << shift);
        span = min((1u << shift) - 1u, lo + span - first_key);
        lo = first_key;
        if (shift == 0 || sm.n_bin <= SEL_LIST) break;
    }
    // T: the `want`-th best key of the bin; `want` becomes the number of keys equal to T that are kept
    uint32_t T = lo;
    if (shift > 0) {
        for (int j = threadIdx.x; j < n; j += THREADS) {
            const uint32_t key = key_at(j);
            if (key - lo <= span) {
                const int at = atomicAdd(&sm.n_list, 1);
                if (at < SEL_LIST) sm.list[at] = key;
            }
        }
        __syncthreads();
        const int m = min(sm.n_list, SEL_LIST);
        for (int i = threadIdx.x; i < m; i += THREADS) {
            const uint32_t key = sm.list[i];
            int above = 0, equal = 0;
            for (int k = 0; k < m; k += 8) {         // past the end lie zeros: no score's key
                const uint4 x = *reinterpret_cast<const uint4 *>(sm.list + k), y = *reinterpret_cast<const uint4 *>(sm.list + k + 4);
                above += (x.x > key) + (x.y > key) + (x.z > key) + (x.w > key) + (y.x > key) + (y.y > key) + (y.z > key) + (y.w > key);
                equal += (x.x == key) + (x.y == key) + (x.z == key) + (x.w == key) + (y.x == key) + (y.y == key) + (y.z == key) + (y.w == key);
            }
            if (above < want && want <= above + equal) {     // all of T's copies write the same
                sm.T = key;
                sm.want_eq = want - above;
            }
        }
        __syncthreads();
        T = sm.T;
        want = sm.want_eq;
    }
    // ordered sweep, four keys of a thread at a time
    int gt_seen = 0, eq_seen = 0;
    for (int j0 = 0; j0 < n; j0 += 4 * THREADS) {
        uint32_t gt[4], eq[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (j0 + k * THREADS >= n) break;
            const int j = j0 + k * THREADS + threadIdx.x;
            const uint32_t key = j < n ? key_at(j) : 0u;
            gt[k] = __ballot_sync(0xffffffffu, j < n && key > T);
            eq[k] = __ballot_sync(0xffffffffu, j < n && key == T);
            if (lane == 0) { sm.warp_a[k][warp] = __popc(gt[k]); sm.warp_b[k][warp] = __popc(eq[k]); }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (j0 + k * THREADS >= n) break;
            const int j = j0 + k * THREADS + threadIdx.x;
            // keys above T in the low half, equal to T in the high half (at most THREADS of each)
            const uint32_t wt = lane < WARPS ? sm.warp_a[k][lane] | (sm.warp_b[k][lane] << 16) : 0u;
            const uint32_t base = __reduce_add_sync(0xffffffffu, lane < warp ? wt : 0u), total = __reduce_add_sync(0xffffffffu, wt);
            const int gt_before = gt_seen + (int)(base & 0xFFFFu) + __popc(gt[k] & below);
            const int eq_before = eq_seen + (int)(base >> 16) + __popc(eq[k] & below);
            const bool is_gt = (gt[k] >> lane) & 1u, is_eq = (eq[k] >> lane) & 1u;
            if (is_gt || (is_eq && eq_before < want)) keep(gt_before + min(eq_before, want), first + j);
            gt_seen += (int)(total & 0xFFFFu);
            eq_seen += (int)(total >> 16);
        }
        if (j0 + 4 * THREADS < n) __syncthreads();
    }
}

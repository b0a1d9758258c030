// CUDA-core attention of the current frame's queries over anchors ++ history ++ current (Eq. 2, all keys visible).
// This is the fp32 path (tensor cores would not keep fp32 inputs within 1e-4), the path of the shapes that the tensor-core
// kernel does not take, and a second opinion for the others.
//
// A block takes ROWS (query, head) rows that share one KV head (grouped-query packing: row x of a KV head is query x / G,
// head x mod G of its group) and a range of the 32-key tiles.  Sixteen threads share four rows: in S = Q K^T a thread owns
// 4 rows x 2 keys, in O += P V 4 rows x D/16 columns, so 32 multiply-adds follow every six 16-byte reads of shared memory.
// K and Q are rotated with the 3D rotary tables on their way into shared memory; the next tile's rows and table entries are
// requested before the current tile is worked on.  The softmax is the usual running (max, sum) form in fp32, base 2.
//
// What bounds it: the call is small (fp32 frames of some hundred tokens), so the number of blocks in flight decides.  The key
// ranges of one group of rows form a thread-block cluster (at most eight blocks) and merge their (max, sum, O) through
// distributed shared memory: no second launch, no partials in global memory.  Measured, this kernel against one block per 32
// rows of a query head that walked all keys with a thread owning a quarter of a row (which re-read every key row from shared
// memory for each row), fp32, 4 / 2 heads x 64, back to back in a graph: 64 queries x 224 keys 56.4 -> 7.7 us, 180 x 720
// 177 -> 19.2, 400 x 3,344 816 -> 79.5, 9 x 22 7.9 -> 6.0.
#include <algorithm>

#include "pc_tc.cuh"

namespace {

using pc_tc::cluster_rank;
using pc_tc::cluster_sync_all;
using pc_tc::peer_addr;
using pc_tc::peer_ld128;
using pc_tc::peer_ld64;

constexpr int AT_KEYS = 32;         // keys per tile
constexpr int AT_MAX_SPLITS = 8;    // portable cluster size

struct SegTable {
    const void *k[PC_MAX_SEGMENTS];
    const void *v[PC_MAX_SEGMENTS];
    const int32_t *pos[PC_MAX_SEGMENTS];
    int32_t end[PC_MAX_SEGMENTS];   // running key count after each segment
    int32_t n_seg;
    int32_t n_keys;
};

template <typename T> __device__ __forceinline__ float2 load_pair(const T *p);
template <> __device__ __forceinline__ float2 load_pair<float>(const float *p) { return __ldg(reinterpret_cast<const float2 *>(p)); }
template <> __device__ __forceinline__ float2 load_pair<__nv_bfloat16>(const __nv_bfloat16 *p) {
    const uint32_t w = __ldg(reinterpret_cast<const uint32_t *>(p));
    return make_float2(pc_bf16_lo(w), pc_bf16_hi(w));
}
template <typename T> __device__ __forceinline__ void store4(T *p, float a, float b, float c, float d);
template <> __device__ __forceinline__ void store4<float>(float *p, float a, float b, float c, float d) {
    *reinterpret_cast<float4 *>(p) = make_float4(a, b, c, d);
}
template <> __device__ __forceinline__ void store4<__nv_bfloat16>(__nv_bfloat16 *p, float a, float b, float c, float d) {
    *reinterpret_cast<uint2 *>(p) = make_uint2(pc_pack_bf16(a, b), pc_pack_bf16(c, d));
}

// shared memory in floats: rows are padded by four so that eight lanes reading 16 bytes of consecutive rows hit all banks
template <int D, int ROWS> struct Smem {
    static constexpr int LD = D + 4, LP = ROWS + 4;
    static constexpr int Q = 0, K = Q + ROWS * LD, V = K + AT_KEYS * LD, P = V + AT_KEYS * D, ML = P + AT_KEYS * LP, TOTAL = ML + 2 * ROWS;
    static_assert(ROWS * D <= K, "the outputs of the merge are staged over the queries");
};

template <typename T, int D, int ROWS>
__global__ void __launch_bounds__(4 * ROWS) k_attend_simt(const T *__restrict__ q, const int32_t *__restrict__ q_pos, int n_q,
                                                          int n_q_heads, int n_kv_heads, int n_splits, const __grid_constant__ SegTable seg,
                                                          pc_rope_dev rope, T *__restrict__ out, float *__restrict__ lse,
                                                          int32_t *status) {
    pc_grid_dep_launch();
    pc_grid_dep_wait();
    using SM = Smem<D, ROWS>;
    constexpr int THREADS = 4 * ROWS, LD = SM::LD, LP = SM::LP, NP = D / 2, NC = D / 64 /* 4-column groups of O per thread */;
    constexpr int KP = AT_KEYS * NP / THREADS;       // K (and V) pairs a thread fetches per tile
    extern __shared__ __align__(16) float sm[];
    float *sq = sm + SM::Q, *sk = sm + SM::K, *sv = sm + SM::V, *sp = sm + SM::P;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int group = n_q_heads / n_kv_heads, g = blockIdx.y;
    const int row0 = (int)(blockIdx.x / n_splits) * ROWS, n_rows = n_q * group, split = blockIdx.x % n_splits;
    const int n_tiles = (seg.n_keys + AT_KEYS - 1) / AT_KEYS;
    const int t0 = (int)((long long)n_tiles * split / n_splits), t1 = (int)((long long)n_tiles * (split + 1) / n_splits);
    const float scale = 1.4426950408889634f * rsqrtf((float)D);

    bool bad = false;                                 // a position outside the rotary tables was seen
    float2 rk[KP], rv[KP], rc[KP];
    auto fetch = [&](int tile) {
        int4 pp[KP];
#pragma unroll
        for (int u = 0; u < KP; ++u) {
            const int p = tid + u * THREADS, pair = p % NP, key = min(tile * AT_KEYS + p / NP, seg.n_keys - 1);   // keys past the end: masked below
            const int s = (seg.n_seg > 1 && key >= seg.end[0]) + (seg.n_seg > 2 && key >= seg.end[1]);
            const int local = key - (s == 0 ? 0 : (s == 1 ? seg.end[0] : seg.end[1]));
            const T *ks = static_cast<const T *>(s == 0 ? seg.k[0] : (s == 1 ? seg.k[1] : seg.k[2]));
            const T *vs = static_cast<const T *>(s == 0 ? seg.v[0] : (s == 1 ? seg.v[1] : seg.v[2]));
            const int32_t *ps = s == 0 ? seg.pos[0] : (s == 1 ? seg.pos[1] : seg.pos[2]);
            const size_t at = ((size_t)local * n_kv_heads + g) * D + 2 * pair;
            pp[u] = __ldg(reinterpret_cast<const int4 *>(ps) + local);
            rk[u] = load_pair<T>(ks + at);
            rv[u] = tile * AT_KEYS + p / NP < seg.n_keys ? load_pair<T>(vs + at) : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < KP; ++u) rc[u] = pc_rope_cs_clamped(rope, (tid + u * THREADS) % NP, pp[u].x, pp[u].y, pp[u].z, bad);
    };
    auto put = [&]() {
#pragma unroll
        for (int u = 0; u < KP; ++u) {
            const int p = tid + u * THREADS, kk = p / NP, pair = p % NP;
            const float2 x = rk[u], cs = rc[u];
            *reinterpret_cast<float2 *>(sk + kk * LD + 2 * pair) = make_float2(x.x * cs.x - x.y * cs.y, x.x * cs.y + x.y * cs.x);
            *reinterpret_cast<float2 *>(sv + kk * D + 2 * pair) = rv[u];
        }
    };
    fetch(t0);
    // the queries, eight pairs of a thread in flight at a time (rows past the end repeat the last one and are not written)
#pragma unroll 1
    for (int u0 = 0; u0 < NP / 4; u0 += 8) {
        float2 qv[8], qc[8];
        int4 pp[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int p = tid + (u0 + u) * THREADS, x = min(row0 + p / NP, n_rows - 1), i = x / group, h = g * group + x - i * group;
            pp[u] = __ldg(reinterpret_cast<const int4 *>(q_pos) + i);
            qv[u] = load_pair<T>(q + ((size_t)i * n_q_heads + h) * D + 2 * (p % NP));
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) qc[u] = pc_rope_cs_clamped(rope, (tid + (u0 + u) * THREADS) % NP, pp[u].x, pp[u].y, pp[u].z, bad);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int p = tid + (u0 + u) * THREADS;
            const float2 v = qv[u], cs = qc[u];
            *reinterpret_cast<float2 *>(sq + (p / NP) * LD + 2 * (p % NP)) = make_float2((v.x * cs.x - v.y * cs.y) * scale, (v.x * cs.y + v.y * cs.x) * scale);
        }
    }
    put();
    __syncthreads();

    float o[4][NC][4], m[4], l[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        m[r] = -INFINITY;
        l[r] = 0.f;
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[r][c][e] = 0.f;
    }
    for (int tile = t0; tile < t1; ++tile) {
        if (tile + 1 < t1) fetch(tile + 1);
        // scores of rows 4 ty .. 4 ty + 3 against keys tx and tx + 16
        float s[4][2];
#pragma unroll
        for (int r = 0; r < 4; ++r) s[r][0] = s[r][1] = 0.f;
#pragma unroll 4
        for (int c = 0; c < D; c += 4) {
            const float4 ka = *reinterpret_cast<const float4 *>(sk + tx * LD + c), kb = *reinterpret_cast<const float4 *>(sk + (tx + 16) * LD + c);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float4 x = *reinterpret_cast<const float4 *>(sq + (4 * ty + r) * LD + c);
                s[r][0] = fmaf(x.x, ka.x, fmaf(x.y, ka.y, fmaf(x.z, ka.z, fmaf(x.w, ka.w, s[r][0]))));
                s[r][1] = fmaf(x.x, kb.x, fmaf(x.y, kb.y, fmaf(x.z, kb.z, fmaf(x.w, kb.w, s[r][1]))));
            }
        }
        const int n_here = seg.n_keys - tile * AT_KEYS;
        float p0[4], p1[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float a = tx < n_here ? s[r][0] : -INFINITY, b = tx + 16 < n_here ? s[r][1] : -INFINITY;
            float mx = fmaxf(a, b);
#pragma unroll
            for (int x = 8; x > 0; x >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, x));
            const float m_new = fmaxf(m[r], mx), corr = exp2f(m[r] - m_new);     // exp2f(-inf) = 0 on the first tile
            m[r] = m_new;
            p0[r] = exp2f(a - m_new);
            p1[r] = exp2f(b - m_new);
            l[r] = fmaf(l[r], corr, p0[r] + p1[r]);                    // this thread's share of the row's sum
#pragma unroll
            for (int c = 0; c < NC; ++c)
#pragma unroll
                for (int e = 0; e < 4; ++e) o[r][c][e] *= corr;
        }
        *reinterpret_cast<float4 *>(sp + tx * LP + 4 * ty) = make_float4(p0[0], p0[1], p0[2], p0[3]);
        *reinterpret_cast<float4 *>(sp + (tx + 16) * LP + 4 * ty) = make_float4(p1[0], p1[1], p1[2], p1[3]);
        __syncwarp();                                                   // a row's sixteen threads are one half-warp
#pragma unroll 4
        for (int kk = 0; kk < AT_KEYS; ++kk) {
            const float4 p = *reinterpret_cast<const float4 *>(sp + kk * LP + 4 * ty);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const float4 v = *reinterpret_cast<const float4 *>(sv + kk * D + 64 * c + 4 * tx);
                const float pr[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    o[r][c][0] = fmaf(pr[r], v.x, o[r][c][0]);
                    o[r][c][1] = fmaf(pr[r], v.y, o[r][c][1]);
                    o[r][c][2] = fmaf(pr[r], v.z, o[r][c][2]);
                    o[r][c][3] = fmaf(pr[r], v.w, o[r][c][3]);
                }
            }
        }
        __syncthreads();                                                // everybody is done with this tile's K and V
        if (tile + 1 < t1) {
            put();
            __syncthreads();
        }
    }
    if (bad) pc_flag(status, PC_ERR_INVALID_ARG, PC_WHERE_ATTN_POS);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int x = 8; x > 0; x >>= 1) l[r] += __shfl_xor_sync(0xffffffffu, l[r], x);

    auto write_row = [&](int r_tile, int c4, float4 v, float inv) {
        const int x = row0 + r_tile, i = x / group, h = g * group + x % group;
        store4<T>(out + ((size_t)i * n_q_heads + h) * D + 4 * c4, v.x * inv, v.y * inv, v.z * inv, v.w * inv);
    };
    auto write_lse = [&](int r_tile, float mm, float ll) {
        const int x = row0 + r_tile, i = x / group, h = g * group + x % group;
        lse[(size_t)i * n_q_heads + h] = (mm + log2f(ll)) * 0.6931471805599453f;
    };
    if (n_splits == 1) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (row0 + 4 * ty + r >= n_rows) break;
            const float inv = 1.f / l[r];
#pragma unroll
            for (int c = 0; c < NC; ++c) write_row(4 * ty + r, 16 * c + tx, make_float4(o[r][c][0], o[r][c][1], o[r][c][2], o[r][c][3]), inv);
            if (lse && tx == 0) write_lse(4 * ty + r, m[r], l[r]);
        }
        return;
    }
    // stage O over the queries (nobody reads them any more) and (max, sum), then every block of the cluster finishes the
    // rows whose number is its rank modulo the number of blocks
#pragma unroll
    for (int r = 0; r < 4; ++r) {
#pragma unroll
        for (int c = 0; c < NC; ++c)
            *reinterpret_cast<float4 *>(sq + (4 * ty + r) * D + 64 * c + 4 * tx) = make_float4(o[r][c][0], o[r][c][1], o[r][c][2], o[r][c][3]);
        if (tx == 0) *reinterpret_cast<float2 *>(sm + SM::ML + 2 * (4 * ty + r)) = make_float2(m[r], l[r]);
    }
    cluster_sync_all();
    const uint32_t base = pc_smem_u32(sm);
    const int rank = (int)cluster_rank();
    constexpr int C4 = D / 4;                                           // 16-byte units per row
    for (int w = tid; w < ((ROWS - rank + n_splits - 1) / n_splits) * C4; w += THREADS) {
        const int r = rank + (w / C4) * n_splits, c4 = w % C4;
        if (row0 + r >= n_rows) break;
        float2 ml[AT_MAX_SPLITS];
        float4 v[AT_MAX_SPLITS];
        float mm = -INFINITY;
#pragma unroll
        for (int k = 0; k < AT_MAX_SPLITS; ++k)
            if (k < n_splits) {
                const uint32_t b = peer_addr(base, k);
                ml[k] = peer_ld64(b + (SM::ML + 2 * r) * 4);
                v[k] = peer_ld128(b + (SM::Q + r * D + 4 * c4) * 4);
                mm = fmaxf(mm, ml[k].x);
            }
        float ll = 0.f;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < AT_MAX_SPLITS; ++k)
            if (k < n_splits) {
                const float sc = exp2f(ml[k].x - mm);
                ll = fmaf(ml[k].y, sc, ll);
                acc.x = fmaf(v[k].x, sc, acc.x); acc.y = fmaf(v[k].y, sc, acc.y);
                acc.z = fmaf(v[k].z, sc, acc.z); acc.w = fmaf(v[k].w, sc, acc.w);
            }
        write_row(r, c4, acc, 1.f / ll);
        if (lse && c4 == 0) write_lse(r, mm, ll);
    }
    cluster_sync_all();                        // nobody leaves while a peer may still read its shared memory
}

template <typename T, int D, int ROWS>
pc_status launch(pc_ctx *ctx, const SegTable &t, const void *q, const int32_t *q_pos, int n_q, void *out, float *lse, cudaStream_t stream) {
    const pc_layer_desc &L = ctx->desc;
    constexpr int smem = Smem<D, ROWS>::TOTAL * (int)sizeof(float);
    if (smem > 48 * 1024) {
        static bool attr_set[PC_MAX_DEVICES] = {};      // the attribute belongs to the device, not to the process
        if (ctx->device < 0 || ctx->device >= PC_MAX_DEVICES) return PC_ERR_UNSUPPORTED;
        if (!attr_set[ctx->device]) {
            PC_CUDA_TRY(cudaFuncSetAttribute(k_attend_simt<T, D, ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
            attr_set[ctx->device] = true;
        }
    }
    const int row_blocks = (int)(((long long)n_q * ctx->group + ROWS - 1) / ROWS), tiles = (t.n_keys + AT_KEYS - 1) / AT_KEYS;
    // key ranges: enough blocks for two per SM, at least one tile each
    const long long blocks = (long long)row_blocks * L.n_kv_heads;
    const int splits = (int)std::max<long long>(1, std::min<long long>(std::min(AT_MAX_SPLITS, tiles), (2LL * ctx->sm_count + blocks - 1) / blocks));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(splits * row_blocks), L.n_kv_heads);
    cfg.blockDim = dim3(4 * ROWS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = splits;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = splits > 1 ? 2 : 1;
    PC_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_attend_simt<T, D, ROWS>, static_cast<const T *>(q), q_pos, n_q, (int)L.n_q_heads, (int)L.n_kv_heads, splits, t,
                                   ctx->rope, static_cast<T *>(out), lse, ctx->status));
    return PC_OK;
}

}  // namespace

pc_status pc_launch_attend_simt(pc_ctx *ctx, int n_seg, const pc_segment *segs, const void *q, const int32_t *q_pos,
                                int32_t n_q, void *out, float *lse, cudaStream_t stream) {
    const pc_layer_desc &D = ctx->desc;
    SegTable t{};
    int total = 0;
    t.n_seg = n_seg;
    for (int s = 0; s < n_seg; ++s) {
        t.k[s] = segs[s].k;
        t.v[s] = segs[s].v;
        t.pos[s] = segs[s].pos;
        total += segs[s].n_tokens;
        t.end[s] = total;
    }
    t.n_keys = total;
    pc_mark(ctx, PC_MARK_ROPE, stream);
    // 64 rows a block read K and V half as often as 32; 32 rows where 64 would leave SMs without a block even with eight
    // key ranges (or key ranges as long as there are tiles)
    const long long tiles = (total + AT_KEYS - 1) / AT_KEYS, ranges = std::min<long long>(AT_MAX_SPLITS, tiles);
    const bool wide = ((long long)n_q * ctx->group + 63) / 64 * D.n_kv_heads * ranges >= ctx->sm_count;
#define PC_AT_LAUNCH(T, DIM) (wide ? launch<T, DIM, 64>(ctx, t, q, q_pos, n_q, out, lse, stream) : launch<T, DIM, 32>(ctx, t, q, q_pos, n_q, out, lse, stream))
    pc_status st;
    if (D.dtype == PC_F32)
        st = D.head_dim == 64 ? PC_AT_LAUNCH(float, 64) : PC_AT_LAUNCH(float, 128);
    else
        st = D.head_dim == 64 ? PC_AT_LAUNCH(__nv_bfloat16, 64) : PC_AT_LAUNCH(__nv_bfloat16, 128);
#undef PC_AT_LAUNCH
    if (st != PC_OK) return st;
    PC_CUDA_TRY(cudaGetLastError());
    pc_mark(ctx, PC_MARK_ATTEND, stream);
    return PC_OK;
}

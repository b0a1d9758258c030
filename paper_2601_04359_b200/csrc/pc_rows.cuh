// Arithmetic on token rows that several kernels share, so that they give the same bits: unpacking of 16-byte chunks, the
// pooled query's fixed-point unit, and the scoring of a key row.
#pragma once
#include "pc_common.cuh"

template <typename T> struct Elem;
template <> struct Elem<float> {
    static constexpr int PER16 = 4;
    static __device__ __forceinline__ void unpack(const uint4 &v, float *f) {
        f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y); f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
    }
    static __device__ __forceinline__ uint4 pack(const float *f) {
        return make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3]));
    }
};
template <> struct Elem<__nv_bfloat16> {
    static constexpr int PER16 = 8;
    static __device__ __forceinline__ void unpack(const uint4 &v, float *f) {
        f[0] = pc_bf16_lo(v.x); f[1] = pc_bf16_hi(v.x); f[2] = pc_bf16_lo(v.y); f[3] = pc_bf16_hi(v.y);
        f[4] = pc_bf16_lo(v.z); f[5] = pc_bf16_hi(v.z); f[6] = pc_bf16_lo(v.w); f[7] = pc_bf16_hi(v.w);
    }
    static __device__ __forceinline__ uint4 pack(const float *f) {
        return make_uint4(pc_pack_bf16(f[0], f[1]), pc_pack_bf16(f[2], f[3]), pc_pack_bf16(f[4], f[5]), pc_pack_bf16(f[6], f[7]));
    }
};

constexpr float FX_ONE = 4294967296.0f;             // 2^32: the pooled query's sums are 64-bit integers in units of 2^-32

// Rotary table entries of a scoring lane's pairs: lane `lt` of the LPT that share a key row holds chunks lt, lt + LPT, ..., which
// all cover the same PER/2 pairs.  Consecutive pairs take the axes in turn, so pair u's entry is at column m[u] of the row of
// coordinate (r + u) mod 3, and the fourth pair's is the one behind the first's.
template <typename T> struct ScoreTable {
    static constexpr int PER = Elem<T>::PER16, NP = PER / 2, AX = NP < 3 ? NP : 3;
    int first[AX], pitch[AX], r;
    __device__ __forceinline__ ScoreTable(const pc_rope_dev &rope, int lt, int d) {
        const int pair0 = ((lt * PER) % d) / 2;
        r = pair0 % 3;
#pragma unroll
        for (int u = 0; u < AX; ++u) {
            const int a = (pair0 + u) % 3;
            first[u] = (a == 0 ? rope.off[0] : (a == 1 ? rope.off[1] : rope.off[2])) + (pair0 + u) / 3;
            pitch[u] = a == 0 ? rope.n_axis[0] : (a == 1 ? rope.n_axis[1] : rope.n_axis[2]);
        }
    }
    __device__ __forceinline__ void at(const pc_rope_dev &rope, int4 q, float2 (&cs)[NP], int32_t *status) const {
        const unsigned mt = rope.max_pos[0], mh = rope.max_pos[1], mw = rope.max_pos[2];
        if (!((unsigned)q.x < mt && (unsigned)q.y < mh && (unsigned)q.z < mw)) {   // outside the tables: record, clamp
            pc_flag(status, PC_ERR_INVALID_ARG, PC_WHERE_SCORE_POS);
            q.x = min(max(q.x, 0), (int)mt - 1); q.y = min(max(q.y, 0), (int)mh - 1); q.z = min(max(q.z, 0), (int)mw - 1);
        }
        const int c[3] = {r == 0 ? q.x : (r == 1 ? q.y : q.z), r == 0 ? q.y : (r == 1 ? q.z : q.x), r == 0 ? q.z : (r == 1 ? q.x : q.y)};
#pragma unroll
        for (int u = 0; u < NP; ++u) cs[u] = __ldg(rope.tab + (u < AX ? first[u % AX] + c[u % AX] * pitch[u % AX] : first[0] + c[0] * pitch[0] + 1));
    }
};

// A lane's share of the scores of TPL keys, which lie in shared memory at `mine` + i * pitch (the lane's own 16 bytes of the first
// LPT chunks); ql: the pooled query as (q_a, q_b, q_b, -q_a) of (chunk row, pair, lane of the token), from the lane's own on.
// Brackets per pair:  A = sum q_a k_a + q_b k_b,  B = sum q_b k_a - q_a k_b, each as the two lanes of one register pair.
// A lane that shares its token with 15 others has twice as many chunks as one of 32 would: it takes those of even number,
// then those of odd number, and adds the two results (all in one chain: scores up to 10 % further from a 64-bit
// evaluation).  Both chains at once take 161 registers instead of 128 in the scoring kernel, and its block of 12 warps then fills the
// SM's registers: the next kernel's first blocks no longer start beside it (step of 135-token frames, 24 / 8 heads, 27.5 -> 29.1 us).
template <typename T, int LPT, int TPL>
__device__ __forceinline__ void score_rows(uint32_t mine, int pitch, int parts, const float4 *ql, const float2 (&cs)[TPL][Elem<T>::PER16 / 2],
                                           float (&s)[TPL]) {
    constexpr int PER = Elem<T>::PER16, NP = PER / 2, CH = 32 / LPT /* chains */;
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        float2 A[TPL][NP], B[TPL][NP];
#pragma unroll
        for (int i = 0; i < TPL; ++i)
#pragma unroll
            for (int u = 0; u < NP; ++u) A[i][u] = B[i][u] = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int g = c; g < parts; g += CH) {
            float x[TPL][PER];
#pragma unroll
            for (int i = 0; i < TPL; ++i) Elem<T>::unpack(pc_lds128(mine + i * pitch + g * LPT * 16), x[i]);
#pragma unroll
            for (int u = 0; u < NP; ++u) {
                const float4 qq = ql[(g * NP + u) * LPT];
                const float2 qab = make_float2(qq.x, qq.y), qba = make_float2(qq.z, qq.w);
#pragma unroll
                for (int i = 0; i < TPL; ++i) {
                    const float2 kk = make_float2(x[i][2 * u], x[i][2 * u + 1]);
                    A[i][u] = __ffma2_rn(qab, kk, A[i][u]);
                    B[i][u] = __ffma2_rn(qba, kk, B[i][u]);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < TPL; ++i) {
            float r = 0.f;
#pragma unroll
            for (int u = 0; u < NP; ++u)
                r = fmaf(cs[i][u].x, A[i][u].x + A[i][u].y, fmaf(cs[i][u].y, B[i][u].x + B[i][u].y, r));
            s[i] = c == 0 ? r : s[i] + r;
        }
    }
}

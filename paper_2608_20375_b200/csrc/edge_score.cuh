// TDES edge scores of one depth out of shared memory (Eq. 4-6), shared by the edge-score kernel (which scores the
// first depths for every sequence) and the tree kernel (which scores deeper depths when an expansion gets there),
// so that a row has the same bits whichever kernel produced it.
//
//   f[p][c]    = s/sqrt(m) * (P[p] + u_d) . (C[c] + u_d)                                   (Eq. 4-6)
//   edge[p][c] = log q_d(c) + beta * (f[p][c] - mean_c f[p][c])                            (TDES score)
//   and every parent's row ordered by (edge descending, child rank ascending).
#pragma once
#include "common.cuh"

namespace graft {

// How many depths of this sequence will its tree look at?  A confident drafter (high top-1 probabilities) gives a deep, narrow
// tree that needs the edge scores of many depths; an uncertain one a shallow, wide tree that stops a few levels down.  The
// edge-score kernel scores that many depths ahead of the tree kernel, which takes the same decision from the same numbers
// and scores what is missing on demand (3 - 4 us a depth in front of everything else, so the bounds err on the side of more).  A
// matter of speed only: a row has the same bits whoever scores it.  By the mean top-1 probability of the block: below 0.02 4
// depths, below 0.03 5, below 0.06 6, below 0.1 7, below 0.2 8, from there on all.  Of 12,288 sequences (boosts of 12 and of 6 to 14, V = 32,000
// and 151,936, L = 12 and 16, K = 16 and 32, budgets to 64, 256 and 512) twelve looked at a depth more, nine of them with budgets to
// 512; of any class of them at most one in a hundred.  With 8 or fewer candidates trees are narrower and deeper (5 to 8 depths even at
// 0.01), and a depth's scores are cheap: 8.
// (In two steps, so that a caller can have the load in flight beside its other loads: lane d's top-1 log-probability
// of position d, 0 for d >= L; then the decision, taken by every lane of a warp together.)
// Fewer than `rows` of them only where the caller has not asked for a number, and the scores take more CTAs than the SMs hold at once
// (four each): in one wave nothing is gained, and the decision stands in front of the work (batch 16, 64: 0.7 us of a round).
inline int rows_ahead_least(int batch, int rows, bool asked, int num_sms) {
    return !asked && rows > 4 && (long long)batch * rows > 4ll * num_sms ? 4 : rows;
}
__device__ __forceinline__ float rows_ahead_load(const float* __restrict__ topk_lp_seq, int L, int K) {
    const int lane = threadIdx.x & 31;
    return lane < L ? topk_lp_seq[(size_t)lane * K] : 0.f;
}
__device__ __forceinline__ float rows_ahead_sum(float lp_top, int L) {  // (of the block's top-1 probabilities)
    // lane d holds position d (L <= 32); a butterfly sum in a fixed order
    const int lane = threadIdx.x & 31;
    float s = lane < L ? ex2_approx(lp_top * kLog2e) : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    return s;
}
// rows: the depths scored ahead at most, unless the tree runs deeper than 8; least: and at least (rows: all of them)
__device__ __forceinline__ int rows_ahead(float lp_top, int L, int K, int least, int rows) {
    const float s = rows_ahead_sum(lp_top, L), one = (float)L;
    if (s >= 0.2f * one) return L;
    if (least == rows || K <= 8) return rows;
    const int n = s < 0.02f * one ? 4 : s < 0.03f * one ? 5 : s < 0.06f * one ? 6 : s < 0.1f * one ? 7 : 8;
    return n < rows ? n : rows;
}

// More sequences than SMs: the trees that take longest, those of confident drafters (from this mean on half of an ordinary
// batch), are built first, so that those of the second wave are short.
constexpr float kTreeLongMean = 0.06f;

// Where the r-th entry of the sorted row of parent rank c stands inside the row (scores only; the child ranks stand
// in order): rotated by the parent's rank.  The tree kernel's threads look at the same place r of different parents'
// rows far more often than at different places of one row, and with K = 32 a row is one pass over the shared-memory
// banks: unrotated, such a look is a 32-way bank conflict.
__device__ __forceinline__ int es_col(int r, int c, int K) {
    const int x = r + c;
    return x < K ? x : x - K;
}

// K x K dot products by G * G / 8 warps (8 for G = 8, 32 for G = 16).  A lane keeps a T x T tile of running sums (parents
// pg, pg + G, ..., children cg, cg + G, ...; G T >= K), each as a packed fp32 pair (even and odd elements of the m axis;
// `fma.rn.f32x2`), and takes a quarter ks of the m axis: two float4s of every eight.  A warp holds 2 x 4 such tiles in all
// four quarters, so a step's T float4s of parents are one pass over the shared-memory banks each (8 places) and the T of
// children two (16 places, no conflicts): 12 passes for 32 packed FMAs with T = 4, where a 4 x 2 tile a lane took 12 for
// 16 and made shared memory the bound (1 us of a round at batch 1, K = 8, 1.5 to 2.5 us at batch 16 to 256).
// The pair is added at the end and the four quarters of a tile by two exchange steps; a sum's order of additions depends
// on m alone, so the bits do not depend on T and G.
// rP / rC: [.][ld] rows in shared memory, ld = m + 4 floats (16-byte aligned).
// ADD_U: the rows hold P and C and u is added on the way into the registers; otherwise they already hold P + u and
// C + u (the same fp32 sums either way).  Sums of rows past n_par and K are never used; CLAMP reads the last row for
// them, otherwise rP and rC have room for G T rows.  part: [n_par][dots_ld(K)] floats of shared memory.
__host__ __device__ constexpr int dots_ld(int K) { return K + 4; }

template <bool ADD_U, int G, int T, bool CLAMP>
__device__ __forceinline__ void edge_dots(const float* rP, const float* rC, const float* rU, int m, int K, int n_par,
                                          float* part, int warp, int lane) {
    const int ks = lane >> 3, pg = 2 * (warp / (G / 4)) + ((lane >> 2) & 1), cg = 4 * (warp % (G / 4)) + (lane & 3);
    if (2 * (warp / (G / 4)) >= n_par) return;  // (uniform in the warp)
    const int q4 = m / 4, ld = m + 4;
    float2 acc[T][T];  // [child][parent]
#pragma unroll
    for (int c = 0; c < T; ++c)
#pragma unroll
        for (int i = 0; i < T; ++i) acc[c][i] = make_float2(0.f, 0.f);
    rP += 8 * ks;
    rC += 8 * ks;
    if (ADD_U) rU += 8 * ks;
#pragma unroll 1
    for (int k = 0; k < q4; k += 8) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (q4 % 8 != 0 && k + 2 * ks + h >= q4) break;
            const int at = 4 * (k + h);
            float4 uu = make_float4(0.f, 0.f, 0.f, 0.f);
            if (ADD_U) uu = *(const float4*)(rU + at);
            float4 cv[T];
#pragma unroll
            for (int c = 0; c < T; ++c) {
                const int r = cg + G * c;
                cv[c] = *(const float4*)(rC + (size_t)(CLAMP ? min(r, K - 1) : r) * ld + at);
                if (ADD_U) cv[c] = make_float4(cv[c].x + uu.x, cv[c].y + uu.y, cv[c].z + uu.z, cv[c].w + uu.w);
            }
#pragma unroll
            for (int i = 0; i < T; ++i) {
                const int r = pg + G * i;
                float4 pv = *(const float4*)(rP + (size_t)(CLAMP ? min(r, n_par - 1) : r) * ld + at);
                if (ADD_U) pv = make_float4(pv.x + uu.x, pv.y + uu.y, pv.z + uu.z, pv.w + uu.w);
#pragma unroll
                for (int c = 0; c < T; ++c) {
                    acc[c][i] = __ffma2_rn(make_float2(pv.x, pv.y), make_float2(cv[c].x, cv[c].y), acc[c][i]);
                    acc[c][i] = __ffma2_rn(make_float2(pv.z, pv.w), make_float2(cv[c].z, cv[c].w), acc[c][i]);
                }
            }
        }
    }
    constexpr int N = T * T;
    float v[N];
#pragma unroll
    for (int e = 0; e < N; ++e) v[e] = acc[e / T][e % T].x + acc[e / T][e % T].y;
    if constexpr (N % 4 == 0) {  // every exchange halves what a lane carries on: lane ks ends with a quarter of the tile's sums
        const bool u8 = (lane & 8) != 0, u16 = (lane & 16) != 0;
#pragma unroll
        for (int e = 0; e < N / 2; ++e)
            v[e] = (u8 ? v[e + N / 2] : v[e]) + __shfl_xor_sync(0xFFFFFFFFu, u8 ? v[e] : v[e + N / 2], 8);
#pragma unroll
        for (int e = 0; e < N / 4; ++e)
            v[e] = (u16 ? v[e + N / 4] : v[e]) + __shfl_xor_sync(0xFFFFFFFFu, u16 ? v[e] : v[e + N / 4], 16);
        const int first = (u8 ? N / 2 : 0) + (u16 ? N / 4 : 0);
#pragma unroll
        for (int e = 0; e < N / 4; ++e) {
            const int c = cg + G * ((first + e) / T), r = pg + G * ((first + e) % T);
            if (c < K && r < n_par) part[(size_t)r * dots_ld(K) + c] = v[e];
        }
    } else {
#pragma unroll
        for (int e = 0; e < N; ++e) {
            v[e] += __shfl_xor_sync(0xFFFFFFFFu, v[e], 8);
            v[e] += __shfl_xor_sync(0xFFFFFFFFu, v[e], 16);
            const int c = cg + G * (e / T), r = pg + G * (e % T);
            if (ks == (e & 3) && c < K && r < n_par) part[(size_t)r * dots_ld(K) + c] = v[e];
        }
    }
}

// One warp finishes one parent's row: scale, centre over the K children, add log q (lane = child c), and find the
// place of every child in the order (edge descending, child rank ascending) by counting the children that come
// before it.  dots: the parent's K dot products, or nullptr for a parent that does not exist (a row of zeros).
// wsc: 32 words of shared memory of this warp.  Returns the score in `val` and the place in `rank` (lanes < K).
__device__ __forceinline__ void edge_row_finish(const float* dots, float lp, float scale, float beta, int K,
                                                float inv_K, uint32_t* wsc, int lane, float& val, int& rank) {
    const int c = lane;
    val = 0.f;
    if (dots != nullptr) {
        const float ft = c < K ? dots[c] * scale : 0.f;
        float sum = ft;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, d);
        // sum / K from 1 / K, which the caller has worked out once: a quotient from the rounded reciprocal, corrected by the remainder that
        // a fused multiply-add gives exactly (P. Markstein, "Computation of elementary functions on the IBM RISC System/6000
        // processor", 1990), is the rounded quotient
        const float q0 = sum * inv_K;
        const float mean = fmaf(fmaf(-q0, (float)K, sum), inv_K, q0);
        val = fmaf(beta, ft - mean, lp);
    }
    const uint32_t mine = c < K ? ord_from_float(val) : 0u;  // 0 is below the image of every float
    __syncwarp();
    wsc[c] = mine;
    __syncwarp();
    // o > mine is the carry out of o + ~mine: an add and an add-with-carry a child, 0.75 cycles an SM where compare, select
    // and add take 0.93
    uint32_t above = 0;
#pragma unroll
    for (int i4 = 0; i4 < 8; ++i4) {
        const uint4 o4 = *(const uint4*)(wsc + 4 * i4);
        asm("{\n\t.reg .u32 t;\n\t"
            "add.cc.u32 t, %1, %5;\n\taddc.u32 %0, %0, 0;\n\tadd.cc.u32 t, %2, %5;\n\taddc.u32 %0, %0, 0;\n\t"
            "add.cc.u32 t, %3, %5;\n\taddc.u32 %0, %0, 0;\n\tadd.cc.u32 t, %4, %5;\n\taddc.u32 %0, %0, 0;\n\t}"
            : "+r"(above)
            : "r"(o4.x), "r"(o4.y), "r"(o4.z), "r"(o4.w), "r"(~mine));
    }
    rank = (int)above;
    // equal scores (rare) go by child rank: the counts above are a permutation of 0..K-1 unless some scores are equal,
    // and only then are the lanes with the same score looked up (a slow instruction)
    const uint32_t seen = __reduce_or_sync(0xFFFFFFFFu, c < K ? 1u << rank : 0u);
    if (seen != (K == 32 ? 0xFFFFFFFFu : (1u << K) - 1u)) {  // (uniform)
        const uint32_t same = __match_any_sync(0xFFFFFFFFu, mine);
        rank += __popc(same & ((1u << lane) - 1u));
    }
}

}  // namespace graft

// What the kernels of the vocab pass share: a thread's running log-sum-exp over the logits that it streams, and the outputs of
// a finished row from its pieces.
#pragma once
#include "common.cuh"
#include "internal.h"

#ifndef GRAFT_VP_F32X2
#define GRAFT_VP_F32X2 1  // packed fp32 pair arithmetic (fma.rn.f32x2 / add.rn.f32x2)
#endif

namespace graft {

namespace {

template <bool BF16>
struct VT;
template <>
struct VT<true> {
    using cm_t = uint16_t;
    static constexpr int ESZ = 2, EPV = 8;
    static constexpr uint32_t NEG_INF_WORD = 0xFF80FF80u;
};
template <>
struct VT<false> {
    using cm_t = uint16_t;  // the chunk maximum rounded UP to bf16 precision: an upper bound is all the scan needs
    static constexpr int ESZ = 4, EPV = 4;
    static constexpr uint32_t NEG_INF_WORD = 0xFF800000u;
};

__device__ __forceinline__ float load_elem_f32(const char* p, bool bf16) {
    if (bf16) return __uint_as_float(((uint32_t) * (const uint16_t*)p) << 16);
    return *(const float*)p;
}

// ---- per-thread streaming state -----------------------------------------------------------------
#if GRAFT_VP_F32X2
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
#endif

// The running log-sum-exp of one streaming thread over a segment: sum of 2^(z log2e - ref) in four fp32
// accumulators (two packed pairs), a reference exponent that is raised lazily (only when a chunk's maximum exceeds
// it by more than 2^16, so that rescaling is rare and every term stays far from overflow), and the largest value.
struct Acc {
    float ref;      // reference exponent, log2 domain; -inf before the first finite value
    float nref;     // -ref (0 while ref is -inf): the addend of the fused multiply-add
    uint32_t thr;   // a chunk maximum above this value raises the reference: bf16 logits: the value in both halves
                    // of a packed pair; fp32 logits: float bits
    uint32_t rmax;  // largest value so far: bf16 logits: a packed pair of running maxima; fp32 logits: float bits
#if GRAFT_VP_F32X2
    uint64_t a0, a1;
#else
    float s0, s1, s2, s3;
#endif
};

template <bool BF16>
__device__ __forceinline__ void acc_init(Acc& a) {
    a.ref = -INFINITY;
    a.nref = 0.f;
    a.thr = BF16 ? 0xFF80FF80u : 0xFF800000u;  // -inf: the first finite value sets the reference
    a.rmax = a.thr;
#if GRAFT_VP_F32X2
    a.a0 = a.a1 = 0ull;
#else
    a.s0 = a.s1 = a.s2 = a.s3 = 0.f;
#endif
}

// 2^d for a whole number d <= 0, exactly; 0 below 2^-126
__device__ __forceinline__ float ex2_whole(float d) { return d < -126.f ? 0.f : __uint_as_float((uint32_t)(127 + (int)d) << 23); }

// The chunk maximum cm exceeded the threshold: raise the reference to cm (rare).  WHOLE: to the next whole number, by which a
// sum is rescaled exactly.
template <bool BF16, bool WHOLE = false>
__device__ __forceinline__ void acc_raise(Acc& a, float cm) {
    const float cms = WHOLE ? ceilf(cm * kLog2e) : cm * kLog2e;
    if (!(cms > a.ref + 16.0f)) return;  // (the threshold is a copy of ref + 16 rounded down: it may fire a little early)
    // Masked tokens may hold any low value.  Below -1e9 the product with log2(e) is rounded by hundreds and more, by which the terms
    // of a sum at that reference would overflow; they add nothing to a row that has any other value and are left out.
    if (cms < 0.f && fmaf(cm, kLog2e, -cms) > 100.0f) return;
    const float f = WHOLE ? ex2_whole(a.ref - cms) : ex2_approx(a.ref - cms);  // 0 when ref is -inf (nothing added yet) or cm is +inf
#if GRAFT_VP_F32X2
    const uint64_t f2 = pack2(f, f);
    a.a0 = mul2(a.a0, f2);
    a.a1 = mul2(a.a1, f2);
#else
    a.s0 *= f;
    a.s1 *= f;
    a.s2 *= f;
    a.s3 *= f;
#endif
    a.ref = cms;
    a.nref = -cms;
    // values above (ref + 16) / log2e raise the reference again; the bound need not be exact (terms overflow only 2^111 above it), so
    // it is kept as its leading 16 bits for the packed comparison of bf16 chunks, always rounded down: neighbours among values
    // below -8192 (bf16) or -1e9 are further apart than that
    const float z = (cms + 16.0f) * 0.6931471805599453f;
    const uint32_t zb = __float_as_uint(fmaf(fabsf(z), -0x1p-22f, z));
    const uint32_t z16 = (zb + (zb >> 31 ? 0xFFFFu : 0u)) >> 16;
    a.thr = BF16 ? (z16 | (z16 << 16)) : zb;
}

__device__ __forceinline__ float pair_max_bf16(uint32_t pm) {  // the larger half of a packed bf16 pair, as fp32
    return fmaxf(__uint_as_float(pm << 16), __uint_as_float(pm & 0xFFFF0000u));
}

// 16-byte vectors of logits into the running sum (four a step).
constexpr int VEC_PER_LANE = 4;
template <bool BF16, int N>
__device__ __forceinline__ void acc_add(const uint4 (&v)[N], Acc& a) {
#if GRAFT_VP_F32X2
    const uint64_t c2 = pack2(kLog2e, kLog2e), r2 = pack2(a.nref, a.nref);
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const uint32_t w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
        if (BF16) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint64_t x2 = pack2(__uint_as_float(w[k] << 16), __uint_as_float(w[k] & 0xFFFF0000u));
                float t0, t1;
                unpack2(fma2(x2, c2, r2), t0, t1);
                const uint64_t e2 = pack2(ex2_approx(t0), ex2_approx(t1));
                if (k & 1)
                    a.a1 = add2(a.a1, e2);
                else
                    a.a0 = add2(a.a0, e2);
            }
        } else {
            float t0, t1, t2, t3;
            unpack2(fma2(pack2(__uint_as_float(w[0]), __uint_as_float(w[1])), c2, r2), t0, t1);
            unpack2(fma2(pack2(__uint_as_float(w[2]), __uint_as_float(w[3])), c2, r2), t2, t3);
            a.a0 = add2(a.a0, pack2(ex2_approx(t0), ex2_approx(t1)));
            a.a1 = add2(a.a1, pack2(ex2_approx(t2), ex2_approx(t3)));
        }
    }
#else
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const uint32_t w[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
        if (BF16) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float lo = __uint_as_float(w[k] << 16), hi = __uint_as_float(w[k] & 0xFFFF0000u);
                const float e0 = ex2_approx(fmaf(lo, kLog2e, a.nref)), e1 = ex2_approx(fmaf(hi, kLog2e, a.nref));
                if (k & 1) {
                    a.s2 += e0;
                    a.s3 += e1;
                } else {
                    a.s0 += e0;
                    a.s1 += e1;
                }
            }
        } else {
            a.s0 += ex2_approx(fmaf(__uint_as_float(w[0]), kLog2e, a.nref));
            a.s1 += ex2_approx(fmaf(__uint_as_float(w[1]), kLog2e, a.nref));
            a.s2 += ex2_approx(fmaf(__uint_as_float(w[2]), kLog2e, a.nref));
            a.s3 += ex2_approx(fmaf(__uint_as_float(w[3]), kLog2e, a.nref));
        }
    }
#endif
}

template <bool BF16>
__device__ __forceinline__ float acc_sum(const Acc& a) {
#if GRAFT_VP_F32X2
    float s0, s1, s2, s3;
    unpack2(a.a0, s0, s1);
    unpack2(a.a1, s2, s3);
    return (s0 + s1) + (s2 + s3);
#else
    return (a.s0 + a.s1) + (a.s2 + a.s3);
#endif
}

// The log-sum-exp of a row from its pieces: C, S with sum_v 2^(z_v c) = S 2^C (c = fp32(log2 e)) and the largest logit.
// The stream accumulates 2^(z c - ref), so (C + log2 S) ln 2 is the log-sum-exp of the logits scaled by
// a = c ln 2 = 1 + 1.3e-8.  To first order that adds (a - 1) E_q[z]; the largest logit stands in for the mean under q (the
// difference is a few units times 1e-8).
__device__ __forceinline__ double vp_lse(double Cd, double Sd, float vmax) {
    const double a_minus_1 = (double)kLog2e * kLn2 - 1.0;
    return (Cd + log2(Sd)) * kLn2 - a_minus_1 * (double)vmax;
}
// Is something wrong with the row's logits (NaN, an infinity, fewer than K finite ones)?
__device__ __forceinline__ bool vp_bad_row(double Sd, uint32_t Vm, int nk, int K) {
    const float vmax = __uint_as_float(bits_from_ord(Vm));
    return !(Sd > 0.0) || !(Sd < 1e300) || Vm == 0u || vmax == INFINITY || vmax == -INFINITY || nk < K;
}
// The outputs of a finished row: its log-sum-exp and the K best keys, a lane a key.  One warp.
__device__ __forceinline__ void vp_write_row(double lse_d, int status, int nk, int K, uint64_t key, int lane,
                                             int32_t* topk_id, float* topk_lp, float* lse, int32_t* row_status) {
    if (lane < K) {
        topk_id[lane] = lane < nk ? (int32_t)key_id(key) : -1;
        topk_lp[lane] = lane < nk ? (float)((double)key_value(key) - lse_d) : 0.f;
    }
    if (lane == 0) {
        *lse = (float)lse_d;
        *row_status = status;
    }
}
// Both of them from a row's pieces.  `internal`: a bounded wait ran out in a CTA that worked on this row.
__device__ __forceinline__ void vp_finalize(double Cd, double Sd, uint32_t Vm, int nk, int K, const uint64_t* keys,
                                            int lane, int32_t* topk_id, float* topk_lp, float* lse,
                                            int32_t* row_status, bool internal) {
    // every lane must use the same bits: the folds that produced C and S are butterflies of fused multiply-adds,
    // which leave the lanes an ulp apart, and log-probabilities of equal logits (and their order) must not depend on
    // the lane that writes them
    Cd = __shfl_sync(0xFFFFFFFFu, Cd, 0);
    Sd = __shfl_sync(0xFFFFFFFFu, Sd, 0);
    Vm = __shfl_sync(0xFFFFFFFFu, Vm, 0);
    const double lse_d = vp_lse(Cd, Sd, __uint_as_float(bits_from_ord(Vm)));
    const int status = (vp_bad_row(Sd, Vm, nk, K) ? GRAFT_ST_BAD_LOGITS : 0) | (internal ? GRAFT_ST_INTERNAL : 0);
    vp_write_row(lse_d, status, nk, K, lane < nk ? keys[lane] : 0ull, lane, topk_id, topk_lp, lse, row_status);
}

}  // namespace

}  // namespace graft

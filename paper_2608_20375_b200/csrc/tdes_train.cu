// TDES training objective, forward and backward in one kernel (Sec. 3.2 "Training", Eq. 7-12).
//
//   f(p,c,d)    = s (P[p] + u_d) . (C[c] + u_d) / sqrt(m)                                       (Eq. 6)
//   L_KL        = mean over groups of KL(softmax_c z_tgt || softmax_c (log q_d(c) + f(p,c,d)))   (Eq. 7-9)
//   L_pair      = mean over pairs of softplus(gamma - f(v+) + f(v-))                             (Eq. 10)
//   L_BCE       = mean over edges of w1 y softplus(-f) + (1 - y) softplus(f)                     (Eq. 11)
//   L           = lambda_KL L_KL + lambda_pair L_pair + lambda_BCE L_BCE                         (Eq. 12)
// and the gradient of L with respect to the table rows P[p], C[c], the depth embeddings u_d and the scale s.
//
// The work is a gather of table rows (m floats each) and a scatter-add of as many gradient rows: memory and atomic
// traffic out of L2, no tensor-core path.  One warp per item (a group of K children, a few pairs or edges): a lane holds
// four consecutive floats of every 128-float chunk of a row, gradient rows go out as 16-byte vector atomics
// (`red.global.add.v4.f32`), gu is accumulated in shared memory and flushed once, losses and the scale's gradient are
// reduced per CTA.  Two kernels: tdes_loss_rows_kernel for m <= 128, tdes_loss_kernel for wider rows.
// The order of the atomic additions is not fixed, so the gradients are reproducible only up to fp32 rounding.
#include <cuda_runtime.h>
#include <math.h>

#include "common.cuh"
#include "internal.h"

namespace graft {
namespace {

constexpr int kTrThreads = 256;
constexpr int kTrWarps = kTrThreads / 32;
constexpr int kTrMaxChunks = 4;  // m <= 512

struct TrainParams {
    const float* P;
    const float* C;
    const float* u;
    float k0;  // s / sqrt(m)
    float inv_sqrt_m;
    int V, L, m, K;
    int n_groups;
    const int32_t* g_parent;
    const int32_t* g_depth;
    const int32_t* g_child;
    const float* g_logq;
    const float* g_ztgt;
    int n_pairs;
    const int32_t* pairs;
    int n_edges;
    const int32_t* edges;
    float gamma, w1;
    float w_kl, w_pair, w_bce;      // lambda / number of items
    float lam_kl, lam_pair, lam_bce;
    double* loss;      // [4], zero at launch
    int32_t* skipped;  // [1] or NULL, zero at launch
    double* acc;       // m <= 128: [5] loss sums, skipped items, arrival counter; zero between calls
    int gu_copies;     // m <= 128: copies of gu in shared memory: one per warp, or one
    int sample;        // m <= 128: look for hot tokens
    float* gP;
    float* gC;
    float* gu;
    float* gs;
};

template <int NCH>
struct Row {
    float4 v[NCH];
};

// row[tok] + u_d, four floats per lane per chunk (zeros past m)
template <int NCH>
__device__ __forceinline__ Row<NCH> load_row_plus_u(const float* table, const float* urow, int tok, int m, int lane) {
    Row<NCH> r;
#pragma unroll
    for (int ch = 0; ch < NCH; ++ch) {
        const int k4 = ch * 32 + lane;
        r.v[ch] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k4 < m / 4) {
            const float4 t = __ldg((const float4*)(table + (size_t)tok * m) + k4);
            const float4 uu = __ldg((const float4*)urow + k4);
            r.v[ch] = make_float4(t.x + uu.x, t.y + uu.y, t.z + uu.z, t.w + uu.w);
        }
    }
    return r;
}
template <int NCH>
__device__ __forceinline__ float warp_dot(const Row<NCH>& a, const Row<NCH>& b) {
    float acc = 0.f;
#pragma unroll
    for (int ch = 0; ch < NCH; ++ch) {
        acc = fmaf(a.v[ch].x, b.v[ch].x, acc);
        acc = fmaf(a.v[ch].y, b.v[ch].y, acc);
        acc = fmaf(a.v[ch].z, b.v[ch].z, acc);
        acc = fmaf(a.v[ch].w, b.v[ch].w, acc);
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, d);
    return acc;
}
// dst_row += coef * r  (global memory, vector atomics)
template <int NCH>
__device__ __forceinline__ void add_row_global(float* dst, int tok, int m, int lane, float coef, const Row<NCH>& r) {
#pragma unroll
    for (int ch = 0; ch < NCH; ++ch) {
        const int k4 = ch * 32 + lane;
        if (k4 < m / 4)
            atomicAdd((float4*)(dst + (size_t)tok * m) + k4,
                      make_float4(coef * r.v[ch].x, coef * r.v[ch].y, coef * r.v[ch].z, coef * r.v[ch].w));
    }
}
// the CTA's copy of gu: row d-1 += coef * (a + b)
template <int NCH>
__device__ __forceinline__ void add_u_shared(float* su, int d, int m, int lane, float coef, const Row<NCH>& a,
                                             const Row<NCH>& b) {
#pragma unroll
    for (int ch = 0; ch < NCH; ++ch) {
        const int k4 = ch * 32 + lane;
        if (k4 < m / 4) {
            float* q = su + (size_t)(d - 1) * m + 4 * k4;
            atomicAdd(q + 0, coef * (a.v[ch].x + b.v[ch].x));
            atomicAdd(q + 1, coef * (a.v[ch].y + b.v[ch].y));
            atomicAdd(q + 2, coef * (a.v[ch].z + b.v[ch].z));
            atomicAdd(q + 3, coef * (a.v[ch].w + b.v[ch].w));
        }
    }
}
__device__ __forceinline__ float softplus_f(float x) { return x > 0.f ? x + log1pf(expf(-x)) : log1pf(expf(x)); }
__device__ __forceinline__ float sigmoid_f(float x) {
    return x >= 0.f ? 1.f / (1.f + expf(-x)) : expf(x) / (1.f + expf(x));
}
__device__ __forceinline__ bool tok_ok(int t, int V) { return t >= 0 && t < V; }

// one edge (p, c, d): returns f; the rows stay in a and b for the backward step
template <int NCH>
__device__ __forceinline__ float edge_forward(const TrainParams& p, int tp, int tc, int d, int lane, Row<NCH>& a,
                                              Row<NCH>& b, float& dot) {
    const float* urow = p.u + (size_t)(d - 1) * p.m;
    a = load_row_plus_u<NCH>(p.P, urow, tp, p.m, lane);
    b = load_row_plus_u<NCH>(p.C, urow, tc, p.m, lane);
    dot = warp_dot<NCH>(a, b);
    return p.k0 * dot;
}
template <int NCH>
__device__ __forceinline__ void edge_backward(const TrainParams& p, float* su, int tp, int tc, int d, int lane, float gf,
                                              const Row<NCH>& a, const Row<NCH>& b, float dot, float& gs) {
    const float coef = gf * p.k0;
    add_row_global<NCH>(p.gP, tp, p.m, lane, coef, b);
    add_row_global<NCH>(p.gC, tc, p.m, lane, coef, a);
    add_u_shared<NCH>(su, d, p.m, lane, coef, a, b);
    gs += gf * dot * p.inv_sqrt_m;
}

template <int NCH>
__global__ void __launch_bounds__(kTrThreads) tdes_loss_kernel(const TrainParams p) {
    extern __shared__ __align__(16) float su[];  // [L][m] this CTA's share of gu
    __shared__ double s_loss[3];
    __shared__ float s_gs;
    __shared__ int s_skip;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool grad = p.gP != nullptr;
    for (int i = threadIdx.x; i < p.L * p.m; i += kTrThreads) su[i] = 0.f;
    if (threadIdx.x < 3) s_loss[threadIdx.x] = 0.0;
    if (threadIdx.x == 0) {
        s_gs = 0.f;
        s_skip = 0;
    }
    __syncthreads();
    const int wid = blockIdx.x * kTrWarps + warp, nw = gridDim.x * kTrWarps;
    double l_kl = 0.0, l_pair = 0.0, l_bce = 0.0;  // this warp's sums (every lane holds the same value)
    float gs = 0.f;
    int skipped = 0;

    // ---- distribution level (Eq. 7-9): lane c owns child c
    for (int g = wid; g < p.n_groups; g += nw) {
        const int tp = p.g_parent[g], d = p.g_depth[g];
        const int tc = lane < p.K ? p.g_child[(size_t)g * p.K + lane] : 0;
        const bool ok = tok_ok(tp, p.V) && d >= 1 && d <= p.L && __all_sync(0xFFFFFFFFu, tok_ok(tc, p.V));
        if (!ok) {
            ++skipped;
            continue;
        }
        const float* urow = p.u + (size_t)(d - 1) * p.m;
        const Row<NCH> a = load_row_plus_u<NCH>(p.P, urow, tp, p.m, lane);
        float dot_c = 0.f;
#pragma unroll 4
        for (int c = 0; c < p.K; ++c) {
            const int t = __shfl_sync(0xFFFFFFFFu, tc, c);
            const Row<NCH> b = load_row_plus_u<NCH>(p.C, urow, t, p.m, lane);
            const float dt = warp_dot<NCH>(a, b);
            if (lane == c) dot_c = dt;
        }
        const float f_c = p.k0 * dot_c;
        const float z = lane < p.K ? p.g_ztgt[(size_t)g * p.K + lane] : -INFINITY;
        const float al = lane < p.K ? p.g_logq[(size_t)g * p.K + lane] + f_c : -INFINITY;
        float zmax = z, amax = al;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            zmax = fmaxf(zmax, __shfl_xor_sync(0xFFFFFFFFu, zmax, o));
            amax = fmaxf(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, o));
        }
        float ez = lane < p.K ? expf(z - zmax) : 0.f, ea = lane < p.K ? expf(al - amax) : 0.f;
        float zsum = ez, asum = ea;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            zsum += __shfl_xor_sync(0xFFFFFFFFu, zsum, o);
            asum += __shfl_xor_sync(0xFFFFFFFFu, asum, o);
        }
        const float pt = ez / zsum, ph = ea / asum;
        float kl = 0.f;
        if (lane < p.K && pt > 0.f) kl = pt * ((z - zmax - logf(zsum)) - (al - amax - logf(asum)));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) kl += __shfl_xor_sync(0xFFFFFFFFu, kl, o);
        l_kl += (double)kl;
        if (grad) {
            const float gf_c = lane < p.K ? p.w_kl * (ph - pt) : 0.f;  // d L / d f_c
            Row<NCH> accP, accU;
#pragma unroll
            for (int ch = 0; ch < NCH; ++ch) accP.v[ch] = accU.v[ch] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
            for (int c = 0; c < p.K; ++c) {
                const int t = __shfl_sync(0xFFFFFFFFu, tc, c);
                const float coef = __shfl_sync(0xFFFFFFFFu, gf_c, c) * p.k0;
                const Row<NCH> b = load_row_plus_u<NCH>(p.C, urow, t, p.m, lane);
                add_row_global<NCH>(p.gC, t, p.m, lane, coef, a);
#pragma unroll
                for (int ch = 0; ch < NCH; ++ch) {
                    accP.v[ch].x = fmaf(coef, b.v[ch].x, accP.v[ch].x);
                    accP.v[ch].y = fmaf(coef, b.v[ch].y, accP.v[ch].y);
                    accP.v[ch].z = fmaf(coef, b.v[ch].z, accP.v[ch].z);
                    accP.v[ch].w = fmaf(coef, b.v[ch].w, accP.v[ch].w);
                    accU.v[ch].x = fmaf(coef, a.v[ch].x + b.v[ch].x, accU.v[ch].x);
                    accU.v[ch].y = fmaf(coef, a.v[ch].y + b.v[ch].y, accU.v[ch].y);
                    accU.v[ch].z = fmaf(coef, a.v[ch].z + b.v[ch].z, accU.v[ch].z);
                    accU.v[ch].w = fmaf(coef, a.v[ch].w + b.v[ch].w, accU.v[ch].w);
                }
            }
            add_row_global<NCH>(p.gP, tp, p.m, lane, 1.f, accP);
            Row<NCH> zero;
#pragma unroll
            for (int ch = 0; ch < NCH; ++ch) zero.v[ch] = make_float4(0.f, 0.f, 0.f, 0.f);
            add_u_shared<NCH>(su, d, p.m, lane, 1.f, accU, zero);
            float gsc = gf_c * dot_c * p.inv_sqrt_m;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) gsc += __shfl_xor_sync(0xFFFFFFFFu, gsc, o);
            gs += gsc;
        }
    }
    // ---- pairwise level (Eq. 10)
    for (int i = wid; i < p.n_pairs; i += nw) {
        const int32_t* q = p.pairs + (size_t)i * 6;
        const int p1 = q[0], c1 = q[1], d1 = q[2], p2 = q[3], c2 = q[4], d2 = q[5];
        if (!(tok_ok(p1, p.V) && tok_ok(c1, p.V) && tok_ok(p2, p.V) && tok_ok(c2, p.V) && d1 >= 1 && d1 <= p.L &&
              d2 >= 1 && d2 <= p.L)) {
            ++skipped;
            continue;
        }
        Row<NCH> a1, b1, a2, b2;
        float dot1, dot2;
        const float f1 = edge_forward<NCH>(p, p1, c1, d1, lane, a1, b1, dot1);
        const float f2 = edge_forward<NCH>(p, p2, c2, d2, lane, a2, b2, dot2);
        const float x = p.gamma - f1 + f2;
        l_pair += (double)softplus_f(x);
        if (grad) {
            const float gx = p.w_pair * sigmoid_f(x);
            edge_backward<NCH>(p, su, p1, c1, d1, lane, -gx, a1, b1, dot1, gs);
            edge_backward<NCH>(p, su, p2, c2, d2, lane, gx, a2, b2, dot2, gs);
        }
    }
    // ---- edge level (Eq. 11)
    for (int i = wid; i < p.n_edges; i += nw) {
        const int32_t* e = p.edges + (size_t)i * 4;
        const int tp = e[0], tc = e[1], d = e[2];
        const float y = e[3] ? 1.f : 0.f;
        if (!(tok_ok(tp, p.V) && tok_ok(tc, p.V) && d >= 1 && d <= p.L)) {
            ++skipped;
            continue;
        }
        Row<NCH> a, b;
        float dot;
        const float f = edge_forward<NCH>(p, tp, tc, d, lane, a, b, dot);
        l_bce += (double)(p.w1 * y * softplus_f(-f) + (1.f - y) * softplus_f(f));
        if (grad) {
            const float gf = p.w_bce * (-p.w1 * y * sigmoid_f(-f) + (1.f - y) * sigmoid_f(f));
            edge_backward<NCH>(p, su, tp, tc, d, lane, gf, a, b, dot, gs);
        }
    }
    // ---- per-CTA reduction, then one round of global atomics
    if (lane == 0) {
        atomicAdd(&s_loss[0], l_kl);
        atomicAdd(&s_loss[1], l_pair);
        atomicAdd(&s_loss[2], l_bce);
        atomicAdd(&s_gs, gs);
        if (skipped) atomicAdd(&s_skip, skipped);
    }
    __syncthreads();
    if (grad)
        for (int i = threadIdx.x; i < p.L * p.m; i += kTrThreads)
            if (su[i] != 0.f) atomicAdd(p.gu + i, su[i]);
    if (threadIdx.x == 0) {
        const double kl = s_loss[0] / (double)(p.n_groups > 0 ? p.n_groups : 1);
        const double pr = s_loss[1] / (double)(p.n_pairs > 0 ? p.n_pairs : 1);
        const double bc = s_loss[2] / (double)(p.n_edges > 0 ? p.n_edges : 1);
        atomicAdd(p.loss + 0, kl);
        atomicAdd(p.loss + 1, pr);
        atomicAdd(p.loss + 2, bc);
        atomicAdd(p.loss + 3, (double)p.lam_kl * kl + (double)p.lam_pair * pr + (double)p.lam_bce * bc);
        if (grad && s_gs != 0.f) atomicAdd(p.gs, s_gs);
        if (p.skipped && s_skip) atomicAdd(p.skipped, s_skip);
    }
}

// ---- m <= 128: one float4 of a row per lane -----------------------------------------------------------------------------
// What bounded the kernel above at these widths was its own instructions (287 M of them at the shapes below, L1 83 %
// busy, L2 31 %), not the atomics: shared-memory atomics for gu (compare-and-swap loops), five shuffles a dot product,
// the replacement of cached rows, and the children's rows read twice.  Here
//   * a group's children stay in registers between the forward and the backward step (KC rows at most), all their
//     loads in flight together; pairs go four at a time and edges eight;
//   * dot products are summed across the warp together (31 shuffles for 32 of them), which leaves dot i in the lanes
//     that own item i: the transcendental functions are worked out once per item, not once per lane;
//   * every warp adds into a copy of gu of its own (a plain load, add and store);
//   * the few hottest tokens' gradient rows (additions to one row serialise in L2) are picked once per CTA from a sample of
//     the tokens, and every warp keeps its sums of them in shared memory; everything else is a 16-byte vector atomic.
// Measured (B200, V = 151,936, m = 128, L = 16, 32,768 groups of 32, 131,072 pairs, 262,144 edges): 323 us (420 us by the
// one-item-a-warp kernel with replaced cached rows; 500 of 8, 2000 and 4000: 16.6 and 19.6 us).  What bounds it now: the vector atomics -- a million rows spread
// evenly take 96 us whether from 8 or from 32 warps an SM or as bulk reductions from shared memory, a million with the
// Zipf(1.1) tokens of these traces 790 us, without their eight hottest 152 us -- and, in front of them in the same
// queue, 1.6 million row loads (138 us for the losses alone).  One copy of gu with atomics instead of one a warp leaves
// more L1 for the rows but costs more than it saves (360 us).
constexpr int kTsThreads = 384;
constexpr int kTsWarps = kTsThreads / 32;
constexpr int kTsSample = 256;
// References to rows from which looking for hot ones is worth its time (10 us: two rounds of loads, 256 x 256 compares).
// With and without: 41 thousand references 26.8 and 22.8 us, 65 thousand 34.0 and 26.7, 74 thousand 33.0 and 35.0, 164
// thousand 47.4 and 61.0.
constexpr int kTsSampleMin = 65536;

constexpr int kTsSlots = 8;  // hot rows per table
struct __align__(16) TrainHot {
    int tok[2][kTsSlots];
};

__device__ __forceinline__ float2 lo2(const float4& v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(const float4& v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float4 add4(const float4& a, const float4& b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float4 sub4(const float4& a, const float4& b) { return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w); }
__device__ __forceinline__ float4 mul4(float c, const float4& a) { return make_float4(c * a.x, c * a.y, c * a.z, c * a.w); }
__device__ __forceinline__ float4 fma4(float c, const float4& a, const float4& b) {
    const float2 cc = make_float2(c, c), l = __ffma2_rn(cc, lo2(a), lo2(b)), h = __ffma2_rn(cc, hi2(a), hi2(b));
    return make_float4(l.x, l.y, h.x, h.y);
}
__device__ __forceinline__ float dot4(const float4& a, const float4& b) {
    const float2 s = __ffma2_rn(lo2(a), lo2(b), __fmul2_rn(hi2(a), hi2(b)));
    return s.x + s.y;
}
// Sums of N values over the warp (N = 8, 16, 32), each lane's partial sums in v: value i is returned to the lanes with
// (lane >> (5 - log2 N)) == i.
template <int N>
__device__ __forceinline__ float warp_sums(float (&v)[N], int lane) {
    int mask = 16;
#pragma unroll
    for (int n = N / 2; n >= 1; n /= 2, mask >>= 1) {
        const bool up = (lane & mask) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float give = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
            v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, mask);
        }
    }
    float s = v[0];
#pragma unroll
    for (; mask >= 1; mask >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, mask);
    return s;
}
__device__ __forceinline__ float warp_sum(float s) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    return s;
}
__device__ __forceinline__ int hot_slot(const TrainHot& h, int t, int tok) {
    const int4 x = *(const int4*)h.tok[t], y = *((const int4*)h.tok[t] + 1);
    int s = tok == x.x ? 0 : -1;
    s = tok == x.y ? 1 : s;
    s = tok == x.z ? 2 : s;
    s = tok == x.w ? 3 : s;
    s = tok == y.x ? 4 : s;
    s = tok == y.y ? 5 : s;
    s = tok == y.z ? 6 : s;
    return tok == y.w ? 7 : s;
}
__device__ __forceinline__ void smem_add4(float4* q, const float4& v) { *q = add4(*q, v); }

// What the warps of a CTA share, and this warp's place in it.
struct TrainCtx {
    const float* u;   // [L][m] shared copy of the depth embeddings
    float* gu;        // [L][m] this warp's sums (or the CTA's, with atomics)
    float4* hot;      // [2][kTsSlots][32] this warp's sums of the hot rows
    bool gu_shared, on;  // on: this lane holds a part of a row
    int lane, m;
};
// FULL: m = 128, every lane holds a part of a row
template <bool FULL>
__device__ __forceinline__ float4* ctx_at(const TrainCtx& c, const float* table, int tok) {
    return (float4*)(table + (size_t)tok * (FULL ? 128 : c.m)) + c.lane;
}
template <bool FULL>
__device__ __forceinline__ void ctx_add_row(const TrainParams& p, const TrainCtx& c, int t, int tok, int slot, const float4& v) {
    if (slot >= 0)  // (uniform)
        smem_add4(c.hot + (t * kTsSlots + slot) * 32 + c.lane, v);
    else if (FULL || c.on)
        atomicAdd(ctx_at<FULL>(c, t == 0 ? p.gP : p.gC, tok), v);
}
template <bool FULL>
__device__ __forceinline__ void ctx_add_u(const TrainCtx& c, int d, const float4& v) {
    if (!FULL && !c.on) return;
    float4* q = ctx_at<FULL>(c, c.gu, d - 1);
    if (!c.gu_shared) {
        smem_add4(q, v);
    } else {
        float* f = (float*)q;
        atomicAdd(f + 0, v.x);
        atomicAdd(f + 1, v.y);
        atomicAdd(f + 2, v.z);
        atomicAdd(f + 3, v.w);
    }
}
template <bool FULL>
__device__ __forceinline__ float4 ctx_load(const TrainCtx& c, const float* table, int tok) {
    return FULL || c.on ? __ldg(ctx_at<FULL>(c, table, tok)) : make_float4(0.f, 0.f, 0.f, 0.f);
}
template <bool FULL>
__device__ __forceinline__ float4 ctx_u(const TrainCtx& c, int d) {
    return FULL || c.on ? *ctx_at<FULL>(c, c.u, d - 1) : make_float4(0.f, 0.f, 0.f, 0.f);
}

// The i-th of kTsSample tokens spread evenly over the references to a table (0: P, 1: C), or -1.
__device__ __forceinline__ int train_sample(const TrainParams& p, int t, int i) {
    const long long ng = t == 0 ? p.n_groups : (long long)p.n_groups * p.K, np = 2ll * p.n_pairs;
    const long long n = ng + np + p.n_edges;
    long long at = n * i / kTsSample;
    int tok;
    if (at < ng) {
        tok = t == 0 ? p.g_parent[at] : p.g_child[at];
    } else if ((at -= ng) < np) {
        tok = p.pairs[(at >> 1) * 6 + (at & 1) * 3 + t];
    } else {
        at -= np;
        tok = at < p.n_edges ? p.edges[at * 4 + t] : -1;
    }
    return tok >= 0 && tok < p.V ? tok : -1;
}

// The work is one list -- groups, blocks of eight pairs, blocks of eight edges -- dealt to the warps in turn: the first of a
// kind, with `ahead` entries of other kinds ahead of it, that warp wid of nw gets.  (Dealt kind by kind, the first warps got
// one of each, one after the other, while the rest had nothing: half of a small call's time.)
__device__ __forceinline__ int first_block(int wid, long long ahead, int nw) {
    const int r = wid - (int)(ahead % nw);
    return r < 0 ? r + nw : r;
}

// KC: children held in registers, a multiple of 8 (K <= KC)
template <int KC, bool FULL>
__global__ void __launch_bounds__(kTsThreads, 1) tdes_loss_rows_kernel(const TrainParams p) {
    extern __shared__ __align__(16) float smem_f[];
    __shared__ TrainHot s_hot;
    __shared__ int s_tok[2][kTsSample], s_cnt[2][kTsSample];
    __shared__ double s_loss[3];
    __shared__ float s_gs;
    __shared__ int s_skip;
    __shared__ bool s_last;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, Lm = p.L * p.m;
    const bool grad = p.gP != nullptr;
    // [L][m] u, then the copies of gu, then the warps' hot rows
    float* s_gu = smem_f + Lm;
    float* s_rows = s_gu + (size_t)Lm * p.gu_copies;
    TrainCtx c;
    c.u = smem_f;
    c.gu_shared = p.gu_copies == 1;
    c.gu = s_gu + (c.gu_shared ? 0 : (size_t)warp * Lm);
    c.hot = (float4*)(s_rows + (size_t)warp * 2 * kTsSlots * 128);
    c.on = lane < p.m / 4;
    c.lane = lane;
    c.m = p.m;
    for (int i = tid; i < Lm; i += kTsThreads) smem_f[i] = p.u[i];
    if (grad) {
        for (int i = tid; i < Lm / 4 * p.gu_copies; i += kTsThreads) ((float4*)s_gu)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (p.sample)
            for (int i = tid; i < kTsWarps * 2 * kTsSlots * 32; i += kTsThreads) ((float4*)s_rows)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (tid < 3) s_loss[tid] = 0.0;
    if (tid == 0) {
        s_gs = 0.f;
        s_skip = 0;
    }
    if (tid < 2 * kTsSlots) s_hot.tok[tid / kTsSlots][tid % kTsSlots] = -1;
    if (grad && p.sample) {  // (uniform) the tokens met most often in the sample get the slots
        for (int i = tid; i < 2 * kTsSample; i += kTsThreads) s_tok[i / kTsSample][i % kTsSample] = train_sample(p, i / kTsSample, i % kTsSample);
        __syncthreads();
        for (int i = tid; i < 2 * kTsSample; i += kTsThreads) {
            const int t = i / kTsSample, me = i % kTsSample, tok = s_tok[t][me];
            int n = 0, first = me;
            for (int j = kTsSample - 1; j >= 0; --j)
                if (s_tok[t][j] == tok) {
                    ++n;
                    first = j;
                }
            s_cnt[t][me] = tok >= 0 && first == me && n >= 2 ? n * kTsSample + (kTsSample - 1 - me) : 0;  // (distinct, 0: none)
        }
        __syncthreads();
        for (int i = tid; i < 2 * kTsSample; i += kTsThreads) {
            const int t = i / kTsSample, me = i % kTsSample, mine = s_cnt[t][me];
            if (mine > 0) {
                int rank = 0;
                for (int j = 0; j < kTsSample; ++j) rank += s_cnt[t][j] > mine ? 1 : 0;
                if (rank < kTsSlots) s_hot.tok[t][rank] = s_tok[t][me];
            }
        }
    }
    __syncthreads();
    const TrainHot& hot = s_hot;
    const int wid = blockIdx.x * kTsWarps + warp, nw = gridDim.x * kTsWarps;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    double l_kl = 0.0, l_pair = 0.0, l_bce = 0.0;  // per lane; summed at the end
    float gs = 0.f;
    int skipped = 0;

    // ---- distribution level (Eq. 7-9): lane i owns child i; the next group's ids are on their way while one is worked on
    int n_tp = 0, n_d = 0, n_tc = 0;
    float n_z = 0.f, n_lq = 0.f;
    auto fetch = [&](int g) {
        if (g >= p.n_groups) return;
        n_tp = p.g_parent[g];
        n_d = p.g_depth[g];
        const size_t at = (size_t)g * p.K + lane;
        n_tc = lane < p.K ? p.g_child[at] : 0;
        n_z = lane < p.K ? p.g_ztgt[at] : -INFINITY;
        n_lq = lane < p.K ? p.g_logq[at] : -INFINITY;
    };
    fetch(wid);
    for (int g = wid; g < p.n_groups; g += nw) {
        const int tp = n_tp, d = n_d, tc = n_tc;
        const float z = n_z, lq = n_lq;
        fetch(g + nw);
        if (!(tok_ok(tp, p.V) && d >= 1 && d <= p.L && __all_sync(0xFFFFFFFFu, tok_ok(tc, p.V)))) {
            skipped += lane == 0 ? 1 : 0;
            continue;
        }
        const float4 prow = ctx_load<FULL>(c, p.P, tp);
        float4 rows[KC];
#pragma unroll
        for (int i = 0; i < KC; ++i) {
            const int t = __shfl_sync(0xFFFFFFFFu, tc, i);
            rows[i] = i < p.K ? ctx_load<FULL>(c, p.C, t) : zero4;
        }
        const float4 u = ctx_u<FULL>(c, d), a = add4(prow, u);
        // f = k0 (a . C + a . u)
        const float au = dot4(a, u);
        float part[KC];
#pragma unroll
        for (int i = 0; i < KC; ++i) part[i] = au + dot4(a, rows[i]);
        const float dots = warp_sums<KC>(part, lane);
        constexpr int SH = KC == 32 ? 0 : (KC == 16 ? 1 : 2);
        const float dot_c = SH == 0 ? dots : __shfl_sync(0xFFFFFFFFu, dots, (lane << SH) & 31);
        const float al = lane < p.K ? lq + p.k0 * dot_c : -INFINITY;
        float zmax = z, amax = al;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            zmax = fmaxf(zmax, __shfl_xor_sync(0xFFFFFFFFu, zmax, o));
            amax = fmaxf(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, o));
        }
        const float ez = lane < p.K ? expf(z - zmax) : 0.f, ea = lane < p.K ? expf(al - amax) : 0.f;
        const float zsum = warp_sum(ez), asum = warp_sum(ea);
        const float pt = ez / zsum, ph = ea / asum;
        if (lane < p.K && pt > 0.f) l_kl += (double)(pt * ((z - zmax - logf(zsum)) - (al - amax - logf(asum))));
        if (!grad) continue;
        const float gf = lane < p.K ? p.w_kl * (ph - pt) : 0.f;  // d L / d f
        if (lane < p.K) gs += gf * dot_c * p.inv_sqrt_m;
        const float coef = gf * p.k0;
        const int slot = lane < p.K ? hot_slot(hot, 1, tc) : -1;
        const uint32_t hots = __ballot_sync(0xFFFFFFFFu, slot >= 0);
        // sum_c coef_c (C_c + u) = sum_c coef_c C_c: the coefficients, differences of two distributions, add up to 0
        float4 acc = zero4;
#pragma unroll
        for (int i = 0; i < KC; ++i) {
            if (i < p.K) {
                const float cf = __shfl_sync(0xFFFFFFFFu, coef, i);
                const int t = __shfl_sync(0xFFFFFFFFu, tc, i);
                acc = fma4(cf, rows[i], acc);
                if (!((hots >> i) & 1u) && (FULL || c.on)) atomicAdd(ctx_at<FULL>(c, p.gC, t), mul4(cf, a));
            }
        }
        for (uint32_t left = hots; left != 0u; left &= left - 1u) {  // (uniform)
            const int i = __ffs(left) - 1;
            smem_add4(c.hot + (kTsSlots + __shfl_sync(0xFFFFFFFFu, slot, i)) * 32 + lane, mul4(__shfl_sync(0xFFFFFFFFu, coef, i), a));
        }
        ctx_add_row<FULL>(p, c, 0, tp, hot_slot(hot, 0, tp), acc);
        ctx_add_u<FULL>(c, d, acc);
    }
    // ---- pairwise level (Eq. 10): blocks of eight pairs, four at a time; lanes 0-7 hold the block's ids
    for (int b0 = first_block(wid, p.n_groups, nw) * 8; b0 < p.n_pairs; b0 += nw * 8) {
        int id[6] = {0, 0, 1, 0, 0, 1};
        bool ok = false;
        if (lane < 8 && b0 + lane < p.n_pairs) {
            const int32_t* q = p.pairs + (size_t)(b0 + lane) * 6;
#pragma unroll
            for (int k = 0; k < 6; ++k) id[k] = q[k];
            ok = tok_ok(id[0], p.V) && tok_ok(id[1], p.V) && tok_ok(id[3], p.V) && tok_ok(id[4], p.V) && id[2] >= 1 &&
                 id[2] <= p.L && id[5] >= 1 && id[5] <= p.L;
            if (!ok) {
                ++skipped;
                id[0] = id[1] = id[3] = id[4] = 0;
                id[2] = id[5] = 1;
            }
        }
        const uint32_t oks = __ballot_sync(0xFFFFFFFFu, ok);
        const int sp1 = hot_slot(hot, 0, id[0]), sc1 = hot_slot(hot, 1, id[1]), sp2 = hot_slot(hot, 0, id[3]), sc2 = hot_slot(hot, 1, id[4]);
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            if (((oks >> (4 * h)) & 15u) == 0u) continue;  // (uniform)
            float4 a1[4], b1[4], a2[4], b2[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int s = 4 * h + i;
                a1[i] = ctx_load<FULL>(c, p.P, __shfl_sync(0xFFFFFFFFu, id[0], s));
                b1[i] = ctx_load<FULL>(c, p.C, __shfl_sync(0xFFFFFFFFu, id[1], s));
                a2[i] = ctx_load<FULL>(c, p.P, __shfl_sync(0xFFFFFFFFu, id[3], s));
                b2[i] = ctx_load<FULL>(c, p.C, __shfl_sync(0xFFFFFFFFu, id[4], s));
            }
            float part[8];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int s = 4 * h + i, d1 = __shfl_sync(0xFFFFFFFFu, id[2], s), d2 = __shfl_sync(0xFFFFFFFFu, id[5], s);
                const float4 u1 = ctx_u<FULL>(c, d1);
                const float4 u2 = ctx_u<FULL>(c, d2);
                a1[i] = add4(a1[i], u1);
                b1[i] = add4(b1[i], u1);
                a2[i] = add4(a2[i], u2);
                b2[i] = add4(b2[i], u2);
                part[2 * i] = dot4(a1[i], b1[i]);
                part[2 * i + 1] = dot4(a2[i], b2[i]);
            }
            const float dot = warp_sums<8>(part, lane);  // lanes 8 i .. 8 i + 3: v+ of pair i, the next four: v-
            const float other = __shfl_xor_sync(0xFFFFFFFFu, dot, 4);
            const float dp = (lane & 4) ? other : dot, dm = (lane & 4) ? dot : other;
            const float x = p.gamma - p.k0 * dp + p.k0 * dm;
            const bool mine = (oks >> (4 * h + (lane >> 3))) & 1u;
            const float gx = mine && grad ? p.w_pair * sigmoid_f(x) : 0.f;
            if (mine && (lane & 7) == 0) {
                l_pair += (double)softplus_f(x);
                gs += gx * (dm - dp) * p.inv_sqrt_m;
            }
            if (!grad) continue;
            const float coef = gx * p.k0;  // of v-; v+ gets its negative
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int s = 4 * h + i;
                if (!((oks >> s) & 1u)) continue;  // (uniform)
                const float cf = __shfl_sync(0xFFFFFFFFu, coef, 8 * i);
                const int p1 = __shfl_sync(0xFFFFFFFFu, id[0], s), c1 = __shfl_sync(0xFFFFFFFFu, id[1], s), d1 = __shfl_sync(0xFFFFFFFFu, id[2], s);
                const int p2 = __shfl_sync(0xFFFFFFFFu, id[3], s), c2 = __shfl_sync(0xFFFFFFFFu, id[4], s), d2 = __shfl_sync(0xFFFFFFFFu, id[5], s);
                const int h1 = __shfl_sync(0xFFFFFFFFu, sp1, s), h2 = __shfl_sync(0xFFFFFFFFu, sc1, s);
                if (p1 == p2) {  // (uniform; an alternative keeps the pair's parent or its child: one addition for both)
                    ctx_add_row<FULL>(p, c, 0, p1, h1, mul4(cf, sub4(b2[i], b1[i])));
                } else {
                    ctx_add_row<FULL>(p, c, 0, p1, h1, mul4(-cf, b1[i]));
                    ctx_add_row<FULL>(p, c, 0, p2, __shfl_sync(0xFFFFFFFFu, sp2, s), mul4(cf, b2[i]));
                }
                if (c1 == c2) {
                    ctx_add_row<FULL>(p, c, 1, c1, h2, mul4(cf, sub4(a2[i], a1[i])));
                } else {
                    ctx_add_row<FULL>(p, c, 1, c1, h2, mul4(-cf, a1[i]));
                    ctx_add_row<FULL>(p, c, 1, c2, __shfl_sync(0xFFFFFFFFu, sc2, s), mul4(cf, a2[i]));
                }
                const float4 s1 = add4(a1[i], b1[i]), s2 = add4(a2[i], b2[i]);
                if (d1 == d2) {
                    ctx_add_u<FULL>(c, d1, mul4(cf, sub4(s2, s1)));
                } else {
                    ctx_add_u<FULL>(c, d1, mul4(-cf, s1));
                    ctx_add_u<FULL>(c, d2, mul4(cf, s2));
                }
            }
        }
    }
    // ---- edge level (Eq. 11): eight edges at a time; lanes 0-7 hold their ids
    for (int b0 = first_block(wid, p.n_groups + (p.n_pairs + 7ll) / 8, nw) * 8; b0 < p.n_edges; b0 += nw * 8) {
        int tp = 0, tc = 0, d = 1, y = 0;
        bool ok = false;
        if (lane < 8 && b0 + lane < p.n_edges) {
            const int32_t* e = p.edges + (size_t)(b0 + lane) * 4;
            tp = e[0], tc = e[1], d = e[2], y = e[3];
            ok = tok_ok(tp, p.V) && tok_ok(tc, p.V) && d >= 1 && d <= p.L;
            if (!ok) {
                ++skipped;
                tp = tc = 0;
                d = 1;
            }
        }
        const uint32_t oks = __ballot_sync(0xFFFFFFFFu, ok);
        const int sp = hot_slot(hot, 0, tp), sc = hot_slot(hot, 1, tc);
        float4 a[8], b[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            a[i] = ctx_load<FULL>(c, p.P, __shfl_sync(0xFFFFFFFFu, tp, i));
            b[i] = ctx_load<FULL>(c, p.C, __shfl_sync(0xFFFFFFFFu, tc, i));
        }
        float part[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int dd = __shfl_sync(0xFFFFFFFFu, d, i);
            const float4 u = ctx_u<FULL>(c, dd);
            a[i] = add4(a[i], u);
            b[i] = add4(b[i], u);
            part[i] = dot4(a[i], b[i]);
        }
        const float dot = warp_sums<8>(part, lane);  // lanes 4 i .. 4 i + 3: edge i
        const float f = p.k0 * dot, yy = __shfl_sync(0xFFFFFFFFu, y, lane >> 2) ? 1.f : 0.f;
        const bool mine = (oks >> (lane >> 2)) & 1u;
        const float gf = mine && grad ? p.w_bce * (-p.w1 * yy * sigmoid_f(-f) + (1.f - yy) * sigmoid_f(f)) : 0.f;
        if (mine && (lane & 3) == 0) {
            l_bce += (double)(p.w1 * yy * softplus_f(-f) + (1.f - yy) * softplus_f(f));
            gs += gf * dot * p.inv_sqrt_m;
        }
        if (!grad) continue;
        const float coef = gf * p.k0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (!((oks >> i) & 1u)) continue;  // (uniform)
            const float cf = __shfl_sync(0xFFFFFFFFu, coef, 4 * i);
            ctx_add_row<FULL>(p, c, 0, __shfl_sync(0xFFFFFFFFu, tp, i), __shfl_sync(0xFFFFFFFFu, sp, i), mul4(cf, b[i]));
            ctx_add_row<FULL>(p, c, 1, __shfl_sync(0xFFFFFFFFu, tc, i), __shfl_sync(0xFFFFFFFFu, sc, i), mul4(cf, a[i]));
            ctx_add_u<FULL>(c, __shfl_sync(0xFFFFFFFFu, d, i), mul4(cf, add4(a[i], b[i])));
        }
    }
    // ---- per-CTA sums, then one round of global atomics
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        l_kl += __shfl_xor_sync(0xFFFFFFFFu, l_kl, o);
        l_pair += __shfl_xor_sync(0xFFFFFFFFu, l_pair, o);
        l_bce += __shfl_xor_sync(0xFFFFFFFFu, l_bce, o);
    }
    gs = warp_sum(gs);
    skipped = __reduce_add_sync(0xFFFFFFFFu, skipped);
    if (lane == 0) {
        atomicAdd(&s_loss[0], l_kl);
        atomicAdd(&s_loss[1], l_pair);
        atomicAdd(&s_loss[2], l_bce);
        atomicAdd(&s_gs, gs);
        if (skipped) atomicAdd(&s_skip, skipped);
    }
    __syncthreads();
    if (grad) {
        for (int i = tid; i < Lm; i += kTsThreads) {
            float v = s_gu[i];
            for (int w = 1; w < p.gu_copies; ++w) v += s_gu[(size_t)w * Lm + i];
            if (v != 0.f) atomicAdd(p.gu + i, v);
        }
        for (int i = tid; p.sample && i < 2 * kTsSlots * 32; i += kTsThreads) {
            const int r = i >> 5, l = i & 31, tok = s_hot.tok[r / kTsSlots][r % kTsSlots];
            if (tok < 0 || l >= p.m / 4) continue;
            float4 v = zero4;
            for (int w = 0; w < kTsWarps; ++w) v = add4(v, ((const float4*)s_rows)[(size_t)w * 2 * kTsSlots * 32 + i]);
            atomicAdd((float4*)((r < kTsSlots ? p.gP : p.gC) + (size_t)tok * p.m) + l, v);
        }
    }
    if (tid == 0) {
        atomicAdd(p.acc + 0, s_loss[0]);
        atomicAdd(p.acc + 1, s_loss[1]);
        atomicAdd(p.acc + 2, s_loss[2]);
        if (s_skip) atomicAdd((int*)(p.acc + 3), s_skip);
        if (grad && s_gs != 0.f) atomicAdd(p.gs, s_gs);
        __threadfence();
        s_last = atomicAdd((unsigned int*)(p.acc + 4), 1u) == gridDim.x - 1;
        if (s_last) {  // the CTA that finishes last writes the losses and clears the sums for the next call
            __threadfence();
            const double kl = __ldcg(p.acc + 0) / (double)(p.n_groups > 0 ? p.n_groups : 1);
            const double pr = __ldcg(p.acc + 1) / (double)(p.n_pairs > 0 ? p.n_pairs : 1);
            const double bc = __ldcg(p.acc + 2) / (double)(p.n_edges > 0 ? p.n_edges : 1);
            p.loss[0] = kl;
            p.loss[1] = pr;
            p.loss[2] = bc;
            p.loss[3] = (double)p.lam_kl * kl + (double)p.lam_pair * pr + (double)p.lam_bce * bc;
            if (p.skipped) *p.skipped = __ldcg((const int*)(p.acc + 3));
            for (int i = 0; i < 5; ++i) p.acc[i] = 0.0;
        }
    }
}

}  // namespace

// One copy of gu a warp where they fit beside the rest (the usual L m = 2048), else one with atomics.
static int rows_gu_copies(const graft_config& cfg) { return cfg.L * cfg.m <= 2048 ? kTsWarps : 1; }
static size_t tdes_loss_smem(const graft_config& cfg) {
    const size_t lm = (size_t)((cfg.L * cfg.m + 3) & ~3);
    if (cfg.m > 128) return lm * sizeof(float);  // gu
    return (lm * (1 + rows_gu_copies(cfg)) + (size_t)kTsWarps * 2 * kTsSlots * 128) * sizeof(float);
}
static void (*rows_kernel(const graft_config& cfg))(const TrainParams) {
    if (cfg.m == 128) return cfg.K <= 8 ? tdes_loss_rows_kernel<8, true> : (cfg.K <= 16 ? tdes_loss_rows_kernel<16, true> : tdes_loss_rows_kernel<32, true>);
    return cfg.K <= 8 ? tdes_loss_rows_kernel<8, false> : (cfg.K <= 16 ? tdes_loss_rows_kernel<16, false> : tdes_loss_rows_kernel<32, false>);
}

cudaError_t tdes_loss_launch(graft_ctx* ctx, const graft_tdes_traces* tr, const graft_tdes_loss_config* lc,
                             double* d_loss, int32_t* d_skipped, float* d_gP, float* d_gC, float* d_gu, float* d_gs,
                             cudaStream_t st) {
    const graft_config& cfg = ctx->cfg;
    TrainParams p;
    p.P = ctx->d_P;
    p.C = ctx->d_C;
    p.u = ctx->d_u;
    p.k0 = ctx->tdes_s / sqrtf((float)cfg.m);
    p.inv_sqrt_m = 1.0f / sqrtf((float)cfg.m);
    p.V = cfg.V;
    p.L = cfg.L;
    p.m = cfg.m;
    p.K = cfg.K;
    p.n_groups = tr->n_groups;
    p.g_parent = tr->d_g_parent;
    p.g_depth = tr->d_g_depth;
    p.g_child = tr->d_g_child;
    p.g_logq = tr->d_g_logq;
    p.g_ztgt = tr->d_g_ztgt;
    p.n_pairs = tr->n_pairs;
    p.pairs = tr->d_pairs;
    p.n_edges = tr->n_edges;
    p.edges = tr->d_edges;
    p.gamma = lc->gamma;
    p.w1 = lc->w1;
    p.lam_kl = lc->lambda_kl;
    p.lam_pair = lc->lambda_pair;
    p.lam_bce = lc->lambda_bce;
    p.w_kl = tr->n_groups > 0 ? lc->lambda_kl / (float)tr->n_groups : 0.f;
    p.w_pair = tr->n_pairs > 0 ? lc->lambda_pair / (float)tr->n_pairs : 0.f;
    p.w_bce = tr->n_edges > 0 ? lc->lambda_bce / (float)tr->n_edges : 0.f;
    p.loss = d_loss;
    p.skipped = d_skipped;
    p.gP = d_gP;
    p.gC = d_gC;
    p.gu = d_gu;
    p.gs = d_gs;
    const long long items = (long long)tr->n_groups + tr->n_pairs + tr->n_edges;
    const size_t smem = tdes_loss_smem(cfg);
    if (cfg.m <= 128 && items > 0) {
        p.acc = ctx->w_loss;
        p.gu_copies = rows_gu_copies(cfg);
        p.sample = (long long)tr->n_groups * (cfg.K + 1) + 4ll * tr->n_pairs + 2ll * tr->n_edges >= kTsSampleMin;
        // a warp takes a group, eight pairs or eight edges at a time
        const long long work = (long long)tr->n_groups + (tr->n_pairs + 7ll) / 8 + (tr->n_edges + 7ll) / 8;
        long long grid = (work + kTsWarps - 1) / kTsWarps;
        if (grid > ctx->num_sms) grid = ctx->num_sms;
        rows_kernel(cfg)<<<(int)grid, kTsThreads, smem, st>>>(p);
        ctx->launches += 1;
        return cudaGetLastError();
    }
    cudaError_t e = cudaMemsetAsync(d_loss, 0, 4 * sizeof(double), st);
    if (e != cudaSuccess) return e;
    if (d_skipped) {
        e = cudaMemsetAsync(d_skipped, 0, sizeof(int32_t), st);
        if (e != cudaSuccess) return e;
    }
    if (items == 0) return cudaSuccess;
    long long grid = (items + kTrWarps - 1) / kTrWarps;
    const long long cap = (long long)ctx->num_sms * 4;
    if (grid > cap) grid = cap;
    if (cfg.m <= 256)
        tdes_loss_kernel<2><<<(int)grid, kTrThreads, smem, st>>>(p);
    else
        tdes_loss_kernel<kTrMaxChunks><<<(int)grid, kTrThreads, smem, st>>>(p);
    ctx->launches += 1;
    return cudaGetLastError();
}

cudaError_t tdes_loss_configure(const graft_config& cfg) {
    const size_t smem = tdes_loss_smem(cfg);
    if (cfg.m <= 128) return allow_smem((const void*)rows_kernel(cfg), smem);
    return allow_smem((const void*)(cfg.m <= 256 ? tdes_loss_kernel<2> : tdes_loss_kernel<kTrMaxChunks>), smem);
}
bool tdes_loss_supported(const graft_config& cfg) { return cfg.m % 4 == 0 && cfg.m <= 128 * kTrMaxChunks; }

}  // namespace graft

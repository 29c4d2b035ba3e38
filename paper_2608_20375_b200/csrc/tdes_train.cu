// TDES training objective, forward and backward in one pass over the traces (Sec. 3.2 "Training", Eq. 7-12).
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
// reduced per CTA.  tdes_loss_rows_kernel for m <= 128, tdes_groups_kernel and tdes_items_kernel for m <= 128 and many
// traces, tdes_loss_kernel for wider rows.
// The order of the atomic additions is not fixed, so the gradients are reproducible only up to fp32 rounding.
#include <cuda_runtime.h>
#include <math.h>

#include "common.cuh"
#include "internal.h"

namespace graft {
namespace {

// *q += v in global memory, nothing returned (an atomicAdd of a float4 brings the old values back, used or not: 1.6 million
// rows in one step took 305 us so and 320 with it).
__device__ __forceinline__ void red_add4(float4* q, const float4& v) {
    asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(q), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w));
}

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
    double* acc;       // m <= 128: [6] loss sums, skipped items, arrival counter, gradient of the scale; zero between calls
    int gu_copies;     // m <= 128: copies of gu in shared memory: one per warp, or one
    int g_batch;       // m <= 128: groups of a batch
    int ctas;          // m <= 128: CTAs of the call, that arrive at acc
    float* gu_parts;   // [kTgParts][L][m] or NULL: where the groups' kernel adds its share of gu, for the items' to collect; zero between calls
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
            red_add4((float4*)(dst + (size_t)tok * m) + k4,
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
//   * with 65 thousand references and more, frequent tokens' rows are summed up on chip too (HOT).
// Many traces have kernels of their own, further down.
constexpr int kTsThreads = 384;
constexpr int kTsWarps = kTsThreads / 32;
// References to rows from which the two kernels for many traces are used.  With gradients (K = 32, tokens by a power of 1.1 of their
// rank, the kernel below and the two, us: 98 thousand 30.3 and 34.2, 130 thousand 33.8 and 37.3, 163 thousand 38.6 and 41.6, 195
// thousand 47.2 and 43.9, 293 thousand 59.2 and 57.8; by 1.6 195 thousand 42.2 and 45.0, 293 thousand 53.3 and 58.4) the line lies
// below where their times meet, because the two add to a row of gC less often (error against 64 bits, 163 thousand: 3.3e-7 and
// 2.5e-7, 260 thousand 3.8e-7 and 2.6e-7).  For the losses alone: 260 thousand 21.0 and 29.2, 520 thousand 35.4 and 37.4, a million
// 63.7 and 56.5.
constexpr long long kTsMany = 131072, kTsManyLoss = 655360;
// References to rows from which, with gradients, the frequent tokens' rows are summed up on chip (below it a step is over before a
// sample is worth its 1.5 us: 65 thousand references 21.5 us).
constexpr long long kTsHotMin = 65536;

constexpr int kTsSlots = 8;  // hot rows per table
struct __align__(16) TrainHot {
    int tok[2][kTsSlots];
};

__device__ __forceinline__ float2 lo2(const float4& v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(const float4& v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float4 join4(const float2& l, const float2& h) { return make_float4(l.x, l.y, h.x, h.y); }
__device__ __forceinline__ float4 add4(const float4& a, const float4& b) { return join4(__fadd2_rn(lo2(a), lo2(b)), __fadd2_rn(hi2(a), hi2(b))); }
__device__ __forceinline__ float4 mul4(float c, const float4& a) {
    const float2 cc = make_float2(c, c);
    return join4(__fmul2_rn(cc, lo2(a)), __fmul2_rn(cc, hi2(a)));
}
__device__ __forceinline__ float4 fma4(float c, const float4& a, const float4& b) {
    const float2 cc = make_float2(c, c), l = __ffma2_rn(cc, lo2(a), lo2(b)), h = __ffma2_rn(cc, hi2(a), hi2(b));
    return join4(l, h);
}
__device__ __forceinline__ float4 sub4(const float4& a, const float4& b) { return fma4(-1.f, b, a); }
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
// Sums of N values over either half of the warp (N = 4, 8, 16): value i is returned to the half's lanes with
// (l >> (4 - log2 N)) == i.
template <int N>
__device__ __forceinline__ float half_sums(float (&v)[N], int lane) {
    int mask = 8;
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
__device__ __forceinline__ int tok_hash(int tok, int bits) { return (int)((uint32_t)tok * 2654435761u >> (32 - bits)); }
// The tokens counted most often get the slots.  cnt, tok: [2][HASH] counters by a hash of the token, and the last token counted;
// least: what is worth a slot; at most kTsCand of either table's counters may have that many.  Every thread calls this, and is past a
// barrier when it returns.  (The first eight that reach it instead of the largest: 4,500 groups, tokens by a power of 1.6, of which ten
// reach it, 86 us instead of 58; 9,000 groups by a power of 1.1 97 instead of 83.)
constexpr int kTsCand = 64;
struct __align__(16) TrainCand {  // (zero at the start)
    int key[2][kTsCand];  // count and counter of those that reach it
    int n[2];
};
template <int HASH>
__device__ __forceinline__ void hot_pick(TrainHot& h, TrainCand& cand, const int* cnt, const int* tok, int least, int tid, int threads) {
    for (int i = tid; i < 2 * HASH; i += threads)
        if (cnt[i] >= least) {
            const int t = i / HASH, at = atomicAdd(&cand.n[t], 1);
            if (at < kTsCand) cand.key[t][at] = cnt[i] * HASH + i % HASH;
            if (at < kTsSlots) h.tok[t][at] = tok[i];
        }
    __syncthreads();
    if (max(cand.n[0], cand.n[1]) <= kTsSlots) return;  // (uniform)
    if (tid < 2 * kTsCand) {
        const int t = tid / kTsCand, at = tid % kTsCand, key = cand.key[t][at];
        if (cand.n[t] > kTsSlots && key > 0) {
            int rank = 0;
#pragma unroll 4
            for (int j = 0; j < kTsCand; j += 4) {
                const int4 o = *(const int4*)(cand.key[t] + j);
                rank += (o.x > key) + (o.y > key) + (o.z > key) + (o.w > key);
            }
            if (rank < kTsSlots) h.tok[t][rank] = tok[t * HASH + key % HASH];
        }
    }
    __syncthreads();
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
        red_add4(ctx_at<FULL>(c, t == 0 ? p.gP : p.gC, tok), v);
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

// The sums of the frequent tokens' rows that the warps in the mask kept, [warp][2][kTsSlots][32], go out: one addition a row and CTA.
__device__ __forceinline__ void flush_hot(const TrainParams& p, const TrainHot& h, const float4* rows, uint32_t warps, int tid, int threads) {
    for (int i = tid; i < 2 * kTsSlots * 32; i += threads) {
        const int r = i >> 5, l = i & 31, tok = h.tok[r / kTsSlots][r % kTsSlots];
        if (tok < 0 || l >= p.m / 4) continue;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int w = 0; w < 32; ++w)
            if (warps >> w & 1u) v = add4(v, rows[w * 2 * kTsSlots * 32 + i]);
        red_add4((float4*)((r < kTsSlots ? p.gP : p.gC) + (size_t)tok * p.m) + l, v);
    }
}
// The i-th of kTsThreads tokens spread evenly over the references to a table (0: P, 1: C), or -1; every CTA has a sample of its own,
// so that what one misses by chance the others find.  (Fewer than kTsMany references.)
__device__ __forceinline__ int train_sample(const TrainParams& p, int t, int i) {
    const int ng = t == 0 ? p.n_groups : p.n_groups * p.K, np = 2 * p.n_pairs;
    int at = (int)((float)(ng + np + p.n_edges) * ((float)(i * (int)gridDim.x + (int)blockIdx.x) / (float)(kTsThreads * (int)gridDim.x)));
    int tok = -1;
    if (at < ng) {
        tok = t == 0 ? p.g_parent[at] : p.g_child[at];
    } else if ((at -= ng) < np) {
        tok = p.pairs[(at >> 1) * 6 + (at & 1) * 3 + t];
    } else if ((at -= np) < p.n_edges) {
        tok = p.edges[at * 4 + t];
    }
    return tok_ok(tok, p.V) ? tok : -1;
}

// The work is one list -- groups, blocks of eight pairs, blocks of eight edges -- dealt to the warps in turn: the first of a
// kind, with `ahead` entries of other kinds ahead of it, that warp wid of nw gets.  (Dealt kind by kind, the first warps got
// one of each, one after the other, while the rest had nothing: half of a small call's time.)
__device__ __forceinline__ int first_block(int wid, long long ahead, int nw) {
    const int r = wid - (int)(ahead % nw);
    return r < 0 ? r + nw : r;
}

// The CTA's share of the losses: sums over its warps, one addition each; the CTA that arrives last (of p.ctas) writes the
// losses and clears the sums for the next call.  Every thread calls this.
struct TrainSums {
    double loss[3];
    float gs;
    int skip;
};
__device__ __forceinline__ void train_finish(const TrainParams& p, TrainSums& s, double l_kl, double l_pair, double l_bce, float gs,
                                             int skipped, int lane) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        l_kl += __shfl_xor_sync(0xFFFFFFFFu, l_kl, o);
        l_pair += __shfl_xor_sync(0xFFFFFFFFu, l_pair, o);
        l_bce += __shfl_xor_sync(0xFFFFFFFFu, l_bce, o);
    }
    gs = warp_sum(gs);
    skipped = __reduce_add_sync(0xFFFFFFFFu, skipped);
    if (lane == 0) {
        atomicAdd(&s.loss[0], l_kl);
        atomicAdd(&s.loss[1], l_pair);
        atomicAdd(&s.loss[2], l_bce);
        atomicAdd(&s.gs, gs);
        if (skipped) atomicAdd(&s.skip, skipped);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicAdd(p.acc + 0, s.loss[0]);
        atomicAdd(p.acc + 1, s.loss[1]);
        atomicAdd(p.acc + 2, s.loss[2]);
        if (s.skip) atomicAdd((int*)(p.acc + 3), s.skip);
        if (p.gu_parts != nullptr)  // (two kernels' CTAs: twice as many roundings, unless in 64 bits)
            atomicAdd(p.acc + 5, (double)s.gs);
        else if (p.gP != nullptr && s.gs != 0.f)
            atomicAdd(p.gs, s.gs);
        __threadfence();
        if (atomicAdd((unsigned int*)(p.acc + 4), 1u) == (unsigned)p.ctas - 1) {
            __threadfence();
            const double scale = p.gu_parts != nullptr ? __ldcg(p.acc + 5) : 0.0;
            const int skipped_all = __ldcg((const int*)(p.acc + 3));
            const double kl = __ldcg(p.acc + 0) / (double)(p.n_groups > 0 ? p.n_groups : 1);
            const double pr = __ldcg(p.acc + 1) / (double)(p.n_pairs > 0 ? p.n_pairs : 1);
            const double bc = __ldcg(p.acc + 2) / (double)(p.n_edges > 0 ? p.n_edges : 1);
            p.loss[0] = kl;
            p.loss[1] = pr;
            p.loss[2] = bc;
            p.loss[3] = (double)p.lam_kl * kl + (double)p.lam_pair * pr + (double)p.lam_bce * bc;
            if (p.skipped) *p.skipped = skipped_all;
            if (p.gu_parts != nullptr) atomicAdd(p.gs, (float)scale);
            for (int i = 0; i < 6; ++i) p.acc[i] = 0.0;
        }
    }
}

// HOT: additions to one row follow one another in L2, and what is behind them waits too; and each is rounded.  So the most frequent
// tokens' rows are summed up per warp in shared memory: those with a 48th of a sample of 384 references or more, eight a table at most.
// Captured, K = 32, without and with, us: 1,100 groups by a power of 1.1 of the tokens' rank 23.8 and 25.2, by 1.6 40.9 and 24.2; 2,000 by
// 1.1 39.2 and 33.3, by 1.6 70.7 and 31.1, by 2.5 103 and 31.4, spread nearly evenly (0.5) 25.9 and 28.1.  Error against 64 bits, root mean
// square, 2,000 by 1.1: gP 1.1e-6 and 2.3e-7, gC 7.0e-7 and 3.0e-7 (four slots and a 24th: 2.9e-7 and 4.1e-7, 1 to 3 us less).
constexpr int kTsHashBits = 9, kTsHash = 1 << kTsHashBits;
constexpr int kTsLeast = kTsThreads / 48;
constexpr int kTsPicked = 256;  // s_ready: a picked table, and its slots
constexpr int kTsTries = 4096;  // looks for the picked tokens before a warp does without

// KC: children held in registers, a multiple of 8 (K <= KC).  HOT: frequent tokens, found in a sample of the references, have their
// rows summed up per warp.
template <int KC, bool FULL, bool HOT>
__global__ void __launch_bounds__(kTsThreads, 1) tdes_loss_rows_kernel(const TrainParams p) {
    extern __shared__ __align__(16) float smem_f[];
    __shared__ TrainSums s_sum;
    __shared__ TrainHot s_hot;
    __shared__ int s_cnt[HOT ? 2 * kTsHash : 1], s_tok[HOT ? 2 * kTsThreads : 1], s_ready;  // counters by a hash, the sample
    __shared__ uint32_t s_used;  // the warps that keep sums
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, Lm = p.L * p.m;
    const bool grad = p.gP != nullptr;
    float* s_gu = smem_f + Lm;  // [L][m] u, then the copies of gu
    TrainCtx c;
    c.u = smem_f;
    c.gu_shared = p.gu_copies == 1;
    c.gu = s_gu + (c.gu_shared ? 0 : (size_t)warp * Lm);
    float4* s_rows = (float4*)(s_gu + (size_t)Lm * p.gu_copies);  // HOT: [kTsWarps][2][kTsSlots][32] sums of the frequent tokens' rows
    c.hot = s_rows + (size_t)warp * 2 * kTsSlots * 32;
    c.on = lane < p.m / 4;
    c.lane = lane;
    c.m = p.m;
    const int mine[2] = {HOT ? train_sample(p, 0, tid) : -1, HOT ? train_sample(p, 1, tid) : -1};
    for (int i = tid; i < Lm; i += kTsThreads) smem_f[i] = p.u[i];
    if (grad)
        for (int i = tid; i < Lm / 4 * p.gu_copies; i += kTsThreads) ((float4*)s_gu)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (tid < 3) s_sum.loss[tid] = 0.0;
    if (tid == 0) {
        s_sum.gs = 0.f;
        s_sum.skip = 0;
    }
    if (HOT) {
        for (int i = tid; i < 2 * kTsHash; i += kTsThreads) s_cnt[i] = 0;
        if (tid < 2 * kTsSlots) s_hot.tok[tid / kTsSlots][tid % kTsSlots] = -1;
        if (tid == 0) {
            s_ready = 0;
            s_used = 0u;
        }
    }
    __syncthreads();
    // A warp a table picks the tokens from the sample while the others are on their way to their first additions, in front of which they
    // look for them (everybody waiting here: 2.5 us a call instead of 1.5).
    bool seen = false, any = false;  // (uniform)
    if constexpr (HOT) {
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            s_tok[t * kTsThreads + tid] = mine[t];
            if (mine[t] >= 0) atomicAdd(&s_cnt[t * kTsHash + tok_hash(mine[t], kTsHashBits)], 1);
        }
        if (warp < 2) {
            const int t = warp;
            named_bar_sync(1, kTsThreads);
            int slot = 0;
            for (int n = 0; n < 2 * kTsSlots && slot < kTsSlots; ++n) {  // the largest counter first
                int best = 0;
                for (int i = lane; i < kTsHash; i += 32) best = max(best, s_cnt[t * kTsHash + i] << kTsHashBits | i);
                best = __reduce_max_sync(0xFFFFFFFFu, best);
                if (best >> kTsHashBits < kTsLeast) break;
                best &= kTsHash - 1;
                // its token: what a lane meets most often, if that is enough by itself (the last one counted instead: a CTA in ten without
                // the most frequent child, 55 us instead of 30)
                int tok = -1, votes = 0, count = 0;
                for (int i = lane; i < kTsThreads; i += 32) {
                    const int x = s_tok[t * kTsThreads + i];
                    if (x < 0 || tok_hash(x, kTsHashBits) != best) continue;
                    if (votes == 0) tok = x;
                    votes += x == tok ? 1 : -1;
                }
                tok = __shfl_sync(0xFFFFFFFFu, tok, __reduce_max_sync(0xFFFFFFFFu, votes << 5 | lane) & 31);
                for (int i = lane; i < kTsThreads; i += 32) count += s_tok[t * kTsThreads + i] == tok ? 1 : 0;
                count = __reduce_add_sync(0xFFFFFFFFu, count);
                if (lane == 0) {
                    s_cnt[t * kTsHash + best] = 0;
                    if (count >= kTsLeast) s_hot.tok[t][slot] = tok;
                }
                slot += count >= kTsLeast ? 1 : 0;
                __syncwarp();
            }
            __threadfence_block();
            __syncwarp();
            if (lane == 0) atomicAdd(&s_ready, kTsPicked + slot);
        } else {
            named_bar_arrive(1, kTsThreads);
        }
    }
    const auto look = [&] {
        if (!HOT || seen) return;
        int ready = 0;
        for (int i = 0; i < kTsTries && ready < 2 * kTsPicked; ++i) ready = __shfl_sync(0xFFFFFFFFu, *(volatile int*)&s_ready, 0);
        if (ready < 2 * kTsPicked) return;
        __threadfence_block();
        seen = true;
        any = ready > 2 * kTsPicked;
        if (!any) return;
        for (int r = 0; r < 2 * kTsSlots; ++r)
            if (s_hot.tok[r / kTsSlots][r % kTsSlots] >= 0) c.hot[r * 32 + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (lane == 0) atomicOr(&s_used, 1u << warp);
    };
    const auto slot_at = [&](int slot, int from) { return any ? __shfl_sync(0xFFFFFFFFu, slot, from) : -1; };
    const auto slot_of = [&](int t, int tok) { return any ? hot_slot(s_hot, t, tok) : -1; };
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
        look();
        const int slot = lane < p.K ? slot_of(1, tc) : -1;
        const uint32_t hots = any ? __ballot_sync(0xFFFFFFFFu, slot >= 0) : 0u;
        // sum_c coef_c (C_c + u) = sum_c coef_c C_c: the coefficients, differences of two distributions, add up to 0
        float4 acc = zero4;
#pragma unroll
        for (int i = 0; i < KC; ++i) {
            if (i < p.K) {
                const float cf = __shfl_sync(0xFFFFFFFFu, coef, i);
                const int t = __shfl_sync(0xFFFFFFFFu, tc, i);
                acc = fma4(cf, rows[i], acc);
                if (!((hots >> i) & 1u) && (FULL || c.on)) red_add4(ctx_at<FULL>(c, p.gC, t), mul4(cf, a));
            }
        }
        for (uint32_t left = hots; left != 0u; left &= left - 1u) {  // (uniform)
            const int i = __ffs(left) - 1;
            smem_add4(c.hot + (kTsSlots + __shfl_sync(0xFFFFFFFFu, slot, i)) * 32 + lane, mul4(__shfl_sync(0xFFFFFFFFu, coef, i), a));
        }
        ctx_add_row<FULL>(p, c, 0, tp, slot_of(0, tp), acc);
        ctx_add_u<FULL>(c, d, acc);
    }
    // ---- pairwise level (Eq. 10): blocks of eight pairs, four at a time; lanes 0-7 hold the block's ids
    for (int b0 = first_block(wid, p.n_groups, nw) * 8; b0 < p.n_pairs; b0 += nw * 8) {
        look();
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
        const int sp1 = slot_of(0, id[0]), sc1 = slot_of(1, id[1]), sp2 = slot_of(0, id[3]), sc2 = slot_of(1, id[4]);
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
                const int h1 = slot_at(sp1, s), h2 = slot_at(sc1, s);
                if (p1 == p2) {  // (uniform; an alternative keeps the pair's parent or its child: one addition for both)
                    ctx_add_row<FULL>(p, c, 0, p1, h1, mul4(cf, sub4(b2[i], b1[i])));
                } else {
                    ctx_add_row<FULL>(p, c, 0, p1, h1, mul4(-cf, b1[i]));
                    ctx_add_row<FULL>(p, c, 0, p2, slot_at(sp2, s), mul4(cf, b2[i]));
                }
                if (c1 == c2) {
                    ctx_add_row<FULL>(p, c, 1, c1, h2, mul4(cf, sub4(a2[i], a1[i])));
                } else {
                    ctx_add_row<FULL>(p, c, 1, c1, h2, mul4(-cf, a1[i]));
                    ctx_add_row<FULL>(p, c, 1, c2, slot_at(sc2, s), mul4(cf, a2[i]));
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
        look();
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
        const int sp = slot_of(0, tp), sc = slot_of(1, tc);
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
            ctx_add_row<FULL>(p, c, 0, __shfl_sync(0xFFFFFFFFu, tp, i), slot_at(sp, i), mul4(cf, b[i]));
            ctx_add_row<FULL>(p, c, 1, __shfl_sync(0xFFFFFFFFu, tc, i), slot_at(sc, i), mul4(cf, a[i]));
            ctx_add_u<FULL>(c, __shfl_sync(0xFFFFFFFFu, d, i), mul4(cf, add4(a[i], b[i])));
        }
    }
    // ---- per-CTA sums, then one round of global reductions, four values each: of few groups this end was a tenth of the
    //      call (500 groups, K = 32: 15.6 us with one value each, 14.1 so; 2,000 groups: 40.4 and 38.6; 4,000: no change)
    __syncthreads();
    if (grad)
        for (int i = tid; i < Lm / 4; i += kTsThreads) {
            const float4* q = (const float4*)s_gu + i;
            float4 v = *q;
#pragma unroll 4
            for (int w = 1; w < p.gu_copies; ++w) v = add4(v, q[(size_t)w * (Lm / 4)]);
            if (v.x != 0.f || v.y != 0.f || v.z != 0.f || v.w != 0.f) red_add4((float4*)p.gu + i, v);
        }
    if (HOT) flush_hot(p, s_hot, s_rows, s_used, tid, kTsThreads);
    train_finish(p, s_sum, l_kl, l_pair, l_bce, gs, skipped, lane);
}

// ---- many traces: groups first, then pairs and edges ---------------------------------------------------------------------
// What bounds a large step is the vector additions: an SM hands on one row (512 bytes) in 20 cycles, all of them a million
// rows in 94 us however they are spread (row loads are three times faster and overlap them), and rows that meet take 4.6 ns
// each.  So additions are saved where the operands are on chip already, and either half of the work has a kernel that keeps
// what it needs there:
//   * tdes_groups_kernel: a CTA's groups (up to 224) leave their parents' rows in shared memory, and the children are put in
//     the order of their tokens (counting sort by a hash), so that what a token gets from all of them is summed up first: half
//     of the children of 222 groups are met before in real traces (Zipf), 562 thousand additions instead of 965.  A batch goes
//     through it in stages that hold eight rows a warp -- all products, then all distributions, then the additions with the
//     children's rows read a second time -- because 24 warps of 80 registers beat 12 that keep the rows (150 us against 163);
//   * tdes_items_kernel: a batch of pairs and edges is sorted by depth in shared memory, so that a warp keeps u_d and its sum
//     of gu_d in registers; the most frequent tokens of the first batch are summed up per warp in shared memory.
// Measured (B200, V = 151,936, m = 128, L = 16, 32,768 groups of 32, 131,072 pairs, 262,144 edges): 250 us, the two alone 147
// and 99; 320 by the kernel above with the frequent tokens' rows per warp.  1.2 million additions are 115 us of it, the
// rest chains of loads and exchanges.  Tried: the frequent tokens' rows as one dense block whose scores and coefficients are
// single numbers (423 us: four numbers a reference cost what a row does, and the sums lost a digit); two warps a group with
// the rows kept (150 - 190); both kernels on an SM at once, half the warps each (249 against 251); the children's rows read once, with
// a running softmax (163 - 167 against 150: the longer chain of a group costs what the second read does).
constexpr int kTgGroups = 224;  // groups of a batch at most
constexpr int kTgThreads = 768;
// Sums of gu over the grid are rounded with every CTA's addition, and two kernels have twice as many CTAs: with the groups' adding
// to four places by turns the error against 64 bits is that of one kernel (root mean square, before two kernels / two / so: 4,000
// groups 1.82e-7 / 2.10e-7 / 1.76e-7, 32,768 1.85e-7 / 1.98e-7 / 1.83e-7).  Collecting them, and gs in 64 bits (2.4e-7 and 2e-8), are 0.4 us of 41 to 250.
constexpr int kTgParts = 4;
constexpr int kTgBinBits = 13, kTgBins = 1 << kTgBinBits;
constexpr int kTeThreads = 512;
constexpr int kTeWarps = kTeThreads / 32;
constexpr int kTeEdges = 2 * kTeThreads;  // a batch: two edges a thread
constexpr int kTePairs = kTeThreads;      // and a pair
constexpr int kTeHash = 1024;   // counters for the frequent tokens

// KC: children a group has room for, 8, 16 or 32 (K <= KC)
template <int KC, bool FULL>
__global__ void __launch_bounds__(kTgThreads, 1) tdes_groups_kernel(const TrainParams p) {
    extern __shared__ __align__(16) float smem_f[];
    __shared__ TrainSums s_sum;
    __shared__ int s_scan[8];
    __shared__ __align__(16) int s_parent[kTgGroups];
    __shared__ uint8_t s_order[kTgGroups], s_depth[kTgGroups];  // (depth 0: a group that does not count)
    constexpr int W = kTgThreads / 32, NB = kTgBins / 2;
    __shared__ int s_run[W];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, h = lane >> 4, l = lane & 15, Lm = p.L * p.m;
    const bool grad = p.gP != nullptr;
    float4* s_a = (float4*)smem_f;                          // [g_batch][32] the groups' P + u
    float* s_f = (float*)(s_a + p.g_batch * 32);            // [g_batch][KC] products, then coefficients
    int* s_tok = (int*)(s_f + p.g_batch * KC);              // [g_batch][KC] the children
    uint32_t* s_bin = (uint32_t*)(s_tok + p.g_batch * KC);  // [NB] two bins a word: where a bin's next child goes
    float* s_u = (float*)(s_bin + NB);                      // [L][m]
    float* s_gu = s_u + Lm;                                 // [L][m]
    uint16_t* s_rec = (uint16_t*)(s_gu + Lm);               // [g_batch * KC + 32] the children in the order of their bins
    pdl_launch_dependents();  // (the other kernel's work is independent of this one's; it waits for nothing here but the SMs)
    for (int i = tid; i < Lm; i += kTgThreads) {
        s_u[i] = p.u[i];
        s_gu[i] = 0.f;
    }
    if (tid < 3) s_sum.loss[tid] = 0.0;
    if (tid == 0) {
        s_sum.gs = 0.f;
        s_sum.skip = 0;
    }
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const bool on = FULL || lane < p.m / 4, on0 = FULL || l < p.m / 4, on1 = FULL || 16 + l < p.m / 4;
    const int mm = FULL ? 128 : p.m;
    double l_kl = 0.0;
    float gs = 0.f;
    int skipped = 0;
    // Half a warp a row, two float4s a lane (l and 16 + l): a sum over 16 lanes is one exchange shorter, and a lane handles
    // half as many rows.
    const auto half_row = [&](const float* table, int tok, float4 (&v)[2]) {
        const float4* q = (const float4*)(table + (size_t)tok * mm) + l;
        v[0] = on0 ? __ldg(q) : zero4;
        v[1] = on1 ? __ldg(q + 16) : zero4;
    };
    const int g_lo = (int)((long long)p.n_groups * blockIdx.x / gridDim.x), g_hi = (int)((long long)p.n_groups * (blockIdx.x + 1) / gridDim.x);
    const int n_batch = (g_hi - g_lo + p.g_batch - 1) / p.g_batch;
    for (int bt = 0; bt < n_batch; ++bt) {
        const int g0 = g_lo + (int)((long long)(g_hi - g_lo) * bt / n_batch), ng = g_lo + (int)((long long)(g_hi - g_lo) * (bt + 1) / n_batch) - g0;
        __syncthreads();
        // ---- the groups' ids; how many children fall into a bin
        for (int i = tid; i < NB; i += kTgThreads) s_bin[i] = 0u;
        for (int i = ng + tid; i < kTgGroups; i += kTgThreads) s_parent[i] = 0x7FFFFFFF;
        __syncthreads();
#pragma unroll 2
        for (int gl = warp; gl < ng; gl += W) {
            const int g = g0 + gl, tp = p.g_parent[g], d = p.g_depth[g];
            const int tc = p.g_child[(size_t)g * p.K + min(lane, p.K - 1)];  // (places past K: the last child again)
            const bool ok = __all_sync(0xFFFFFFFFu, tok_ok(tc, p.V)) && tok_ok(tp, p.V) && d >= 1 && d <= p.L;
            if (lane < KC) s_tok[gl * KC + lane] = ok ? tc : 0;
            if (ok && grad && lane < p.K) {
                const int b = tok_hash(tc, kTgBinBits);
                atomicAdd(&s_bin[b >> 1], b & 1 ? 0x10000u : 1u);
            }
            if (lane == 0) {
                s_parent[gl] = tp;
                s_depth[gl] = ok ? (uint8_t)d : 0;
                skipped += ok ? 0 : 1;
            }
        }
        __syncthreads();
        // ---- the bins' places: an exclusive sum over them; beside it the order of the groups' parents
        if (grad && warp < 8) {
            uint32_t sum = 0;
#pragma unroll 8
            for (int i = 0; i < NB / 256; ++i) {
                const uint32_t word = s_bin[warp * (NB / 8) + 32 * i + lane];
                sum += (word & 0xFFFFu) + (word >> 16);
            }
            sum = __reduce_add_sync(0xFFFFFFFFu, sum);
            if (lane == 0) s_scan[warp] = (int)sum;
        }
        if (grad && warp >= W - 7 && tid - 32 * (W - 7) < ng) {  // groups of one parent side by side: one addition to its row
            const int i = tid - 32 * (W - 7), mine = s_parent[i];
            int rank = 0;
#pragma unroll 4
            for (int j = 0; j < kTgGroups; j += 4) {
                const int4 o = *(const int4*)(s_parent + j);
                rank += (o.x < mine || (o.x == mine && j < i)) + (o.y < mine || (o.y == mine && j + 1 < i)) +
                        (o.z < mine || (o.z == mine && j + 2 < i)) + (o.w < mine || (o.w == mine && j + 3 < i));
            }
            s_order[rank] = (uint8_t)i;
        }
        __syncthreads();
        int n_rec = 0;
        if (grad) {
            uint32_t base = 0;
            for (int w = 0; w < 8; ++w) {
                base += w < warp ? s_scan[w] : 0;
                n_rec += s_scan[w];
            }
            if (warp < 8) {
#pragma unroll 4
                for (int i = 0; i < NB / 256; ++i) {
                    uint32_t* word = s_bin + warp * (NB / 8) + 32 * i + lane;
                    const uint32_t lo = *word & 0xFFFFu, v = lo + (*word >> 16);
                    uint32_t incl = v;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                        if (lane >= o) incl += t;
                    }
                    const uint32_t at = base + incl - v;
                    *word = at | (at + lo) << 16;
                    base += __shfl_sync(0xFFFFFFFFu, incl, 31);
                }
            }
            if (tid < 32 && n_rec + tid < ((n_rec + 31) & ~31)) s_rec[n_rec + tid] = 0u;
        }
        // ---- products with the parent: eight children at a time
        for (int gl = warp; gl < ng; gl += W) {
            const int d = s_depth[gl];
            if (d == 0) continue;
            float4 a[2];
            half_row(p.P, s_parent[gl], a);
            float au[2] = {};
#pragma unroll 1
            for (int c = 0; c < KC; c += 8) {
                const int4 t = *(const int4*)(s_tok + gl * KC + c + 4 * h);
                float4 rows[4][2];
                half_row(p.C, t.x, rows[0]);
                half_row(p.C, t.y, rows[1]);
                half_row(p.C, t.z, rows[2]);
                half_row(p.C, t.w, rows[3]);
                if (c == 0) {  // f = k0 (a . C + a . u), summed up in the order of tdes_loss_rows_kernel: the same bits
                    const float4* q = (const float4*)(s_u + (d - 1) * p.m) + l;
                    const float4 u0 = on0 ? q[0] : zero4, u1 = on1 ? q[16] : zero4;
                    a[0] = add4(a[0], u0);
                    a[1] = add4(a[1], u1);
                    au[0] = dot4(a[0], u0);
                    au[1] = dot4(a[1], u1);
                    s_a[gl * 32 + lane] = h ? a[1] : a[0];
                }
                float part[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) part[i] = (au[0] + dot4(a[0], rows[i][0])) + (au[1] + dot4(a[1], rows[i][1]));
                const float dot = half_sums<4>(part, lane);  // child i of the half in lanes 16 h + 4 i ..
                if ((l & 3) == 0) s_f[gl * KC + c + 4 * h + (l >> 2)] = dot;
            }
        }
        __syncthreads();
        // ---- the two distributions, the loss, the coefficients (lane i: child i) and the children's places: two groups at a time
        for (int gl = warp; gl < ng; gl += 2 * W) {
            float z[2], al[2], dot[2], zmax[2], amax[2], ez[2], ea[2], zsum[2], asum[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int gq = gl + q * W;
                const bool use = gq < ng && lane < p.K;
                const size_t at = (size_t)(g0 + gq) * p.K + lane;
                dot[q] = use ? s_f[gq * KC + lane] : 0.f;
                z[q] = use ? p.g_ztgt[at] : -INFINITY;
                al[q] = use ? p.g_logq[at] + p.k0 * dot[q] : -INFINITY;
                zmax[q] = z[q];
                amax[q] = al[q];
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    zmax[q] = fmaxf(zmax[q], __shfl_xor_sync(0xFFFFFFFFu, zmax[q], o));
                    amax[q] = fmaxf(amax[q], __shfl_xor_sync(0xFFFFFFFFu, amax[q], o));
                }
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                zsum[q] = ez[q] = lane < p.K ? expf(z[q] - zmax[q]) : 0.f;
                asum[q] = ea[q] = lane < p.K ? expf(al[q] - amax[q]) : 0.f;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    zsum[q] += __shfl_xor_sync(0xFFFFFFFFu, zsum[q], o);
                    asum[q] += __shfl_xor_sync(0xFFFFFFFFu, asum[q], o);
                }
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int gq = gl + q * W;
                if (gq >= ng || s_depth[gq] == 0) continue;  // (uniform)
                const float pt = ez[q] / zsum[q], ph = ea[q] / asum[q];
                if (lane < p.K && pt > 0.f) l_kl += (double)(pt * ((z[q] - zmax[q] - logf(zsum[q])) - (al[q] - amax[q] - logf(asum[q]))));
                if (!grad) continue;
                const float gf = lane < p.K ? p.w_kl * (ph - pt) : 0.f;  // d L / d f
                gs += gf * dot[q] * p.inv_sqrt_m;
                if (lane < KC) s_f[gq * KC + lane] = gf * p.k0;
                if (lane < p.K) {
                    const int b = tok_hash(s_tok[gq * KC + lane], kTgBinBits);
                    const uint32_t old = atomicAdd(&s_bin[b >> 1], b & 1 ? 0x10000u : 1u);
                    s_rec[b & 1 ? old >> 16 : old & 0xFFFFu] = (uint16_t)(gq * KC + lane);
                }
            }
        }
        if (!grad) continue;
        __syncthreads();
        // ---- the additions, turn by turn: a group's sum over its children (to its parent's row and its depth's), and 32 of the
        // sorted children, of which a token's stand side by side (but for the few that share a bin), so that the vector
        // additions to gC and the loads for gP overlap
        const int at_lo = ng * warp / W, at_hi = ng * (warp + 1) / W;
        int run_tp = -1;  // the parent whose groups are summed up in run
        float4 run = zero4;
        const auto flush = [&] {
            if (run_tp >= 0 && on) red_add4((float4*)(p.gP + (size_t)run_tp * mm) + lane, run);
            run = zero4;
        };
        for (int at = at_lo, r0 = warp * 32; at < at_hi || r0 < n_rec; ++at, r0 += kTgThreads) {
            const int gl = at < at_hi ? s_order[at] : 0, d = at < at_hi ? s_depth[gl] : 0;
            if (d != 0) {
                // sum_c coef_c (C_c + u) = sum_c coef_c C_c: the coefficients, differences of two distributions, add up to 0
                float4 acc[2] = {zero4, zero4};
#pragma unroll 1
                for (int c = 0; c < KC; c += 8) {
                    const int4 t = *(const int4*)(s_tok + gl * KC + c + 4 * h);
                    const float4 cf = *(const float4*)(s_f + gl * KC + c + 4 * h);
                    float4 rows[4][2];
                    half_row(p.C, t.x, rows[0]);
                    half_row(p.C, t.y, rows[1]);
                    half_row(p.C, t.z, rows[2]);
                    half_row(p.C, t.w, rows[3]);
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        acc[k] = fma4(cf.x, rows[0][k], acc[k]);
                        acc[k] = fma4(cf.y, rows[1][k], acc[k]);
                        acc[k] = fma4(cf.z, rows[2][k], acc[k]);
                        acc[k] = fma4(cf.w, rows[3][k], acc[k]);
                    }
                }
                const float4 give = h ? acc[0] : acc[1], keep = h ? acc[1] : acc[0];
                const float4 sum = make_float4(keep.x + __shfl_xor_sync(0xFFFFFFFFu, give.x, 16), keep.y + __shfl_xor_sync(0xFFFFFFFFu, give.y, 16),
                                               keep.z + __shfl_xor_sync(0xFFFFFFFFu, give.z, 16), keep.w + __shfl_xor_sync(0xFFFFFFFFu, give.w, 16));
                const int tp = s_parent[gl];
                if (tp != run_tp) {  // (uniform)
                    flush();
                    run_tp = tp;
                }
                run = add4(run, sum);
                if (on) {
                    float* q = s_gu + (d - 1) * p.m + 4 * lane;
                    atomicAdd(q + 0, sum.x);
                    atomicAdd(q + 1, sum.y);
                    atomicAdd(q + 2, sum.z);
                    atomicAdd(q + 3, sum.w);
                }
            }
            if (r0 < n_rec) {
                const int me = s_rec[r0 + lane], tok = r0 + lane < n_rec ? s_tok[me] : -1, next = __shfl_down_sync(0xFFFFFFFFu, tok, 1);
                uint32_t ends = __ballot_sync(0xFFFFFFFFu, tok >= 0 && (lane == 31 || next != tok));  // the last of a token's
                float4 acc = zero4;
#pragma unroll 1
                for (int i0 = 0; i0 < 32; i0 += 8, ends >>= 8) {
                    // (places and coefficients as broadcast loads: from lane to lane they cost two exchanges a row, 152 us against 147)
                    const uint4 recs = *(const uint4*)(s_rec + r0 + i0);
                    const uint32_t word[4] = {recs.x, recs.y, recs.z, recs.w};
                    float4 row[8];
                    float cf[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const uint32_t m = q & 1 ? word[q >> 1] >> 16 : word[q >> 1] & 0xFFFFu;
                        cf[q] = s_f[m];
                        row[q] = s_a[m / KC * 32 + lane];
                    }
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        acc = fma4(cf[q], row[q], acc);
                        if (ends & (1u << q)) {  // (uniform)
                            const int t = __shfl_sync(0xFFFFFFFFu, tok, i0 + q);
                            if (on) red_add4((float4*)(p.gC + (size_t)t * mm) + lane, acc);
                            acc = zero4;
                        }
                    }
                }
            }
        }
        // the runs that the warps end with, neighbours' of one parent together
        __syncthreads();
        s_a[tid] = run;
        if (lane == 0) s_run[warp] = run_tp;
        __syncthreads();
        if (run_tp >= 0 && (warp == 0 || s_run[warp - 1] != run_tp)) {
            for (int w = warp + 1; w < W && s_run[w] == run_tp; ++w) run = add4(run, s_a[w * 32 + lane]);
            flush();
        }
    }
    if (grad) {
        __syncthreads();
        float4* gu = p.gu_parts != nullptr ? (float4*)p.gu_parts + (int)(blockIdx.x % kTgParts) * (Lm / 4) : (float4*)p.gu;
        for (int i = tid; i < Lm / 4; i += kTgThreads) red_add4(gu + i, ((const float4*)s_gu)[i]);
    }
    __syncthreads();
    train_finish(p, s_sum, l_kl, 0.0, 0.0, gs, skipped, lane);
}

// Pairs and edges.
template <bool FULL>
__global__ void __launch_bounds__(kTeThreads, 1) tdes_items_kernel(const TrainParams p) {
    extern __shared__ __align__(16) float smem_f[];
    __shared__ TrainSums s_sum;
    __shared__ TrainHot s_hot;
    __shared__ TrainCand s_cand;
    __shared__ int s_start[2][kMaxL + 1];  // edges, pairs: the first of a depth in the sorted batch
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, Lm = p.L * p.m;
    const bool grad = p.gP != nullptr;
    int4* s_edge = (int4*)smem_f;                   // [kTeEdges] parent, child, label | slots
    int4* s_pair = s_edge + kTeEdges;               // [kTePairs] the four tokens
    int* s_pinfo = (int*)(s_pair + kTePairs);       // [kTePairs] second depth | slots
    float4* s_rows = (float4*)(s_pinfo + kTePairs); // [kTeWarps][2][kTsSlots][32] sums of the frequent tokens' rows
    float* s_u = (float*)(s_rows + kTeWarps * 2 * kTsSlots * 32);  // [L][m]
    float* s_gu = s_u + Lm;                                         // [L][m]
    TrainCtx c;
    c.u = s_u;
    c.gu = nullptr;
    c.hot = s_rows + warp * 2 * kTsSlots * 32;
    c.gu_shared = false;
    c.on = lane < p.m / 4;
    c.lane = lane;
    c.m = p.m;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    int* s_cnt = (int*)s_rows;               // [2][kTeHash] (before the rows)
    int* s_tok = s_cnt + 2 * kTeHash;        // [2][kTeHash]
    for (int i = tid; i < Lm; i += kTeThreads) {
        s_u[i] = p.u[i];
        s_gu[i] = 0.f;
    }
    const auto add_gu = [&](int d, const float4& v) {
        if (d < 1 || !grad || !(FULL || c.on)) return;
        float* q = s_gu + (d - 1) * p.m + 4 * lane;
        atomicAdd(q + 0, v.x);
        atomicAdd(q + 1, v.y);
        atomicAdd(q + 2, v.z);
        atomicAdd(q + 3, v.w);
    };
    for (int i = tid; i < 2 * kTeHash; i += kTeThreads) s_cnt[i] = 0;
    if (tid < 3) s_sum.loss[tid] = 0.0;
    if (tid == 0) {
        s_sum.gs = 0.f;
        s_sum.skip = 0;
    }
    if (tid < (int)(sizeof(TrainCand) / sizeof(int))) ((int*)&s_cand)[tid] = 0;
    if (tid < 2 * kTsSlots) s_hot.tok[tid / kTsSlots][tid % kTsSlots] = -1;
    __syncthreads();
    double l_pair = 0.0, l_bce = 0.0;
    float gs = 0.f;
    int skipped = 0;
    const int e_lo = (int)((long long)p.n_edges * blockIdx.x / gridDim.x), e_hi = (int)((long long)p.n_edges * (blockIdx.x + 1) / gridDim.x);
    const int q_lo = (int)((long long)p.n_pairs * blockIdx.x / gridDim.x), q_hi = (int)((long long)p.n_pairs * (blockIdx.x + 1) / gridDim.x);
    const int n_batch = max((e_hi - e_lo + kTeEdges - 1) / kTeEdges, (q_hi - q_lo + kTePairs - 1) / kTePairs);
    for (int bt = 0; bt < n_batch; ++bt) {
        const auto part = [&](int lo, int hi, int i) { return lo + (int)((long long)(hi - lo) * i / n_batch); };
        const int e0 = part(e_lo, e_hi, bt), ne = part(e_lo, e_hi, bt + 1) - e0, q0 = part(q_lo, q_hi, bt), nq = part(q_lo, q_hi, bt + 1) - q0;
        // ---- the batch in registers, then sorted by depth into shared memory
        int4 edge[2];
        bool e_ok[2];
        int id[6] = {0, 0, 1, 0, 0, 1};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int i = tid + k * kTeThreads;
            edge[k] = make_int4(0, 0, 1, 0);
            if (i < ne) {  // (the lists are aligned to their elements only)
                const int32_t* e = p.edges + (size_t)(e0 + i) * 4;
                edge[k] = make_int4(e[0], e[1], e[2], e[3]);
            }
        }
        if (tid < nq) {
            const int32_t* q = p.pairs + (size_t)(q0 + tid) * 6;
#pragma unroll
            for (int k = 0; k < 6; ++k) id[k] = q[k];
        }
        if (tid < 2 * kMaxL) s_start[tid / kMaxL][tid % kMaxL] = 0;
        __syncthreads();
        int e_rank[2] = {}, q_rank = 0;
        const auto depth_ok = [&](int d) { return d >= 1 && d <= p.L; };
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            e_ok[k] = tid + k * kTeThreads < ne && tok_ok(edge[k].x, p.V) && tok_ok(edge[k].y, p.V) && depth_ok(edge[k].z);
            skipped += tid + k * kTeThreads < ne && !e_ok[k] ? 1 : 0;
            if (e_ok[k]) e_rank[k] = atomicAdd(&s_start[0][edge[k].z - 1], 1);
        }
        const bool q_ok = tid < nq && tok_ok(id[0], p.V) && tok_ok(id[1], p.V) && tok_ok(id[3], p.V) && tok_ok(id[4], p.V) && depth_ok(id[2]) && depth_ok(id[5]);
        skipped += tid < nq && !q_ok ? 1 : 0;
        if (q_ok) q_rank = atomicAdd(&s_start[1][id[2] - 1], 1);
        if (grad && bt == 0) {  // the tokens met most often, by a hash
            const auto count = [&](int t, int tok) {
                const int h = t * kTeHash + tok_hash(tok, 10);
                atomicAdd(&s_cnt[h], 1);
                s_tok[h] = tok;
            };
#pragma unroll
            for (int k = 0; k < 2; ++k)
                if (e_ok[k]) {
                    count(0, edge[k].x);
                    count(1, edge[k].y);
                }
            if (q_ok) {
                count(0, id[0]);
                count(1, id[1]);
                count(0, id[3]);
                count(1, id[4]);
            }
        }
        __syncthreads();
        if (warp < 2) {  // a depth's count becomes the place of its first item, and behind the last depth stands their number
            const int v = s_start[warp][lane];
            int incl = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= o) incl += t;
            }
            s_start[warp][lane] = incl - v;
            if (lane == 31) s_start[warp][kMaxL] = incl;
        }
        if (grad && bt == 0)
            hot_pick<kTeHash>(s_hot, s_cand, s_cnt, s_tok, max(8, (ne + 2 * nq + kTsCand - 1) / kTsCand), tid, kTeThreads);
        else
            __syncthreads();
        if (grad && bt == 0)
            for (int i = tid; i < kTeWarps * 2 * kTsSlots * 32; i += kTeThreads) s_rows[i] = zero4;
        const auto slot_of = [&](int t, int tok) { return grad ? hot_slot(s_hot, t, tok) + 1 : 0; };  // 0: none
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (e_ok[k])
                s_edge[s_start[0][edge[k].z - 1] + e_rank[k]] = make_int4(edge[k].x, edge[k].y, edge[k].w ? 1 : 0, slot_of(0, edge[k].x) | slot_of(1, edge[k].y) << 4);
        if (q_ok) {
            const int at = s_start[1][id[2] - 1] + q_rank;
            s_pair[at] = make_int4(id[0], id[1], id[3], id[4]);
            s_pinfo[at] = id[5] | slot_of(0, id[0]) << 8 | slot_of(1, id[1]) << 12 | slot_of(0, id[3]) << 16 | slot_of(1, id[4]) << 20;
        }
        __syncthreads();
        // ---- edge level (Eq. 11): a warp's stretch of the sorted edges, up to eight of one depth at a time
        {
            const int n = s_start[0][kMaxL];
            int i = n * warp / kTeWarps;
            const int hi = n * (warp + 1) / kTeWarps;
            int d = 0, d_end = 0;
            float4 u = zero4, gu = zero4;
            while (i < hi) {
                if (i >= d_end) {  // the next depth that has an edge
                    add_gu(d, gu);
                    do {
                        ++d;
                        d_end = s_start[0][d];
                    } while (i >= d_end);
                    u = ctx_u<FULL>(c, d);
                    gu = zero4;
                }
                const int cnt = min(8, min(hi, d_end) - i);
                float4 a[8], b[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int2 e = *(const int2*)(s_edge + i + min(q, cnt - 1));  // (past the last: it again, and no additions)
                    a[q] = ctx_load<FULL>(c, p.P, e.x);
                    b[q] = ctx_load<FULL>(c, p.C, e.y);
                }
                const bool mine = (lane >> 2) < cnt;
                const bool good = s_edge[i + min(lane >> 2, cnt - 1)].z != 0;
                float part[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    a[q] = add4(a[q], u);
                    b[q] = add4(b[q], u);
                    part[q] = dot4(a[q], b[q]);
                }
                const float dot = warp_sums<8>(part, lane);  // lanes 4 q .. 4 q + 3: edge q
                const float f = p.k0 * dot;
                const float fy = good ? -f : f, e = expf(-fabsf(fy)), w = good ? p.w1 : 1.f;  // softplus(fy), sigmoid(fy)
                const float gf = mine && grad ? (good ? -p.w_bce : p.w_bce) * w * ((fy >= 0.f ? 1.f : e) / (1.f + e)) : 0.f;
                if (mine && (lane & 3) == 0) {
                    l_bce += (double)(w * (fmaxf(fy, 0.f) + log1pf(e)));
                    gs += gf * dot * p.inv_sqrt_m;
                }
                if (grad) {
                    const float coef = gf * p.k0;
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        if (q >= cnt) break;  // (uniform)
                        const float cf = __shfl_sync(0xFFFFFFFFu, coef, 4 * q);
                        const int4 e = s_edge[i + q];
                        ctx_add_row<FULL>(p, c, 0, e.x, (e.w & 15) - 1, mul4(cf, b[q]));
                        ctx_add_row<FULL>(p, c, 1, e.y, (e.w >> 4) - 1, mul4(cf, a[q]));
                        gu = fma4(cf, add4(a[q], b[q]), gu);
                    }
                }
                i += cnt;
            }
            add_gu(d, gu);
        }
        // ---- pairwise level (Eq. 10): four pairs at a time, sorted by the first one's depth
        {
            const int n = s_start[1][kMaxL];
            int i = n * warp / kTeWarps;
            const int hi = n * (warp + 1) / kTeWarps;
            int d = 0, d_end = 0;
            float4 u = zero4, gu = zero4;
            while (i < hi) {
                if (i >= d_end) {
                    add_gu(d, gu);
                    do {
                        ++d;
                        d_end = s_start[1][d];
                    } while (i >= d_end);
                    u = ctx_u<FULL>(c, d);
                    gu = zero4;
                }
                const int cnt = min(4, min(hi, d_end) - i);
                float4 a1[4], b1[4], a2[4], b2[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int4 e = s_pair[i + min(q, cnt - 1)];
                    a1[q] = ctx_load<FULL>(c, p.P, e.x);
                    b1[q] = ctx_load<FULL>(c, p.C, e.y);
                    a2[q] = ctx_load<FULL>(c, p.P, e.z);
                    b2[q] = ctx_load<FULL>(c, p.C, e.w);
                }
                float part[8];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int d2 = s_pinfo[i + min(q, cnt - 1)] & 255;
                    const float4 u2 = d2 == d ? u : ctx_u<FULL>(c, d2);  // (uniform)
                    a1[q] = add4(a1[q], u);
                    b1[q] = add4(b1[q], u);
                    a2[q] = add4(a2[q], u2);
                    b2[q] = add4(b2[q], u2);
                    part[2 * q] = dot4(a1[q], b1[q]);
                    part[2 * q + 1] = dot4(a2[q], b2[q]);
                }
                const float dot = warp_sums<8>(part, lane);  // lanes 8 q .. 8 q + 3: v+ of pair q, the next four: v-
                const float other = __shfl_xor_sync(0xFFFFFFFFu, dot, 4);
                const float dp = (lane & 4) ? other : dot, dm = (lane & 4) ? dot : other;
                const float x = p.gamma - p.k0 * dp + p.k0 * dm;
                const bool mine = (lane >> 3) < cnt;
                const float e = expf(-fabsf(x));
                const float gx = mine && grad ? p.w_pair * ((x >= 0.f ? 1.f : e) / (1.f + e)) : 0.f;
                if (mine && (lane & 7) == 0) {
                    l_pair += (double)(fmaxf(x, 0.f) + log1pf(e));
                    gs += gx * (dm - dp) * p.inv_sqrt_m;
                }
                if (grad) {
                    const float coef = gx * p.k0;  // of v-; v+ gets its negative
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (q >= cnt) break;  // (uniform)
                        const float cf = __shfl_sync(0xFFFFFFFFu, coef, 8 * q);
                        const int4 e = s_pair[i + q];
                        const int info = s_pinfo[i + q];
                        const int h1 = (info >> 8 & 15) - 1, h2 = (info >> 12 & 15) - 1, h3 = (info >> 16 & 15) - 1, h4 = (info >> 20 & 15) - 1;
                        if (e.x == e.z) {  // (uniform; an alternative keeps the pair's parent or its child: one addition for both)
                            ctx_add_row<FULL>(p, c, 0, e.x, h1, mul4(cf, sub4(b2[q], b1[q])));
                        } else {
                            ctx_add_row<FULL>(p, c, 0, e.x, h1, mul4(-cf, b1[q]));
                            ctx_add_row<FULL>(p, c, 0, e.z, h3, mul4(cf, b2[q]));
                        }
                        if (e.y == e.w) {
                            ctx_add_row<FULL>(p, c, 1, e.y, h2, mul4(cf, sub4(a2[q], a1[q])));
                        } else {
                            ctx_add_row<FULL>(p, c, 1, e.y, h2, mul4(-cf, a1[q]));
                            ctx_add_row<FULL>(p, c, 1, e.w, h4, mul4(cf, a2[q]));
                        }
                        const float4 s1 = add4(a1[q], b1[q]), s2 = add4(a2[q], b2[q]);
                        if ((info & 255) == d) {
                            gu = fma4(cf, sub4(s2, s1), gu);
                        } else {
                            gu = fma4(-cf, s1, gu);
                            add_gu(info & 255, mul4(cf, s2));
                        }
                    }
                }
                i += cnt;
            }
            add_gu(d, gu);
        }
        __syncthreads();
    }
    const int n4 = Lm / 4, col = (int)blockIdx.x + tid * (int)gridDim.x;
    if (grad && n_batch > 0) {
        for (int i = tid; i < n4; i += kTeThreads) red_add4((float4*)p.gu + i, ((const float4*)s_gu)[i]);
        flush_hot(p, s_hot, s_rows, (1u << kTeWarps) - 1, tid, kTeThreads);
    }
    pdl_wait();  // (the end of this kernel stands for the end of both)
    // the groups' share of gu, a few columns a CTA: on its way while the losses are finished
    const bool collect = grad && p.gu_parts != nullptr && col < n4;
    float4 share[kTgParts];
    if (collect) {
#pragma unroll
        for (int k = 0; k < kTgParts; ++k) share[k] = __ldcg((const float4*)p.gu_parts + k * n4 + col);
    }
    train_finish(p, s_sum, 0.0, l_pair, l_bce, gs, skipped, lane);
    if (collect) {
#pragma unroll
        for (int k = 0; k < kTgParts; ++k) ((float4*)p.gu_parts)[k * n4 + col] = zero4;
#pragma unroll
        for (int k = kTgParts / 2; k >= 1; k /= 2)
#pragma unroll
            for (int q = 0; q < k; ++q) share[q] = add4(share[q], share[q + k]);
        red_add4((float4*)p.gu + col, share[0]);
    }
}

}  // namespace

// One copy of gu a warp where they fit beside the rest (the usual L m = 2048), else one with atomics.
static int rows_gu_copies(const graft_config& cfg) { return cfg.L * cfg.m <= 2048 ? kTsWarps : 1; }
static size_t tdes_loss_smem(const graft_config& cfg) {
    const size_t lm = (size_t)((cfg.L * cfg.m + 3) & ~3);
    if (cfg.m > 128) return lm * sizeof(float);  // gu
    return lm * (1 + rows_gu_copies(cfg)) * sizeof(float);
}
static size_t rows_hot_smem(const graft_config& cfg) { return tdes_loss_smem(cfg) + (size_t)kTsWarps * 2 * kTsSlots * 512; }
template <bool HOT>
static void (*rows_kernel(const graft_config& cfg))(const TrainParams) {
    if (cfg.m == 128) return cfg.K <= 8 ? tdes_loss_rows_kernel<8, true, HOT> : (cfg.K <= 16 ? tdes_loss_rows_kernel<16, true, HOT> : tdes_loss_rows_kernel<32, true, HOT>);
    return cfg.K <= 8 ? tdes_loss_rows_kernel<8, false, HOT> : (cfg.K <= 16 ? tdes_loss_rows_kernel<16, false, HOT> : tdes_loss_rows_kernel<32, false, HOT>);
}

static void (*groups_kernel(const graft_config& cfg))(const TrainParams) {
    if (cfg.m == 128) return cfg.K <= 8 ? tdes_groups_kernel<8, true> : (cfg.K <= 16 ? tdes_groups_kernel<16, true> : tdes_groups_kernel<32, true>);
    return cfg.K <= 8 ? tdes_groups_kernel<8, false> : (cfg.K <= 16 ? tdes_groups_kernel<16, false> : tdes_groups_kernel<32, false>);
}
static size_t groups_smem(const graft_config& cfg, int batch) {
    const int kc = cfg.K <= 8 ? 8 : (cfg.K <= 16 ? 16 : 32);
    return (size_t)batch * (512 + kc * (sizeof(float) + sizeof(int) + sizeof(uint16_t))) + 64 + kTgBins / 2 * sizeof(uint32_t) + 2 * (size_t)cfg.L * cfg.m * sizeof(float);
}
static int groups_batch(const graft_config& cfg) {  // (L m = 2048: all 224; 4096: 208)
    int n = kTgGroups;
    while (groups_smem(cfg, n) > (size_t)220 * 1024) n -= 8;
    return n;
}
static size_t items_smem(const graft_config& cfg) {
    return (size_t)(kTeEdges + kTePairs) * sizeof(int4) + kTePairs * sizeof(int) + (size_t)kTeWarps * 2 * kTsSlots * 512 + 2 * (size_t)cfg.L * cfg.m * sizeof(float);
}

size_t tdes_loss_bytes(const graft_config& cfg) {
    return kLossSums * sizeof(double) + (cfg.m <= 128 ? (size_t)kTgParts * cfg.L * cfg.m * sizeof(float) : 0);
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
        p.gu_parts = nullptr;
        p.gu_copies = rows_gu_copies(cfg);
        // a warp takes a group, eight pairs or eight edges at a time
        const long long work = (long long)tr->n_groups + (tr->n_pairs + 7ll) / 8 + (tr->n_edges + 7ll) / 8;
        long long grid = (work + kTsWarps - 1) / kTsWarps;
        if (grid > ctx->num_sms) grid = ctx->num_sms;
        const long long refs = (long long)tr->n_groups * (cfg.K + 1) + 4ll * tr->n_pairs + 2ll * tr->n_edges;
        // (a kernel is loaded with the first call that wants it: a millisecond each, which graft_create need not wait for)
        bool many = refs >= (d_gP ? kTsMany : kTsManyLoss);
        if (many && !ctx->loss_many) {
            cudaError_t e = allow_smem((const void*)groups_kernel(cfg), groups_smem(cfg, groups_batch(cfg)));
            if (e == cudaSuccess) e = allow_smem((const void*)(cfg.m == 128 ? tdes_items_kernel<true> : tdes_items_kernel<false>), items_smem(cfg));
            if (e != cudaSuccess) cudaGetLastError();
            many = ctx->loss_many = e == cudaSuccess;
        }
        if (!many) {
            bool hot = d_gP && refs >= kTsHotMin;
            if (hot && !ctx->loss_hot) {
                ctx->loss_hot = allow_smem((const void*)rows_kernel<true>(cfg), rows_hot_smem(cfg)) == cudaSuccess;
                if (!ctx->loss_hot) cudaGetLastError();
                hot = ctx->loss_hot;
            }
            p.ctas = (int)grid;
            if (hot)
                rows_kernel<true>(cfg)<<<(int)grid, kTsThreads, rows_hot_smem(cfg), st>>>(p);
            else
                rows_kernel<false>(cfg)<<<(int)grid, kTsThreads, smem, st>>>(p);
            ctx->launches += 1;
            return cudaGetLastError();
        }
        const int n_g = tr->n_groups > 0 ? ctx->num_sms : 0, n_i = tr->n_pairs + tr->n_edges > 0 ? ctx->num_sms : 0;
        p.ctas = n_g + n_i;
        p.gu_parts = d_gP && n_g > 0 && n_i > 0 ? (float*)(ctx->w_loss + kLossSums) : nullptr;
        p.g_batch = groups_batch(cfg);
        cudaError_t e = cudaSuccess;
        if (n_g > 0) {
            groups_kernel(cfg)<<<n_g, kTgThreads, groups_smem(cfg, p.g_batch), st>>>(p);
            ctx->launches += 1;
            e = cudaGetLastError();
        }
        if (n_i > 0 && e == cudaSuccess) {
            void (*items)(const TrainParams) = cfg.m == 128 ? tdes_items_kernel<true> : tdes_items_kernel<false>;
            if (n_g > 0)
                e = launch_pdl(items, dim3(n_i), dim3(kTeThreads), items_smem(cfg), st, p);
            else
                items<<<n_i, kTeThreads, items_smem(cfg), st>>>(p);
            ctx->launches += 1;
            if (e == cudaSuccess) e = cudaGetLastError();
        }
        // (thread blocks of a kernel that did start have arrived at sums that the other's would have brought back to zero)
        if (e != cudaSuccess) {
            cudaGetLastError();
            cudaMemsetAsync(ctx->w_loss, 0, tdes_loss_bytes(cfg), st);
        }
        return e;
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
    if (cfg.m > 128) return allow_smem((const void*)(cfg.m <= 256 ? tdes_loss_kernel<2> : tdes_loss_kernel<kTrMaxChunks>), smem);
    return allow_smem((const void*)rows_kernel<false>(cfg), smem);
}
bool tdes_loss_supported(const graft_config& cfg) { return cfg.m % 4 == 0 && cfg.m <= 128 * kTrMaxChunks; }

}  // namespace graft

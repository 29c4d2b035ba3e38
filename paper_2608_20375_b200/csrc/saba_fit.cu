// Least-squares fit of the SABA gain and cost models to replay logs (Sec. 3.3; the paper fits them on held-out
// prompts by same-prefix budget replay and does not say how: ordinary least squares is the reading taken here).
//
//   gain (Eq. 16):  G = 1 - exp(-B / tau), tau = phi . s + bias, so a logged gain 0 < g_i < 1 at budget B_i gives
//                   tau_i = -B_i / ln(1 - g_i); (phi, bias) = argmin sum_i (tau_i - phi . s_i - bias)^2
//   cost (Eq. 17):  (c0, c1, c2) = argmin sum_i (T_i - c0 - c1 B_i - c2 B_i prefix_i)^2
//
// One pass over the tuples accumulates the normal equations in fp64 (per thread, per warp by shuffles, per CTA in shared
// memory, per grid by one atomic a sum); the CTA that finishes last solves the two small systems (columns scaled to unit
// diagonal first, then Gauss-Jordan elimination with partial pivoting) and clears the accumulators for the next call.
//
// 28 bytes are read a tuple and some 55 fp64 operations done on it: with the next tuples' loads in flight and the table of logarithms
// kept by the context a million tuples take 4.4 us (6.3 TB/s, the copy rate; 5.2 without), and a call costs 6 us however few:
// launch, exchange, one round of atomics, the systems (half the threads a CTA for few rounds and the table fetched while the kernel ahead runs: 20,000
// rounds captured 7.5 -> 6.3 us, 100 5.9 -> 5.4).  4 million tuples on a B200, one call after another: 30.0 -> 25.2 us, of
// which 2.5 are the launch behind the call before (one CTA of 512 threads an SM and two of 256 are alike from 200,000 tuples on; the
// CTAs' sums written out and added up in order by the last CTA instead of by atomics: 3 us slower at a million).  Before: 37.3 ->
// 28.9 with logarithms from a table and a short series instead of log, one division for four quotients and whole numbers converted
// on the fp64 pipe (earlier steps, from 56.9: log for log1p, counts as integers, products by one folded, the elimination on a warp
// and sums without shared-memory atomics).
#include <cuda_runtime.h>
#include <math.h>

#include "common.cuh"
#include "internal.h"

namespace graft {
namespace {

constexpr int kFitThreads = 512, kFitFew = 256;  // one CTA an SM
// Turns of a thread (four rounds, or one where the arrays are not aligned) from which a CTA has the larger number: with few, warps that
// have next to nothing to add up take their part in the exchange all the same.  256 and 512, captured, us: four rounds a turn, 20,000 rounds 6.8
// and 7.4, 100,000 6.8 and 7.4, 130,000 7.3 both, 200,000 7.8 and 7.5; one, 20,000 6.3 and 6.6, 40,000 7.1 and 6.9, 400,000 12.2 and 9.3.
constexpr long long kFitMany = 1 << 15;
constexpr int kFitAcc = 25;  // gain: 10 (upper triangle of 4 x 4) + 4 + 1 count; cost: 6 + 3 + 1 count

struct FitParams {
    long long n;
    const float* state;     // [n, 3] conf, degen, hist
    const int32_t* budget;  // [n]
    const float* gain;      // [n]
    const int32_t* prefix;  // [n]
    const float* latency;   // [n]
    const double2* log;     // [kFitLog] table of logarithms (fit_log)
    double* acc;            // [kFitAcc] zero between calls
    unsigned int* ticket;   // zero between calls
    double* out;            // [10]
};

// x = argmin |A x - r| for the normal equations A (n x n, symmetric, upper triangle given row by row; n <= 4), by one warp:
// lane (r, c) of n x (n + 1) holds an entry of the scaled system [A | r], and Gauss-Jordan elimination with partial pivoting
// runs on shuffles, so that a step is one division deep.  One thread with the matrix in local memory took 3 us more.
// Lane r (n + 1) + n returns x[r]; ok is false when a pivot of the scaled system vanishes.
__device__ __forceinline__ double solve_normal(const double* tri, const double* rhs, int n, int lane, bool& ok) {
    const int w = n + 1;
    const bool on = lane < n * w;
    const int r = on ? lane / w : 0, c = on ? lane % w : 0;
    const int i = min(r, c), j = max(r, c);
    const auto diag = [&](int k) { return tri[k * n - k * (k - 1) / 2]; };  // entry (k, k); (i, j) is j - i behind (i, i)
    const double drr = diag(r), dcc = c < n ? diag(c) : 1.0;
    ok = __all_sync(0xFFFFFFFFu, drr > 0.0);
    if (!ok) return 0.0;
    const double dr = 1.0 / sqrt(drr), dc = c < n ? 1.0 / sqrt(dcc) : 1.0;
    double a = (c < n ? tri[i * n - i * (i - 1) / 2 + j - i] : rhs[r]) * (dr * dc);
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
        int piv = k;
        double best = fabs(__shfl_sync(0xFFFFFFFFu, a, k * w + k));
#pragma unroll 1
        for (int q = k + 1; q < n; ++q) {
            const double v = fabs(__shfl_sync(0xFFFFFFFFu, a, q * w + k));
            if (v > best) best = v, piv = q;
        }
        ok = best > 1e-13;
        if (!ok) return 0.0;  // the same in every lane
        a = __shfl_sync(0xFFFFFFFFu, a, (r == k ? piv : r == piv ? k : r) * w + c);
        const double f = __shfl_sync(0xFFFFFFFFu, a, r * w + k) / __shfl_sync(0xFFFFFFFFu, a, k * w + k);
        const double t = __shfl_sync(0xFFFFFFFFu, a, k * w + c);
        if (r != k) a -= f * t;
    }
    return a / __shfl_sync(0xFFFFFFFFu, a, r * w + r) * dr;
}

// The sums of one thread: everything but the two counts in fp64.
struct FitSums {
    double acc[kFitAcc];
    int n_gain, n_cost;
};
// a whole number as fp64, on the fp64 pipe (conversions run at a quarter of its rate)
__device__ __forceinline__ double fit_double(int x) {
    return __hiloint2double(0x43300000, x ^ (int)0x80000000) - 4503601774854144.0;  // 2^52 + 2^31
}
// log(1 - g) for 0 < g < 1 (24 bits, so 1 - g is exact from 2^-29 up), by a table of logarithms and a short series (P. T. P. Tang,
// "Table-driven implementation of the logarithm function in IEEE floating-point arithmetic", 1990): 1 - g = 2^e f, c the
// multiple of 1/512 nearest to f in [1/2, 1), r = f / c - 1, log(1 - g) = e ln 2 + log c + log(1 + r), |r| <= 2^-9; the series' first term
// left out is 2^-57 of r.  With c = 1 for g below 2^-10, where r is -g itself, small results keep their relative precision.
// tab[k]: 1 / c rounded, and minus the logarithm of that, c = 1/2 + k / 512 (saba_fit_table).  Largest relative error 3e-16.
__device__ __forceinline__ double fit_log(const double2* tab, double g) {
    const double x = 1.0 - g;
    const int hi = __double2hiint(x);
    const bool near1 = g < 0x1p-10;
    const double2 t = tab[near1 ? 256 : ((hi & 0xFFFFF) + 0x800) >> 12];
    const double f = __hiloint2double((hi & 0xFFFFF) | 0x3FE00000, __double2loint(x));
    const double e = fit_double(near1 ? 0 : (hi >> 20) - 1022);
    const double r = near1 ? -g : fma(f, t.x, -1.0);
    double q = fma(r, -1.0 / 6.0, 0.2);
    q = fma(r, q, -0.25);
    q = fma(r, q, 1.0 / 3.0);
    q = fma(r, q, -0.5);
    return fma(e, 0.69314718055994530942, t.y) + fma(r * r, q, r);
}
// One logged round into the running sums.  No branch around the gain model (a warp nearly always has both kinds): a round
// that says nothing about tau takes part with zeros.
__device__ __forceinline__ bool fit_ok(float gain) { return gain > 0.0f && gain < 1.0f; }  // a gain of 0 or 1 says nothing about tau
__device__ __forceinline__ void fit_accumulate(FitSums& t, float s0, float s1, float s2, double B, bool ok, double tau, int prefix,
                                               float latency) {
    double* acc = t.acc;
    const double a = (double)(ok ? s0 : 0.f), b = (double)(ok ? s1 : 0.f), c = (double)(ok ? s2 : 0.f);
    acc[0] = fma(a, a, acc[0]);
    acc[1] = fma(a, b, acc[1]);
    acc[2] = fma(a, c, acc[2]);
    acc[3] += a;
    acc[4] = fma(b, b, acc[4]);
    acc[5] = fma(b, c, acc[5]);
    acc[6] += b;
    acc[7] = fma(c, c, acc[7]);
    acc[8] += c;
    acc[10] = fma(a, tau, acc[10]);
    acc[11] = fma(b, tau, acc[11]);
    acc[12] = fma(c, tau, acc[12]);
    acc[13] += tau;
    t.n_gain += ok ? 1 : 0;
    const double T = (double)latency, BP = B * fit_double(prefix);
    acc[16] += B;
    acc[17] += BP;
    acc[18] = fma(B, B, acc[18]);
    acc[19] = fma(B, BP, acc[19]);
    acc[20] = fma(BP, BP, acc[20]);
    acc[21] += T;
    acc[22] = fma(B, T, acc[22]);
    acc[23] = fma(BP, T, acc[23]);
    ++t.n_cost;
}

// VEC: every array is 16-byte aligned, so a thread takes four consecutive rounds with seven 16-byte loads
template <bool VEC, int T>
__global__ void __launch_bounds__(T, 1) saba_fit_kernel(const FitParams p) {
    constexpr int W = T / 32;
    __shared__ double2 s_log[kFitLog];
    __shared__ double s_acc[kFitAcc], s_warp[W][kFitAcc];
    __shared__ bool s_last;
    __shared__ int s_bad[2];
    pdl_launch_dependents();
    for (int i = threadIdx.x; i < kFitLog; i += T) s_log[i] = p.log[i];  // (written once, by graft_create)
    pdl_wait();  // (the logs may come from the kernel ahead, and the one before this may still add up)
    const long long tid = blockIdx.x * (long long)T + threadIdx.x, nth = (long long)gridDim.x * T;
    const long long n4 = VEC ? p.n / 4 : 0;
    // the next four rounds are on their way while four are worked on, the first beside the table
    float4 a, b, c, ga, la;
    int4 bu, pr;
    const auto fetch = [&](long long q) {
        if (q >= n4) return;
        a = __ldg((const float4*)p.state + 3 * q), b = __ldg((const float4*)p.state + 3 * q + 1), c = __ldg((const float4*)p.state + 3 * q + 2);
        bu = __ldg((const int4*)p.budget + q), pr = __ldg((const int4*)p.prefix + q);
        ga = __ldg((const float4*)p.gain + q), la = __ldg((const float4*)p.latency + q);
    };
    if (VEC) fetch(tid);
    __syncthreads();
    FitSums t;
#pragma unroll
    for (int i = 0; i < kFitAcc; ++i) t.acc[i] = 0.0;
    t.n_gain = t.n_cost = 0;
    long long done = 0;
    if (VEC) {
#pragma unroll 1
        for (long long q = tid; q < n4; q += nth) {
            const float4 sa = a, sb = b, sc = c, gn = ga, lt = la;
            const int4 bd = bu, pf = pr;
            fetch(q + nth);
            // tau = -B / log(1 - g), the four quotients by one division: 1 / l0 = (l2 l3 / (l0 l1 l2 l3)) l1 and so on (P. L.
            // Montgomery's simultaneous inversion, 1987); the product of four logarithms is between 1e-180 and 1e5.  A quotient goes
            // through three products more than a division of its own: a few units in the last place of fp64, as does the series above.
            const bool ok[4] = {fit_ok(gn.x), fit_ok(gn.y), fit_ok(gn.z), fit_ok(gn.w)};
            const float g4[4] = {gn.x, gn.y, gn.z, gn.w};
            double l[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) l[i] = ok[i] ? fit_log(s_log, (double)g4[i]) : 1.0;
            const double l01 = l[0] * l[1], l23 = l[2] * l[3], inv = 1.0 / (l01 * l23), i01 = inv * l23, i23 = inv * l01;
            const double B[4] = {fit_double(bd.x), fit_double(bd.y), fit_double(bd.z), fit_double(bd.w)};
            fit_accumulate(t, sa.x, sa.y, sa.z, B[0], ok[0], ok[0] ? -B[0] * (i01 * l[1]) : 0.0, pf.x, lt.x);
            fit_accumulate(t, sa.w, sb.x, sb.y, B[1], ok[1], ok[1] ? -B[1] * (i01 * l[0]) : 0.0, pf.y, lt.y);
            fit_accumulate(t, sb.z, sb.w, sc.x, B[2], ok[2], ok[2] ? -B[2] * (i23 * l[3]) : 0.0, pf.z, lt.z);
            fit_accumulate(t, sc.y, sc.z, sc.w, B[3], ok[3], ok[3] ? -B[3] * (i23 * l[2]) : 0.0, pf.w, lt.w);
        }
        done = n4 * 4;
    }
    for (long long i = done + tid; i < p.n; i += nth) {
        const float gain = p.gain[i];
        const bool ok = fit_ok(gain);
        const double B = fit_double(p.budget[i]);
        const double tau = ok ? -B / fit_log(s_log, (double)gain) : 0.0;
        fit_accumulate(t, p.state[3 * i], p.state[3 * i + 1], p.state[3 * i + 2], B, ok, tau, p.prefix[i], p.latency[i]);
    }
    t.acc[9] = t.acc[14] = (double)t.n_gain;
    t.acc[15] = t.acc[24] = (double)t.n_cost;
    // The warp's sums of all 25 in 31 steps of exchange (each halves what a lane still carries: lane i ends with sum i)
    // instead of 25 x 5, and a CTA's sums by one thread each: shared-memory atomics on doubles are retry loops.
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const bool up = (lane & d) != 0;
#pragma unroll
        for (int i = 0; i < d; ++i) {
            const double lo = t.acc[i], hi = i + d < kFitAcc ? t.acc[i + d] : 0.0;
            t.acc[i] = (up ? hi : lo) + __shfl_xor_sync(0xFFFFFFFFu, up ? lo : hi, d);
        }
    }
    if (lane < kFitAcc) s_warp[warp][lane] = t.acc[0];
    __syncthreads();
    if (threadIdx.x < kFitAcc) {
        double v = s_warp[0][lane];
#pragma unroll
        for (int i = 1; i < W; ++i) v += s_warp[i][lane];
        atomicAdd(p.acc + lane, v);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(p.ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (threadIdx.x < kFitAcc) {
        s_acc[threadIdx.x] = __ldcg(p.acc + threadIdx.x);
        p.acc[threadIdx.x] = 0.0;  // ready for the next call
    }
    if (threadIdx.x == 0) *p.ticket = 0u;
    __syncthreads();
    if (warp < 2) {  // the two systems side by side
        const int n = 4 - warp;
        const double* tri = s_acc + 15 * warp;
        const double* rhs = tri + n * (n + 1) / 2;
        bool ok;
        const double x = solve_normal(tri, rhs, n, lane, ok), count = rhs[n];
        ok = ok && count >= (double)n;
        if (lane < n * (n + 1) && lane % (n + 1) == n) p.out[4 * warp + lane / (n + 1)] = ok ? x : 0.0;
        if (lane == 0) {
            p.out[7 + warp] = count;
            s_bad[warp] = ok ? 0 : 1 + warp;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) p.out[9] = (double)(s_bad[0] | s_bad[1]);
}

}  // namespace

size_t saba_fit_doubles() { return 2 * kFitLog + 2 + kFitAcc; }
void saba_fit_table(double* table) {
    for (int k = 0; k < kFitLog - 1; ++k) {
        const double inv = 1.0 / (0.5 + k * (1.0 / 512.0));
        table[2 * k] = inv;
        table[2 * k + 1] = -log(inv);
    }
    table[2 * (kFitLog - 1)] = 1.0;
    table[2 * (kFitLog - 1) + 1] = 0.0;
}

cudaError_t saba_fit_launch(graft_ctx* ctx, long long n, const float* d_state, const int32_t* d_budget,
                            const float* d_gain, const int32_t* d_prefix, const float* d_latency, double* d_out,
                            cudaStream_t st) {
    FitParams p;
    p.n = n;
    p.state = d_state;
    p.budget = d_budget;
    p.gain = d_gain;
    p.prefix = d_prefix;
    p.latency = d_latency;
    p.log = (const double2*)ctx->w_fit;
    p.ticket = (unsigned int*)(ctx->w_fit + 2 * kFitLog);
    p.acc = ctx->w_fit + 2 * kFitLog + 2;
    p.out = d_out;
    const bool vec = (((uintptr_t)d_state | (uintptr_t)d_budget | (uintptr_t)d_gain | (uintptr_t)d_prefix |
                       (uintptr_t)d_latency) & 15) == 0;
    const long long turns = vec ? n / 4 + 3 : n;
    const int threads = turns < kFitMany ? kFitFew : kFitThreads;
    long long grid = (turns + threads - 1) / threads;
    const long long cap = ctx->num_sms;
    if (grid > cap) grid = cap;
    if (grid < 1) grid = 1;
    void (*kern)(const FitParams) = turns < kFitMany ? (vec ? saba_fit_kernel<true, kFitFew> : saba_fit_kernel<false, kFitFew>)
                                                 : (vec ? saba_fit_kernel<true, kFitThreads> : saba_fit_kernel<false, kFitThreads>);
    const cudaError_t e = launch_pdl(kern, dim3((int)grid), dim3(threads), 0, st, p);
    ctx->launches += 1;
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace graft

// Table precompute on the tensor cores: out[v] = W e_v + b (text after Eq. 6: the projections depend only on the token
// id and are computed once).  This is the one dense contraction of the method, [V, E] x [E, m].
//
// Operands are 16-bit parts of the inputs; products of parts are exact in the fp32 accumulator.
//   bf16 embeddings: out = e W1 + e W2 + e W3, W as three bf16 parts (8 + 8 + 8 mantissa bits; three products a step)
//   fp32 embeddings: out = e1 W1 + (e1 W2 + e2 W1), both as two fp16 parts (11 + 11 bits and the second part's sign; what is
//     dropped, e2 W2, is below 2^-24 of a term and 2^-26 of it on average).  fp16 has few exponents, so a row of W is scaled by
//     its largest entry and the embeddings by a power of two from a sample; second parts are kept times 2^11, and go to an
//     accumulator of their own.  Rows of the embeddings that this does not suit are worked out in fp32.
// so the result differs from an fp32 GEMM by the order and the rounding of the additions.  The accumulators of the tensor
// cores round less carefully than an FMA chain, the less so the more bits the products have: they are emptied into fp32
// registers after 32 (bf16) or 16 (fp32 embeddings) additions to the large products' accumulators, which the small products do not
// share.  (fp16 parts for bf16 embeddings too, two products instead of three: the conversion in shared memory and the shorter
// chunks that the longer products need cost more than the third product, 398 against 375 us a tower, and at 32 additions the
// error was a third larger.)
//
// One persistent kernel.  A worker -- a pair of CTAs (cluster of two, tcgen05 cta_group::2) for bf16 embeddings, one CTA
// for fp32 -- owns a tile of 512 (fp32: 128) rows of V times up to 128 columns of m, and streams E in blocks of 64 (32)
// columns through shared-memory rings.
//   warps 0-7    empty the accumulators (TMEM, two sets of 2 x 128 columns), keep the running sums and write the tile
//   warp 8       TMA loads: W's parts (split once per call into scratch by a small kernel), bf16 embeddings
//   warp 9       issues the matrix instructions
//   warp 10      fp32 only: TMA loads of the raw rows;  warps 11-18  raw rows -> fp16 parts in the operands' layout
// W1 and W2 stand side by side as one operand of N = 256, the third product is an N = 128 of its own (three of N = 128 in a row on one
// accumulator took 122 cycles each: an instruction waits for the one ahead of it on the same columns).  Tiles of 512
// rows halve the passes over W, which comes from L2 every time.  The fp32 kernel works on single CTAs because its rows
// go through threads: telling the other CTA of a pair about every block cost more (136 - 160 us at V = 32,000, E = 2048)
// than the second CTA's half of W saves (120 us).  The embeddings are read from memory once; nothing but the tables is
// written.  What is left when the tiles do not divide by the workers is dealt out along E in shares, whose sums a
// small kernel adds up in order (summing them inside, by the warp that came last, stalled its tile: 462 against 370 us).
//
// Measured (one tower, back to back, B200): V = 151,936, E = 4096, m = 128, bf16: 358 us (375 before rows and W shared a barrier
// and the first row block went two blocks ahead where accumulators are emptied; 798 us with the library template's GEMMs); its products
// take 287 us at the measured dense rate, and the clock falls to 1.5 GHz on the way.  V = 32,000, E = 2048, fp32: 91 us (121 with
// three bf16 parts, seven products; 1180 us by the FMA kernel).  What bounds the fp32 kernel: the one thread that issues, 0.6 k
// cycles a block of 32 columns beside 0.4 k of products, and the eight warps that split.  Error against fp64 products at those
// sizes, largest and root mean square over the results' size: bf16 2.7e-6 and 4.7e-7; fp32 2.2e-6 and 3.4e-7 (bf16 parts 2.7e-6 and 4.7e-7; FMA kernel
// 1.2e-5 at most).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "internal.h"
#include "umma.cuh"

namespace graft {
namespace {

constexpr int kTmEpiWarps = 8;
constexpr int kTmConvWarps = 8;
constexpr int kTmMaxSplit = 16;  // pairs that share a left-over tile, about

// Ring sizes: what a block's copies need in flight (about 2 us of them) beside the blocks being worked on, in 227 KB.
template <bool F32>
struct TablesCfg {
    static constexpr bool PAIR = !F32;         // two CTAs work on a tile together
    static constexpr int MT = F32 ? 1 : 2;     // row blocks of 128 a CTA works on at a time
    static constexpr int ROWS = F32 ? 128 : 512;  // rows of V per tile
    static constexpr int BLK = F32 ? 32 : 64;  // columns of E per block: rows of 64 or 128 bytes of bf16
    static constexpr int CHUNK = 8;            // blocks between two emptyings of an accumulator
    static constexpr int PART = 128 * BLK * 2;                // bytes of 128 rows of 16-bit numbers
    static constexpr int A_BYTES = 2 * PART;                  // a block's embeddings: two row blocks, or two parts
    static constexpr int W_BYTES = (F32 ? 256 : 192) * BLK * 2;  // a block's W; a pair: W1 (even CTA) or W2 (odd), half of W3
    static constexpr int RAW = 128 * BLK * 4;                 // a block's fp32 embeddings
    static constexpr int STAGES = 4, RAW_STAGES = F32 ? 4 : 1;  // (a stage: a block's embeddings and W)
    static constexpr int THREADS = (kTmEpiWarps + 2 + (F32 ? 1 + kTmConvWarps : 0)) * 32;
    // (the rings start on a 1024-byte boundary)
    static constexpr size_t SMEM = (size_t)STAGES * (A_BYTES + W_BYTES) + (F32 ? (size_t)RAW_STAGES * RAW : 0) + 1024;
    static __device__ __forceinline__ uint64_t desc(uint32_t addr) { return F32 ? umma_desc_sw64(addr) : umma_desc_sw128(addr); }
};

constexpr float kTmLow = 2048.0f;  // fp16: second parts are kept times 2^11

// A walk over the N stages of a ring: stages passed so far, the stage, the parity to wait for.
template <uint32_t N>
struct TablesRing {
    uint32_t t = 0, st = 0, ph;
    __device__ __forceinline__ explicit TablesRing(uint32_t parity) : ph(parity) {}
    __device__ __forceinline__ void next() {
        ++t;
        if (++st == N) {
            st = 0;
            ph ^= 1;
        }
    }
    // Wait (bounded) until the stages passed last have been released; after an abort also, where `full` is given, until
    // their copies have landed.
    __device__ __forceinline__ void drain(uint32_t empty, uint32_t full, volatile int* abort_flag) const {
        const uint32_t back = t < N ? t : N;
        for (uint32_t b = 0; b < back; ++b) {
            const uint32_t tt = t - back + b, at = 8 * (tt % N), parity = (tt / N) & 1;
            for (uint32_t tries = 0; !mbar_try_wait_cluster(empty + at, parity) && tries < GRAFT_SPIN_LIMIT; ++tries)
                if (*abort_flag && tries > 4096u) break;
            if (*abort_flag && full != 0u)
                for (uint32_t tries = 0; !mbar_try_wait_cluster(full + at, parity) && tries < 65536u; ++tries) {
                }
        }
    }
};

struct __align__(64) TablesParams {
    CUtensorMap map_w;  // [parts * m_pad, E_pad]: three bf16 parts, or two fp16 ones
    CUtensorMap map_e;  // [V, E] embeddings
    const void* emb;    // [V, E]
    const float* W;     // [m, E]
    const float* bias;  // [m] or NULL
    float* out;         // [V, m]
    float* pieces;      // [pairs][2 pieces][ROWS][128]
    // fp32 embeddings only
    const float2* unscale;  // [m_pad] what a column's sums are multiplied by, as two factors
    const float* scale;     // [1] what the embeddings are multiplied by
    uint8_t* bad_row;       // [tiles][ROWS] rows whose entries fp16 parts do not hold well enough, as the tile's workers saw them
    int32_t* errflag;
    int V, E, m, m_pad, n_mb, n_kb;
    int pairs, full_rounds;
    int left, share_pairs;  // left-over tiles, pairs that share them
    int box_n;              // fp32 embeddings: rows of W's boxes
    int wide;               // rows of the table are whole 32-byte sectors
};

// What a pair works on: its share of the left-over tiles' blocks (no longer than a tile, so it lies in two tiles at most;
// tiles 0 .. left - 1), then whole tiles, one in every round.
struct TablesItem {
    int tile, kb0, kb1;
    int q0, q1;  // a piece: the first and the last worker that work on the tile (q0 == q1: the whole tile)
    int seg;     // 0: the pair's share begins in this tile, 1: it began in the tile before
};
__device__ __forceinline__ int tables_share(const TablesParams& p, int pair) {
    return (int)((long long)pair * p.left * p.n_kb / p.share_pairs);
}
__device__ __forceinline__ int tables_owner(const TablesParams& p, int block) {
    const long long T = (long long)p.left * p.n_kb;
    return (int)(((long long)(block + 1) * p.share_pairs + T - 1) / T - 1);
}
__device__ __forceinline__ bool tables_item(const TablesParams& p, int pair, int i, TablesItem& it) {
    if (pair < p.share_pairs) {
        const int x0 = tables_share(p, pair), x1 = tables_share(p, pair + 1);
        const int t = x0 / p.n_kb + i, b0 = t * p.n_kb, b1 = b0 + p.n_kb;
        if (b0 < x1) {
            it.tile = t;
            it.kb0 = x0 > b0 ? x0 - b0 : 0;
            it.kb1 = x1 < b1 ? x1 - b0 : p.n_kb;
            it.seg = i;
            it.q0 = tables_owner(p, b0);
            it.q1 = tables_owner(p, b1 - 1);
            return true;
        }
        i -= (x1 - 1) / p.n_kb - x0 / p.n_kb + 1;
    }
    if (i >= p.full_rounds) return false;
    it.tile = p.left + pair + i * p.pairs;
    it.kb0 = 0;
    it.kb1 = p.n_kb;
    it.q0 = it.q1 = pair;
    return true;
}

// Columns of an accumulator: those of the tile's block of m, a multiple of 32.  (One CTA: W's parts stand one behind the
// other in a stage, copied in boxes of n rows, so n is the same for every block.)
template <bool F32>
__device__ __forceinline__ int tables_n(const TablesParams& p, int mb) {
    if (F32) return p.box_n;
    return ((p.m - mb * 128 < 128 ? p.m - mb * 128 : 128) + 31) & ~31;
}

// W (fp32, [m, E]) -> three bf16 parts [3][m_pad][E_pad], zero where padded
__global__ void __launch_bounds__(256) weight_split_kernel(const float* __restrict__ W, int m, int E, int m_pad, int E_pad,
                                                           __nv_bfloat16* __restrict__ w) {
    pdl_launch_dependents();
    const size_t part = (size_t)m_pad * E_pad;
    const int r = blockIdx.y;
    for (int e = (blockIdx.x * 256 + threadIdx.x) * 2; e < E_pad; e += gridDim.x * 512) {
        const float x0 = (r < m && e < E) ? W[(size_t)r * E + e] : 0.f;
        const float x1 = (r < m && e + 1 < E) ? W[(size_t)r * E + e + 1] : 0.f;
        const __nv_bfloat162 a = __floats2bfloat162_rn(x0, x1);
        const float y0 = x0 - __low2float(a), y1 = x1 - __high2float(a);
        const __nv_bfloat162 b = __floats2bfloat162_rn(y0, y1);
        const __nv_bfloat162 c = __floats2bfloat162_rn(y0 - __low2float(b), y1 - __high2float(b));
        __nv_bfloat16* dst = w + (size_t)r * E_pad + e;
        *(__nv_bfloat162*)dst = a;
        *(__nv_bfloat162*)(dst + part) = b;
        *(__nv_bfloat162*)(dst + 2 * part) = c;
    }
}

// 2^x for a whole number x, as far as fp32 has it
__device__ __forceinline__ float tables_exp2(int x) { return __uint_as_float((uint32_t)(127 + (x < -126 ? -126 : x > 127 ? 127 : x)) << 23); }

// W (fp32, [m, E]) -> two fp16 parts [2][m_pad][E_pad], zero where padded: a row is multiplied by the power of two that takes
// its largest entry to [2^13, 2^14), W1 is what fp16 holds of it and W2 what it holds of the rest, times 2^11.  Every block
// (a row each) also looks at a sample of the embeddings, the same sample: the power of two that takes the median of 256 threads'
// largest entries to [2^8, 2^9) is what they will be multiplied by, so that rows up to 2^8 times larger or smaller stay within fp16's
// exponents.  And clears the flags of rows that do not.
__global__ void __launch_bounds__(256) weight_split16_kernel(const float* __restrict__ W, const float* __restrict__ emb, int V, int m, int E,
                                                           int m_pad, int E_pad, __half* __restrict__ w, float2* __restrict__ unscale,
                                                           float* __restrict__ scale, uint32_t* __restrict__ flags, int n_flags) {
    __shared__ float s_max[8];
    __shared__ int s_hist[256];
    __shared__ int s_mid;
    pdl_launch_dependents();
    const int r = blockIdx.x, tid = threadIdx.x;
    s_hist[tid] = 0;
    if (tid == 0) s_mid = 127 + 8;  // (nothing but zeros: scale 1)
    for (int i = r * 256 + tid; i < n_flags; i += (int)gridDim.x * 256) flags[i] = 0u;
    // the sample: four pieces of 16 bytes a thread, from a row of its own
    float x = 0.f;
    {
        const size_t row = (size_t)((long long)tid * V / 256) * E;
        const int n4 = E / 4;
        float4 v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            v[i] = __ldg((const float4*)(emb + row) + (int)((long long)(tid * 4 + i) * 37 % n4));
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float q[4] = {fabsf(v[i].x), fabsf(v[i].y), fabsf(v[i].z), fabsf(v[i].w)};
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (q[k] < INFINITY) x = fmaxf(x, q[k]);
        }
    }
    // the row's largest finite entry
    float top = 0.f;
    if (r < m)
        for (int e = tid; e < E; e += 256) {
            const float a = fabsf(W[(size_t)r * E + e]);
            if (a < INFINITY) top = fmaxf(top, a);
        }
    top = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(top)));
    if ((tid & 31) == 0) s_max[tid >> 5] = top;
    __syncthreads();
    const int ex = (int)(__float_as_uint(x) >> 23);  // (biased; 0: zero or denormal)
    if (ex > 0) atomicAdd(&s_hist[ex], 1);
#pragma unroll
    for (int i = 0; i < 8; ++i) top = fmaxf(top, s_max[i]);
    __syncthreads();
    if (tid < 32) {
        int own = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) own += s_hist[8 * tid + i];
        int upto = own;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xFFFFFFFFu, upto, d);
            if (tid >= d) upto += o;
        }
        const int half = (__shfl_sync(0xFFFFFFFFu, upto, 31) + 1) / 2;  // the median is where the count reaches this
        if (half > 0 && upto >= half && upto - own < half) {
            int c = upto - own;
            for (int i = 0; i < 8; ++i) {
                c += s_hist[8 * tid + i];
                if (c >= half) {
                    s_mid = 8 * tid + i;
                    break;
                }
            }
        }
    }
    __syncthreads();
    int s = 127 + 8 - s_mid;
    s = s < -120 ? -120 : s > 120 ? 120 : s;
    int k = top > 0.f ? 13 + 127 - (int)(__float_as_uint(top) >> 23) : 0;
    k = k > 126 ? 126 : k;
    if (tid == 0) {
        const int t = -(k + s), t1 = t / 2;
        unscale[r] = make_float2(tables_exp2(t1), tables_exp2(t - t1));
        if (r == 0) *scale = tables_exp2(s);
    }
    const float f = tables_exp2(k);
    const size_t part = (size_t)m_pad * E_pad;
    for (int e = tid * 2; e < E_pad; e += 512) {
        const float x0 = (r < m && e < E) ? W[(size_t)r * E + e] * f : 0.f;
        const float x1 = (r < m && e + 1 < E) ? W[(size_t)r * E + e + 1] * f : 0.f;
        const __half2 a = __floats2half2_rn(x0, x1);
        const __half2 b = __floats2half2_rn((x0 - __low2float(a)) * kTmLow, (x1 - __high2float(a)) * kTmLow);
        __half* dst = w + (size_t)r * E_pad + e;
        *(__half2*)dst = a;
        *(__half2*)(dst + part) = b;
    }
}

__device__ __forceinline__ uint32_t cvt_f16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// two fp32 numbers, scaled -> their two fp16 parts, packed
__device__ __forceinline__ void split2(float x0, float x1, float scale, uint32_t& a, uint32_t& b) {
    const float2 x = __fmul2_rn(make_float2(x0, x1), make_float2(scale, scale));
    a = cvt_f16x2(x.x, x.y);
    const float2 y = __half22float2(*(const __half2*)&a);
    const float2 z = __fmul2_rn(make_float2(x.x - y.x, x.y - y.y), make_float2(kTmLow, kTmLow));
    b = cvt_f16x2(z.x, z.y);
}
// Is a row whose largest magnitude is m held well enough by the two parts, once scaled?  They are off by 2^-36 at most where fp16 has no
// more bits below them: 2^-26 of the largest entry if that is 2^-10 or more.  Or the row is zero.
__device__ __forceinline__ bool tables_row_ok(float m, float scale) {
    return m == 0.f || (m * scale >= 0.0009765625f && m * scale <= 65504.f);
}
__device__ __forceinline__ void st_shared_v4(uint32_t at, const uint32_t (&v)[4]) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}
__device__ __forceinline__ void st_global_v8(float* dst, const float* v) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                 "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}
__device__ __forceinline__ float4 ld_shared_f4(uint32_t at) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(at));
    return v;
}

// fp32 embeddings: results that are worked out again as one chain of fp32 multiply-adds, which gives what fp32 arithmetic gives:
// rows whose entries fp16 parts do not hold well enough (over 2^7 times larger than most rows, or 2^18 times smaller), and whatever is
// not finite (infinities).  They are rare, so the time does not matter.
__device__ __forceinline__ bool tables_finite(float x) { return fabsf(x) <= 3.402823466e38f; }
__device__ __noinline__ float tables_fp32(const TablesParams& p, int v, int c) {
    const float* e = (const float*)p.emb + (size_t)v * p.E;
    const float* w = p.W + (size_t)c * p.E;
    float a = 0.f;
#pragma unroll 8
    for (int k = 0; k < p.E; ++k) a = fmaf(__ldg(e + k), __ldg(w + k), a);
    return a + (p.bias ? p.bias[c] : 0.f);
}

template <bool F32>
__global__ void __cluster_dims__(F32 ? 1 : 2, 1, 1) __launch_bounds__(TablesCfg<F32>::THREADS, 1)
    tables_mma_kernel(const __grid_constant__ TablesParams p) {
    using C = TablesCfg<F32>;
    constexpr uint32_t NS = C::STAGES, NR = C::RAW_STAGES;
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bars[2 * (NS + NR) + 4];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    __shared__ bool s_mend;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = C::PAIR ? cluster_ctarank() : 0u;
    const int pair = C::PAIR ? (int)blockIdx.x >> 1 : (int)blockIdx.x;
    auto wait = [&](uint32_t bar, uint32_t parity) {
        if (C::PAIR)
            mbar_wait_cluster(bar, parity, &s_abort);
        else
            mbar_wait_bounded(bar, parity, &s_abort);
    };
    const uint32_t a_ring = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t w_ring = a_ring + NS * C::A_BYTES, raw_ring = w_ring + NS * C::W_BYTES;
    // full: a block's rows and its W are there (a pair: in both CTAs; the even CTA's barriers), empty: the instructions that read
    // them are done, rfull / rempty: fp32 rows as loaded.  (One barrier for rows and W: the thread that issues the instructions is
    // the bottleneck of short blocks, every wait and every commit costs it a hundred cycles.)
    const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * NS, rfull0 = empty0 + 8 * NS, rempty0 = rfull0 + 8 * NR;
    const uint32_t accfull0 = rempty0 + 8 * NR, accempty0 = accfull0 + 16;
    if (tid == 0) {
        for (uint32_t s = 0; s < NS; ++s) {
            mbar_init(full0 + 8 * s, F32 ? kTmConvWarps / 2 + 1 : 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        for (uint32_t s = 0; s < NR; ++s) {
            mbar_init(rfull0 + 8 * s, 1);
            mbar_init(rempty0 + 8 * s, kTmConvWarps / 2);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(accfull0 + 8 * s, 1);
            mbar_init(accempty0 + 8 * s, (C::PAIR ? 2 : 1) * kTmEpiWarps);  // (the even CTA's)
        }
        mbar_fence_init();
        s_abort = 0;
        s_mend = false;
    }
    pdl_launch_dependents();  // (the kernel that adds up the pieces; it waits for this grid)
    if (warp == 9) tmem_alloc<C::PAIR>(smem_u32(&s_tmem), 512);
    tc_fence_before();
    cluster_sync();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    pdl_wait();  // W's parts come from the kernel ahead

    TablesItem it;
    if (warp < kTmEpiWarps) {
        // ------------------------------ accumulators -> running sums -> output -------------------
        // One row block a CTA: its two accumulator sets take turns, chunk by chunk.  Two row blocks: a set each; one is
        // emptied while the instructions of the other run.
        const int half = warp >> 2, quarter = warp & 3;
        const uint32_t accempty_even = mapa_u32(accempty0, 0);
        uint32_t cc = 0;  // chunks emptied so far
        float2 check = make_float2(0.f, 0.f);  // fp32 embeddings: NaN once a result of this thread was not finite
        for (int i = 0; tables_item(p, pair, i, it); ++i) {
            const int rt = it.tile / p.n_mb, mb = it.tile - rt * p.n_mb;
            const uint32_t n = (uint32_t)tables_n<F32>(p, mb);
            float acc[C::MT][64];
#pragma unroll
            for (int h = 0; h < C::MT; ++h)
#pragma unroll
                for (int c = 0; c < 64; ++c) acc[h][c] = 0.f;
            for (int kb = it.kb0; kb < it.kb1; kb += C::CHUNK, ++cc) {
#pragma unroll
                for (int h = 0; h < C::MT; ++h) {
                    const uint32_t slot = C::MT == 1 ? (cc & 1u) : (uint32_t)h;
                    wait(accfull0 + 8 * slot, (C::MT == 1 ? cc >> 1 : cc) & 1u);
                    tc_fence_after();
                    const uint32_t t0 = tmem + ((uint32_t)(32 * quarter) << 16) + slot * 256u + (uint32_t)half * 64u;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
#pragma unroll
                        for (int lo = 0; lo < 2; ++lo) {
                            uint32_t d[16];
                            tmem_ld_32x16(t0 + n * lo + 16u * q, d);
                            tmem_wait_ld();
#pragma unroll
                            for (int c = 0; c < 16; ++c) {
                                const float x = __uint_as_float(d[c]);
                                acc[h][16 * q + c] = F32 && lo ? fmaf(x, 1.0f / kTmLow, acc[h][16 * q + c]) : acc[h][16 * q + c] + x;
                            }
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        if (C::PAIR)
                            mbar_arrive_cluster(accempty_even + 8 * slot);
                        else
                            mbar_arrive(accempty0 + 8 * slot);
                    }
                }
            }
            // a piece of a left-over tile goes to scratch, [ROWS][128], without the bias
            const bool piece = it.q0 != it.q1;
            const int ld = piece ? 128 : p.m, rows = piece ? C::ROWS : p.V - rt * C::ROWS, cols = piece ? 64 : p.m - mb * 128 - half * 64;
            const bool wide = piece || p.wide;
            float* base = piece ? p.pieces + (size_t)(pair * 2 + it.seg) * C::ROWS * 128
                                : p.out + (size_t)rt * C::ROWS * p.m + mb * 128;
            const float* bias = piece || p.bias == nullptr ? nullptr : p.bias + mb * 128 + half * 64;
#pragma unroll
            for (int h = 0; h < C::MT; ++h) {
                const int v = h * 256 + (int)rank * 128 + quarter * 32 + lane;
                if (v < rows) {
                    float* dst = base + (size_t)v * ld + half * 64;
#pragma unroll
                    for (int c = 0; c < 64; c += 8) {
                        if (c >= cols) break;
                        const bool both = c + 4 < cols;
                        if (F32) {
#pragma unroll
                            for (int k = 0; k < 8; ++k) {
                                const float2 f = __ldg(p.unscale + mb * 128 + half * 64 + c + k);
                                acc[h][c + k] = acc[h][c + k] * f.x * f.y;
                            }
                        }
                        if (bias) {
#pragma unroll
                            for (int k = 0; k < 8; ++k)
                                if (k < 4 || both) acc[h][c + k] += __ldg(bias + c + k);
                        }
                        if (F32 && !piece) {
#pragma unroll
                            for (int k = 0; k < 8; k += 2)
                                if (k < 4 || both)
                                    check = __ffma2_rn(make_float2(0.f, 0.f), make_float2(acc[h][c + k], acc[h][c + k + 1]), check);
                        }
                        if (wide) {  // (both: m is a multiple of 8)
                            st_global_v8(dst + c, &acc[h][c]);
                        } else {
                            *(float4*)(dst + c) = make_float4(acc[h][c], acc[h][c + 1], acc[h][c + 2], acc[h][c + 3]);
                            if (both)
                                *(float4*)(dst + c + 4) = make_float4(acc[h][c + 4], acc[h][c + 5], acc[h][c + 6], acc[h][c + 7]);
                        }
                    }
                }
            }
        }
        if (F32) {  // (nothing waits for these warps any more)
            if (check.x + check.y != 0.f) s_mend = true;
            __syncwarp();
            named_bar_sync(1, (kTmEpiWarps + kTmConvWarps) * 32);  // (the tiles are written, their rows looked at)
            if (s_mend && !s_abort) {
                for (int i = 0; tables_item(p, pair, i, it); ++i) {
                    if (it.q0 != it.q1) continue;  // (pieces: the kernel that adds them up)
                    const int rt = it.tile / p.n_mb, c0 = (it.tile - rt * p.n_mb) * 128;
                    for (int v = rt * C::ROWS + warp; v < p.V && v < (rt + 1) * C::ROWS; v += kTmEpiWarps) {
                        const bool bad = p.bad_row[(size_t)it.tile * C::ROWS + (v - rt * C::ROWS)] != 0;
                        for (int c = c0 + lane; c < p.m && c < c0 + 128; c += 32) {
                            float* o = p.out + (size_t)v * p.m + c;
                            if (bad || !tables_finite(*o)) *o = tables_fp32(p, v, c);
                        }
                    }
                }
            }
        }
    } else if (warp == 8) {
        // ------------------------------ TMA loads: W, bf16 embeddings ----------------------------
        if (lane == 0) {
            const uint32_t full_even = mapa_u32(full0, 0);
            TablesRing<NS> w(1);
            for (int i = 0; tables_item(p, pair, i, it); ++i) {
                const int rt = it.tile / p.n_mb, mb = it.tile - rt * p.n_mb;
                const int n = tables_n<F32>(p, mb);
                const int w12 = (int)rank * p.m_pad + mb * 128, w3 = 2 * p.m_pad + mb * 128 + (int)rank * (n >> 1);
                for (int kb = it.kb0; kb < it.kb1; ++kb) {
                    const int x = kb * C::BLK;
                    if (w.t >= NS) wait(empty0 + 8 * w.st, w.ph);
                    if (s_abort) break;  // (no copy is started any more)
                    const uint32_t da = a_ring + w.st * C::A_BYTES, dw = w_ring + w.st * C::W_BYTES;
                    if (C::PAIR) {
                        const uint32_t fb = full_even + 8 * w.st;
                        if (rank == 0) mbar_arrive_expect_tx(full0 + 8 * w.st, 2u * (C::A_BYTES + C::W_BYTES));
#pragma unroll
                        for (int h = 0; h < C::MT; ++h)
                            tma_load_2d_pair(da + h * C::PART, &p.map_e, x, rt * C::ROWS + h * 256 + (int)rank * 128, fb);
                        tma_load_2d_pair(dw, &p.map_w, x, w12, fb);
                        tma_load_2d_pair(dw + C::W_BYTES / 3, &p.map_w, x, w12 + 64, fb);
                        tma_load_2d_pair(dw + 2 * (C::W_BYTES / 3), &p.map_w, x, w3, fb);
                    } else {
                        const uint32_t part = (uint32_t)n * C::BLK * 2;
                        mbar_arrive_expect_tx(full0 + 8 * w.st, 2u * part);
#pragma unroll
                        for (int j = 0; j < 2; ++j)
                            tma_load_2d(dw + j * part, &p.map_w, x, j * p.m_pad + mb * 128, full0 + 8 * w.st);
                    }
                    w.next();
                }
            }
            // the last arrivals from the other CTA have come before this CTA retires; after an abort: no copy of the pair
            // is in flight any more
            w.drain(empty0, rank == 0 ? full0 : 0u, &s_abort);
        }
    } else if (warp == 9) {
        // ------------------------------ matrix instructions --------------------------------------
        if (rank == 0 && lane == 0) {
            TablesRing<NS> w(0);
            uint32_t cc = 0;
            for (int i = 0; tables_item(p, pair, i, it); ++i) {
                const int mb = it.tile % p.n_mb;
                const int n = tables_n<F32>(p, mb);
                constexpr int M = C::PAIR ? 256 : 128;
                const uint32_t idesc2 = umma_idesc(M, 2 * n, !F32), idesc1 = umma_idesc(M, n, !F32);
                constexpr uint32_t o_w3 = 2 * (C::W_BYTES / 3);  // (bf16)
                // A pair takes two blocks at a time.  An instruction whose accumulator columns the one just ahead of it wrote waits
                // for those, so with two row blocks their instructions alternate, except in the first and the last two blocks of a
                // chunk, where the first row block goes ahead: its accumulators are emptied (or were) while the second's are filled.
                constexpr int G = C::MT;
                for (int kb = it.kb0; kb < it.kb1; kb += G) {
                    const int g = kb + G <= it.kb1 ? G : it.kb1 - kb;
                    const bool first = (kb - it.kb0) % C::CHUNK == 0;
                    const bool last = kb + g == it.kb1 || (kb + g - it.kb0) % C::CHUNK == 0;
                    uint32_t a0[G], b0[G], done[G];
#pragma unroll
                    for (int k = 0; k < G; ++k) {
                        if (k >= g) break;
                        wait(full0 + 8 * w.st, w.ph);
                        a0[k] = a_ring + w.st * C::A_BYTES;
                        b0[k] = w_ring + w.st * C::W_BYTES;
                        done[k] = empty0 + 8 * w.st;
                        w.next();
                    }
                    tc_fence_after();
                    auto mma = [&](int k, int h, int ks, bool small) {
                        const uint32_t d = tmem + (C::MT == 1 ? (cc & 1u) : (uint32_t)h) * 256u;
                        const uint64_t a1 = C::desc(a0[k] + h * C::PART + 32 * ks), w12 = C::desc(b0[k] + 32 * ks);
                        if (!small)
                            umma<C::PAIR>(d, a1, w12, idesc2, !first || k > 0 || ks > 0);
                        else if (F32)  // (the second part of the embeddings times W1)
                            umma<C::PAIR>(d + (uint32_t)n, C::desc(a0[k] + C::PART + 32 * ks), w12, idesc1, true);
                        else
                            umma<C::PAIR>(d + (uint32_t)n, a1, C::desc(b0[k] + o_w3 + 32 * ks), idesc1, true);
                    };
                    if (C::MT == 2 && !first && !last) {
                        if (!s_abort) {
#pragma unroll
                            for (int k = 0; k < G; ++k) {
                                if (k >= g) break;
#pragma unroll
                                for (int ks = 0; ks < C::BLK / 16; ++ks) {
                                    mma(k, 0, ks, false);
                                    mma(k, 1, ks, false);
                                    mma(k, 0, ks, true);
                                    mma(k, 1, ks, true);
                                }
                            }
                        }
                    } else {
#pragma unroll
                        for (int h = 0; h < C::MT; ++h) {
                            const uint32_t slot = C::MT == 1 ? (cc & 1u) : (uint32_t)h;
                            const uint32_t turn = C::MT == 1 ? cc >> 1 : cc;  // how often the set has been filled before
                            if (first && turn >= 1) {
                                wait(accempty0 + 8 * slot, (turn - 1u) & 1u);
                                tc_fence_after();
                            }
                            if (!s_abort) {
#pragma unroll
                                for (int k = 0; k < G; ++k) {
                                    if (k >= g) break;
#pragma unroll
                                    for (int ks = 0; ks < C::BLK / 16; ++ks) {
                                        mma(k, h, ks, false);
                                        mma(k, h, ks, true);
                                    }
                                }
                            }
                            if (last) umma_commit<C::PAIR>(accfull0 + 8 * slot);
                        }
                    }
#pragma unroll
                    for (int k = 0; k < G; ++k) {
                        if (k >= g) break;
                        umma_commit<C::PAIR>(done[k]);
                    }
                    if (last) ++cc;
                }
            }
        }
    } else if (F32 && warp == 10) {
        // ------------------------------ TMA loads: fp32 embeddings -------------------------------
        if (lane == 0) {
            TablesRing<NR> r(1);
            for (int i = 0; tables_item(p, pair, i, it); ++i) {
                const int row = it.tile / p.n_mb * C::ROWS + (int)rank * 128;
                for (int kb = it.kb0; kb < it.kb1; ++kb) {
                    if (r.t >= NR) wait(rempty0 + 8 * r.st, r.ph);
                    if (s_abort) break;
                    mbar_arrive_expect_tx(rfull0 + 8 * r.st, C::RAW);
                    tma_load_2d(raw_ring + r.st * C::RAW, &p.map_e, kb * C::BLK, row, rfull0 + 8 * r.st);
                    r.next();
                }
            }
            r.drain(rempty0, rfull0, &s_abort);
        }
    } else if (F32) {
        // ------------------------------ fp32 embeddings -> fp16 parts ----------------------------
        // four warps take the even blocks, four the odd ones: a block is a chain of waits and round trips.  A wait on a barrier's parity
        // tells a phase from the ones beside it and not from the one two before, so a half has to wait for every phase of the
        // barriers that it waits on: with an even number of stages every stage is always the same half's.  (Four raw stages or six: V =
        // 32,000, E = 2048, two towers 208.4 and 209.3 us.)
        static_assert(!F32 || (NR % 2 == 0 && NS % 2 == 0), "a stage of either ring belongs to one half of the converting warps");
        const int ct = (tid - (kTmEpiWarps + 3) * 32) & 127, half = (tid - (kTmEpiWarps + 3) * 32) >> 7;
        const int c8 = ct & 3, r0 = ct >> 2;  // columns 8 c8 .. 8 c8 + 7 of rows r0, r0 + 32, r0 + 64 and r0 + 96
        const float scale = *p.scale;
        TablesRing<NS> a(1);
        TablesRing<NR> r(0);
        for (int i = 0; tables_item(p, pair, i, it); ++i) {
            float most[4] = {0.f, 0.f, 0.f, 0.f};  // the largest magnitudes of the rows
            for (int kb = it.kb0; kb < it.kb1; ++kb, a.next(), r.next()) {
                if ((int)(a.t & 1u) != half) continue;
                wait(rfull0 + 8 * r.st, r.ph);
                const uint32_t src = raw_ring + r.st * C::RAW;
                float4 x[4][2];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int row = r0 + 32 * q;
#pragma unroll
                    for (int h = 0; h < 2; ++h)  // (128-byte rows in the 128-byte swizzle)
                        x[q][h] = ld_shared_f4(src + (uint32_t)row * 128u + (uint32_t)(((2 * c8 + h) ^ (row & 7)) * 16));
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(rempty0 + 8 * r.st);
                if (a.t >= NS) wait(empty0 + 8 * a.st, a.ph);
                const uint32_t dst = a_ring + a.st * C::A_BYTES;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int row = r0 + 32 * q;  // (64-byte rows in the 64-byte swizzle)
                    const uint32_t at = dst + (uint32_t)row * 64u + (uint32_t)((c8 ^ ((row >> 1) & 3)) * 16);
                    uint32_t b1[4], b2[4];
                    split2(x[q][0].x, x[q][0].y, scale, b1[0], b2[0]);
                    split2(x[q][0].z, x[q][0].w, scale, b1[1], b2[1]);
                    split2(x[q][1].x, x[q][1].y, scale, b1[2], b2[2]);
                    split2(x[q][1].z, x[q][1].w, scale, b1[3], b2[3]);
                    st_shared_v4(at, b1);
                    st_shared_v4(at + C::PART, b2);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        most[q] = fmaxf(most[q], fmaxf(fabsf(x[q][h].x), fabsf(x[q][h].y)));
                        most[q] = fmaxf(most[q], fmaxf(fabsf(x[q][h].z), fabsf(x[q][h].w)));
                    }
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(full0 + 8 * a.st);
            }
            // rows that fp16 does not hold well enough (in this thread's blocks)
            const int rt = it.tile / p.n_mb;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float mx = fmaxf(most[q], __shfl_xor_sync(0xFFFFFFFFu, most[q], 1));
                mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 2));
                const int v = rt * C::ROWS + r0 + 32 * q;
                if (c8 == 0 && v < p.V && !tables_row_ok(mx, scale)) {
                    p.bad_row[(size_t)it.tile * C::ROWS + r0 + 32 * q] = 1;
                    if (it.q0 == it.q1) s_mend = true;
                }
            }
        }
        a.drain(empty0, 0u, &s_abort);
        __threadfence_block();  // (the flags, for the warps that write the tiles)
        __syncwarp();
        asm volatile("bar.arrive 1, %0;" ::"n"((kTmEpiWarps + kTmConvWarps) * 32) : "memory");
    }
    __syncwarp();
    tc_fence_before();
    cluster_sync();  // (the other CTA's last arrivals on this CTA's barriers, and its reads of this CTA's memory, are done)
    tc_fence_after();
    if (warp == 9) tmem_free<C::PAIR>(tmem, 512);
    if (tid == 0 && s_abort) atomicOr(p.errflag, 1);
}

// The left-over tiles' pieces, added up in order: one thread per four columns of a row.
template <bool F32>
__global__ void __launch_bounds__(256) tables_pieces_kernel(const __grid_constant__ TablesParams p) {
    using C = TablesCfg<F32>;
    pdl_wait();
    const int tile = (int)blockIdx.y, rt = tile / p.n_mb, mb = tile - rt * p.n_mb;
    const int q0 = tables_owner(p, tile * p.n_kb), q1 = tables_owner(p, (tile + 1) * p.n_kb - 1);
    const int v = (int)blockIdx.x * 8 + (threadIdx.x >> 5), c = (threadIdx.x & 31) * 4;
    if (q0 == q1 || rt * C::ROWS + v >= p.V || mb * 128 + c >= p.m) return;  // (q0 == q1: written whole)
    const bool bad = F32 && p.bad_row[(size_t)tile * C::ROWS + v] != 0;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int q = q0; q <= q1; ++q) {
        const int seg = tables_share(p, q) < tile * p.n_kb ? 1 : 0;
        const float4 x = __ldcs((const float4*)(p.pieces + ((size_t)(q * 2 + seg) * C::ROWS + v) * 128 + c));
        s.x += x.x, s.y += x.y, s.z += x.z, s.w += x.w;
    }
    if (p.bias) {
        const float* b = p.bias + mb * 128 + c;
        s.x += b[0], s.y += b[1], s.z += b[2], s.w += b[3];
    }
    const int row = rt * C::ROWS + v, col = mb * 128 + c;
    if (F32 && (bad || fmaf(0.f, s.x, fmaf(0.f, s.y, fmaf(0.f, s.z, 0.f * s.w))) != 0.f)) {
        if (bad || !tables_finite(s.x)) s.x = tables_fp32(p, row, col);
        if (bad || !tables_finite(s.y)) s.y = tables_fp32(p, row, col + 1);
        if (bad || !tables_finite(s.z)) s.z = tables_fp32(p, row, col + 2);
        if (bad || !tables_finite(s.w)) s.w = tables_fp32(p, row, col + 3);
    }
    *(float4*)(p.out + (size_t)row * p.m + col) = s;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled() {
    static const EncodeTiledFn fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            return (EncodeTiledFn) nullptr;
        }
        return (EncodeTiledFn)f;
    }();
    return fn;
}
// [rows, cols], boxes of box_rows rows of box_bytes, in the swizzle of that width, zeros outside
bool encode_map(CUtensorMap* map, const void* base, CUtensorMapDataType type, uint64_t rows, uint64_t cols, uint32_t box_rows, uint32_t box_bytes) {
    const uint32_t esz = type == CU_TENSOR_MAP_DATA_TYPE_FLOAT32 ? 4 : 2;
    const cuuint64_t dims[2] = {cols, rows}, strides[1] = {cols * esz};
    const cuuint32_t box[2] = {box_bytes / esz, box_rows}, step[2] = {1, 1};
    return encode_tiled()(map, type, 2,
                          const_cast<void*>(base), dims, strides, box, step, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          box_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct TablesSizes {
    int n_mb, m_pad, E_pad, pairs;
    size_t o_w, o_unscale, o_scale, o_bad, n_bad, total;  // (fp32 only: from o_unscale on)
};
TablesSizes tables_sizes(int num_sms, int V, int E, int m, bool f32) {
    TablesSizes s;
    s.n_mb = (m + 127) / 128;
    s.m_pad = 128 * s.n_mb;
    s.E_pad = (E + 63) / 64 * 64;
    s.pairs = f32 ? num_sms : num_sms / 2;
    s.o_w = (size_t)s.pairs * 2 * (f32 ? TablesCfg<true>::ROWS : TablesCfg<false>::ROWS) * 128 * sizeof(float);
    s.o_unscale = s.o_w + (size_t)(f32 ? 2 : 3) * s.m_pad * s.E_pad * 2;
    s.o_scale = s.o_unscale + (f32 ? (size_t)s.m_pad * sizeof(float2) : 0);
    s.o_bad = s.o_scale + (f32 ? 256 : 0);
    s.n_bad = f32 ? (size_t)(V + TablesCfg<true>::ROWS - 1) / TablesCfg<true>::ROWS * s.n_mb * TablesCfg<true>::ROWS : 0;
    s.total = s.o_bad + s.n_bad;
    return s;
}
template <bool F32>
cudaError_t tables_run(const TablesParams& p, cudaStream_t st, int* launches) {
    using C = TablesCfg<F32>;
    cudaError_t e = cudaFuncSetAttribute(tables_mma_kernel<F32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
    if (e == cudaSuccess) e = launch_pdl(tables_mma_kernel<F32>, dim3((C::PAIR ? 2 : 1) * p.pairs), dim3(C::THREADS), C::SMEM, st, p);
    *launches += 1;
    if (e == cudaSuccess && p.share_pairs > p.left) {
        e = launch_pdl(tables_pieces_kernel<F32>, dim3(C::ROWS / 8, p.left), dim3(256), 0, st, p);
        *launches += 1;
    }
    return e;
}

}  // namespace

// Can the tensor cores take this table?  16-byte rows for the loads and stores; anything else goes to the FMA kernel.
bool tables_mma_fits(const void* d_emb, graft_dtype dt, int E, const void* d_out) {
    return E % (dt == GRAFT_BF16 ? 8 : 4) == 0 && (((uintptr_t)d_emb | (uintptr_t)d_out) & 15) == 0 && encode_tiled() != nullptr;
}
size_t tables_mma_scratch_bytes(int num_sms, int V, int E, int m, graft_dtype dt) {
    return tables_sizes(num_sms, V, E, m, dt == GRAFT_F32).total;
}

// out [V, m] = emb [V, E] . W^T + bias.  scratch: tables_mma_scratch_bytes, 256-byte aligned.
cudaError_t tables_mma_launch(graft_ctx* ctx, const void* d_emb, graft_dtype dt, int E, const float* d_W, const float* d_b,
                              float* d_out, void* scratch, cudaStream_t st) {
    const int V = ctx->cfg.V, m = ctx->cfg.m;
    const bool f32 = dt == GRAFT_F32;
    const TablesSizes s = tables_sizes(ctx->num_sms, V, E, m, f32);
    void* w = (char*)scratch + s.o_w;
    TablesParams p;
    const int blk = f32 ? TablesCfg<true>::BLK : TablesCfg<false>::BLK;
    p.box_n = s.n_mb > 1 ? 128 : (m + 31) / 32 * 32;
    if (!encode_map(&p.map_w, w, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16,
                    (uint64_t)(f32 ? 2 : 3) * s.m_pad, s.E_pad, f32 ? p.box_n : 64, 2 * blk) ||
        !encode_map(&p.map_e, d_emb, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, V, E, 128, 128))
        return cudaErrorUnknown;
    p.emb = d_emb;
    p.W = d_W;
    p.bias = d_b;
    p.out = d_out;
    p.pieces = (float*)scratch;
    p.unscale = (const float2*)((char*)scratch + s.o_unscale);
    p.scale = (const float*)((char*)scratch + s.o_scale);
    p.bad_row = (uint8_t*)scratch + s.o_bad;
    p.errflag = ctx->w_errflag;
    p.V = V;
    p.E = E;
    p.m = m;
    p.m_pad = s.m_pad;
    p.n_mb = s.n_mb;
    p.n_kb = (E + blk - 1) / blk;
    p.pairs = s.pairs;
    const int rows = f32 ? TablesCfg<true>::ROWS : TablesCfg<false>::ROWS;
    const int tiles = (V + rows - 1) / rows * s.n_mb;
    p.full_rounds = tiles / s.pairs;
    p.left = tiles - p.full_rounds * s.pairs;
    // a share of the left-over tiles: at least a sixteenth of a tile and 256 columns, at most a tile
    long long sp = s.pairs;
    if (sp > (long long)p.left * kTmMaxSplit) sp = (long long)p.left * kTmMaxSplit;
    if (sp > (long long)p.left * p.n_kb * blk / 256) sp = (long long)p.left * p.n_kb * blk / 256;
    if (sp > p.left) {
        // Shares of equal length that cut tiles anywhere, or a whole number q of shares a tile on fewer workers?  A share that
        // lies in two tiles empties its accumulators and writes a piece twice, and with q = 1 nothing has to be added up:
        // the whole number saves 6 us on pairs and 3 us on single CTAs, 22 and 10 us for q = 1, and costs 0.02 and 0.03 us
        // for every column of E by which a share gets longer.  (Measured over 26 to 73 and 52 to 147 tiles left, E = 1024 to
        // 4096, with and without a round of whole tiles ahead.  V = 16,000, bf16: E = 1024 35.0 -> 29.2 us, E = 4096 61.5 ->
        // 57.9; V = 32,000, E = 1024: bf16 47.5 -> 32.7, fp32 71.9 -> 68.4; fp32, E = 2048 stays: 118.7 against 121.2.)
        const long long q = sp / p.left;
        const double longer = (1.0 / (double)q - (double)p.left / (double)sp) * E;
        if (longer <= (f32 ? (q == 1 ? 380 : 130) : (q == 1 ? 850 : 350))) sp = q * p.left;
    }
    p.share_pairs = (int)(sp < p.left ? p.left : sp);
    p.wide = m % 8 == 0 && ((uintptr_t)d_out & 31) == 0;
    if (f32)
        weight_split16_kernel<<<s.m_pad, 256, 0, st>>>(d_W, (const float*)d_emb, V, m, E, s.m_pad, s.E_pad, (__half*)w,
                                                       (float2*)((char*)scratch + s.o_unscale), (float*)((char*)scratch + s.o_scale),
                                                       (uint32_t*)p.bad_row, (int)(s.n_bad / 4));
    else
        weight_split_kernel<<<dim3((s.E_pad + 511) / 512, s.m_pad), 256, 0, st>>>(d_W, m, E, s.m_pad, s.E_pad, (__nv_bfloat16*)w);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    int launches = 1;
    e = f32 ? tables_run<true>(p, st, &launches) : tables_run<false>(p, st, &launches);
    ctx->launches += (uint64_t)launches;
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace graft

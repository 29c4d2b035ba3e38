// Table precompute on the tensor cores: out[v] = W e_v + b (text after Eq. 6: the projections depend only on the token
// id and are computed once).  This is the one dense contraction of the method, [V, E] x [E, m].
//
// Operands are 16-bit parts of the inputs; products of parts are exact in the fp32 accumulator.
//   bf16 embeddings: out = e W1 + e W2 + e W3, W as three bf16 parts (8 + 8 + 8 mantissa bits; three products a step)
//   fp32 embeddings: out = e1 W1 + (e1 W2 + e2 W1), both as two fp16 parts (11 + 11 bits and the second part's sign; what is
//     dropped, e2 W2, is below 2^-22 of a term, 2^-24.6 root mean square).  fp16 has few exponents, so a row of W is scaled by
//     its largest entry and a row of the embeddings by the largest of its first block; second parts are kept times 2^11, and go to
//     an accumulator of their own (H. Ootomo and R. Yokota, "Recovering single precision accuracy from Tensor Cores while surpassing
//     the FP32 theoretical peak performance", 2022).  Rows of the embeddings that this does not suit are worked out in fp32.
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
//   warps 0-7    empty the accumulators (TMEM, two sets of 2 x 128 columns; fp32: kTmLo), keep the running sums and write the tile
//   warp 8       TMA loads: W's parts (split once per call into scratch by a small kernel), bf16 embeddings
//   warp 9       issues the matrix instructions
//   warp 10      fp32 only: TMA loads of the raw rows;  warps 11-18  raw rows -> fp16 parts in TMEM, a thread a row
// W1 and W2 stand side by side as one operand of N = 256, the third product is an N = 128 of its own (three of N = 128 in a row on one
// accumulator took 122 cycles each: an instruction waits for the one ahead of it on the same columns).  Tiles of 512
// rows halve the passes over W, which comes from L2 every time.  The fp32 kernel works on single CTAs because its rows
// go through threads: telling the other CTA of a pair about every block cost more (136 - 160 us at V = 32,000, E = 2048)
// than the second CTA's half of W saves (120 us).  The embeddings are read from memory once; nothing but the tables is
// written.  What is left when the tiles do not divide by the workers is dealt out along E in shares, whose sums a
// small kernel adds up in order (summing them inside, by the warp that came last, stalled its tile: 462 against 370 us).
//
// Measured (one tower, back to back, B200): V = 151,936, E = 4096, m = 128, bf16: 358 us (376 before rows and W shared a barrier
// and the first row block went two blocks ahead where accumulators are emptied; 798 us with the library template's GEMMs); its products
// take 287 us at the measured dense rate, and the clock falls to 1.5 GHz on the way.  V = 32,000, E = 2048, fp32: 76 us (89 with the
// parts in shared memory and one thread in the issuing loop; 120 with three bf16 parts, seven products; 1135 us by the FMA
// kernel).  What bounds the fp32 kernel: the issuing warp, 1.05 k cycles for two blocks of 32 columns beside 0.77 k of products (910
// cycles a block by one thread, whose operands had to be moved for every instruction), and 0.5 k more where a chunk ends; then
// the pieces, 7 us, and W's parts, 3 us.  The parts go through TMEM because in shared memory the copies, the conversion and the
// products' reads together moved 104 KB a block, 0.8 k cycles of its bandwidth; now 72.  Error against fp64 products at those
// sizes, largest and root mean square over the results' size: bf16 3.4e-6 and 4.8e-7 (FMA kernel 1.7e-5, 1.1e-6); fp32 2.2e-6 and
// 3.5e-7 (three bf16 parts 3.3e-6, 4.7e-7; FMA kernel 9.2e-6, 8.1e-7).  The accumulators round towards zero, so terms of one sign
// are off by more: fp32 1.5e-6 and 1.1e-6 (8.0e-7 and 3.9e-7; 3.6e-6 and 6.5e-7), emptied every 8 additions 8.5e-7 and 4.7e-7 in 93
// us instead of 89.
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
    static constexpr int A_BYTES = F32 ? 0 : 2 * PART;        // a block's embeddings: two row blocks (fp32: two parts, in TMEM)
    static constexpr int W_BYTES = (F32 ? 256 : 192) * BLK * 2;  // a block's W; a pair: W1 (even CTA) or W2 (odd), half of W3
    static constexpr int RAW = 128 * BLK * 4;                 // a block's fp32 embeddings
    static constexpr int STAGES = 4, RAW_STAGES = F32 ? 8 : 1;  // (a stage: a block's embeddings and W)
    static constexpr int THREADS = (kTmEpiWarps + 2 + (F32 ? 1 + kTmConvWarps : 0)) * 32;
    // (the rings start on a 1024-byte boundary)
    static constexpr size_t SMEM = (size_t)STAGES * (A_BYTES + W_BYTES) + (F32 ? (size_t)RAW_STAGES * RAW : 0) + 1024;
};

constexpr float kTmLow = 2048.0f;  // fp16: second parts are kept times 2^11
// fp32 embeddings: a row is multiplied by the power of two that takes the largest entry of its first block (in a piece of a tile: of the
// piece's first block) to [16, 32).  Two parts hold a number up to 65504 to 2^-23 of it or to 2^-36, whichever is more; where the
// largest of eight entries side by side is 2^-12 or more, that is 2^-23 of themselves or 2^-24 of that largest.  So the rest of a row may
// be 2^11 times larger than its first block, and any eight entries 2^16 times smaller.  (With one scale for the table, one column 300
// times larger than the others left 40 % of the rows to be worked out again.)
constexpr int kTmTarget = 4;
constexpr float kTmLeast = 0x1p-12f, kTmMost = 65504.f;
constexpr uint32_t kTmScales = 4;  // tiles whose rows' scales are kept

// fp32 embeddings, columns of TMEM: the small products' accumulator (emptied once a tile) with the large products' on either
// side, which take turns from chunk to chunk, so that one instruction of twice the width fills both -- W1 before W2, or behind it --
// and the stages of the embeddings' parts.
constexpr uint32_t kTmLo = 128, kTmParts = 384;
__device__ __forceinline__ uint32_t tables_hi(uint32_t slot, uint32_t n) { return slot ? kTmLo + n : kTmLo - n; }

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
__device__ __forceinline__ int tables_share(const TablesParams& p, int pair) {  // (32 bits: tables_mma_fits)
    return (int)((uint32_t)pair * (uint32_t)(p.left * p.n_kb) / (uint32_t)p.share_pairs);
}
__device__ __forceinline__ int tables_owner(const TablesParams& p, int block) {
    const uint32_t T = (uint32_t)(p.left * p.n_kb);
    return (int)(((uint32_t)(block + 1) * (uint32_t)p.share_pairs + T - 1) / T - 1);
}
// A pair's share, worked out once (by one thread, while the kernel ahead runs): a dozen divisions took the start of every role
// 5 k cycles.
struct TablesShare {
    int n;           // tiles that it lies in
    TablesItem it[2];
};
__device__ __forceinline__ void tables_shares(const TablesParams& p, int pair, TablesShare& s) {
    s.n = 0;
    if (pair >= p.share_pairs) return;
    const int x0 = tables_share(p, pair), x1 = tables_share(p, pair + 1);
    for (int t = x0 / p.n_kb; t * p.n_kb < x1 && s.n < 2; ++t) {
        const int b0 = t * p.n_kb, b1 = b0 + p.n_kb;
        TablesItem& it = s.it[s.n];
        it.tile = t;
        it.kb0 = x0 > b0 ? x0 - b0 : 0;
        it.kb1 = x1 < b1 ? x1 - b0 : p.n_kb;
        it.seg = s.n++;
        it.q0 = tables_owner(p, b0);
        it.q1 = tables_owner(p, b1 - 1);
    }
}
__device__ __forceinline__ bool tables_item(const TablesParams& p, const TablesShare& s, int pair, int i, TablesItem& it) {
    if (i < s.n) {
        it = s.it[i];
        return true;
    }
    i -= s.n;
    if (i >= p.full_rounds) return false;
    it.tile = p.left + pair + i * p.pairs;
    it.kb0 = 0;
    it.kb1 = p.n_kb;
    it.q0 = it.q1 = pair;
    it.seg = 0;
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
struct SplitParams {
    const float* W;
    int m, E, m_pad, E_pad;
    void* w;
    float2* unscale;  // fp32 embeddings only, as the rest
    uint32_t* flags;
    int n_flags;
};
__global__ void __launch_bounds__(256) weight_split_kernel(const SplitParams sp) {
    const float* __restrict__ W = sp.W;
    const int m = sp.m, E = sp.E, m_pad = sp.m_pad, E_pad = sp.E_pad;
    __nv_bfloat16* __restrict__ w = (__nv_bfloat16*)sp.w;
    pdl_launch_dependents();
    pdl_wait();  // (W may come from the kernel ahead, and a table before this one may still be read from the scratch)
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
// What a row is multiplied by whose first block's largest magnitude is m (zero: 1)
__device__ __forceinline__ float tables_row_scale(float m) {
    const int s = m > 0.f ? 127 + kTmTarget - (int)(__float_as_uint(m) >> 23) : 0;
    return tables_exp2(s < -120 ? -120 : s > 120 ? 120 : s);
}
// 2^-s as a product of two factors: results are multiplied by a row's and a column's, and none of the steps leaves fp32 before the result does
__device__ __forceinline__ float2 tables_unscale(int s) { return make_float2(tables_exp2(-s / 2), tables_exp2(-s - -s / 2)); }

// W (fp32, [m, E]) -> two fp16 parts [2][m_pad][E_pad], zero where padded: a row is multiplied by the power of two that takes
// its largest entry to [2^13, 2^14), W1 is what fp16 holds of it and W2 what it holds of the rest, times 2^11.  A block a row.  And
// clears the flags of the embeddings' rows.
__global__ void __launch_bounds__(256) weight_split16_kernel(const SplitParams sp) {
    __shared__ float s_max[8];
    const float* __restrict__ W = sp.W;
    const int m = sp.m, E = sp.E, m_pad = sp.m_pad, E_pad = sp.E_pad, n_flags = sp.n_flags;
    __half* __restrict__ w = (__half*)sp.w;
    float2* __restrict__ unscale = sp.unscale;
    uint32_t* __restrict__ flags = sp.flags;
    pdl_launch_dependents();
    pdl_wait();  // (as above)
    const int r = blockIdx.x, tid = threadIdx.x;
    // the row's largest finite entry; up to E = 4096 the row stays in registers
    constexpr int N = 16;
    const float* const src = W + (size_t)(r < m ? r : 0) * E;
    const bool kept = E <= N * 256;
    float x[N], top = 0.f;
#pragma unroll
    for (int i = 0; i < N; ++i) x[i] = r < m && tid + 256 * i < E ? src[tid + 256 * i] : 0.f;
#pragma unroll
    for (int i = 0; i < N; ++i) top = fmaxf(top, fabsf(x[i]) < INFINITY ? fabsf(x[i]) : 0.f);
    if (r < m && !kept)
        for (int e = N * 256 + tid; e < E; e += 256) top = fmaxf(top, fabsf(src[e]) < INFINITY ? fabsf(src[e]) : 0.f);
    for (int i = r * 256 + tid; i < n_flags; i += (int)gridDim.x * 256) flags[i] = 0u;
    top = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(top)));
    if ((tid & 31) == 0) s_max[tid >> 5] = top;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; ++i) top = fmaxf(top, s_max[i]);
    int k = top > 0.f ? 13 + 127 - (int)(__float_as_uint(top) >> 23) : 0;
    k = k > 126 ? 126 : k;
    if (tid == 0) unscale[r] = tables_unscale(k);
    const float f = tables_exp2(k);
    const size_t part = (size_t)m_pad * E_pad;
    __half* const dst = w + (size_t)r * E_pad;
    auto put = [&](int e, float v) {
        const __half a = __float2half_rn(v * f);
        dst[e] = a;
        dst[part + e] = __float2half_rn((v * f - __half2float(a)) * kTmLow);
    };
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (tid + 256 * i < E_pad) put(tid + 256 * i, x[i]);
    for (int e = N * 256 + tid; e < E_pad; e += 256) put(e, r < m && e < E ? src[e] : 0.f);
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

// fp32 embeddings: rows that are worked out again by fp32 multiply-adds, which give what fp32 arithmetic gives: rows whose entries fp16
// parts do not hold well enough, and whatever has results that are not finite (infinities).  32 rows (-1: none) of 128 columns from
// c0, 256 threads, four rows and four columns each, blocks of 32 columns of E through shared memory, the next on its way meanwhile.  Sums
// of 256 terms are added up apart, so that the error is no larger than that of the other rows.
constexpr int kTmMendRows = 32;
struct __align__(16) TablesMend {
    float w[32][132], e[32][kTmMendRows + 4];
    int rows[kTmMendRows];
};
__device__ __noinline__ void tables_mend(const TablesParams& p, TablesMend* sm, int c0, int tid) {
    const int c = c0 + (tid & 31) * 4, r0 = (tid >> 5) * 4;
    // a warp fetches eight columns of E of four rows of W, four times side by side, then of the next four rows (rows past m: the last)
    const int wk = tid & 7, wc = (tid >> 5) * 16 + ((tid & 31) >> 3), ek = (tid & 7) * 4, er = tid >> 3;
    const int e_row = sm->rows[er];
    const float* const e_src = (const float*)p.emb + (size_t)(e_row < 0 ? 0 : e_row) * p.E;
    const float* w_src[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) w_src[i] = p.W + (size_t)(c0 + wc + 4 * i < p.m ? c0 + wc + 4 * i : p.m - 1) * p.E + wk;
    if (e_row >= 0)  // (the rows come from memory, a line a step: all of them on their way at once)
        for (int k = (tid & 7) * 32; k < p.E; k += 256) asm volatile("prefetch.global.L2 [%0];" ::"l"(e_src + k));
    float sum[4][4] = {}, part[4][4] = {}, w[16];
    float4 x;
    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] = k0 + wk + 8 * (i & 3) < p.E ? __ldg(w_src[i >> 2] + k0 + 8 * (i & 3)) : 0.f;
        x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (e_row >= 0 && k0 + ek < p.E) x = __ldg((const float4*)(e_src + k0 + ek));
    };
    const bool busy = sm->rows[r0] >= 0;  // (a warp's rows: none without the first)
    fetch(0);
    for (int k0 = 0, turn = 1; k0 < p.E; k0 += 32, ++turn) {
        named_bar_sync(3, 256);  // (what was there before has been read)
#pragma unroll
        for (int i = 0; i < 16; ++i) sm->w[wk + 8 * (i & 3)][wc + 4 * (i >> 2)] = w[i];
        sm->e[ek][er] = x.x, sm->e[ek + 1][er] = x.y, sm->e[ek + 2][er] = x.z, sm->e[ek + 3][er] = x.w;
        named_bar_sync(3, 256);
        if (k0 + 32 < p.E) fetch(k0 + 32);
        if (!busy) continue;
#pragma unroll 4
        for (int k = 0; k < 32; ++k) {
            const float4 wv = *(const float4*)&sm->w[k][(tid & 31) * 4], ev = *(const float4*)&sm->e[k][r0];
            const float ee[4] = {ev.x, ev.y, ev.z, ev.w}, ww[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) part[i][j] = fmaf(ee[i], ww[j], part[i][j]);
        }
        if (turn % 8 == 0 || k0 + 32 >= p.E) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) sum[i][j] += part[i][j], part[i][j] = 0.f;
        }
    }
    if (c < p.m) {
        float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
        if (p.bias) b = make_float4(p.bias[c], p.bias[c + 1], p.bias[c + 2], p.bias[c + 3]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (sm->rows[r0 + i] >= 0)
                *(float4*)(p.out + (size_t)sm->rows[r0 + i] * p.m + c) =
                    make_float4(sum[i][0] + b.x, sum[i][1] + b.y, sum[i][2] + b.z, sum[i][3] + b.w);
    }
    named_bar_sync(3, 256);
}

template <bool F32>
__global__ void __cluster_dims__(F32 ? 1 : 2, 1, 1) __launch_bounds__(TablesCfg<F32>::THREADS, 1)
    tables_mma_kernel(const __grid_constant__ TablesParams p) {
    using C = TablesCfg<F32>;
    constexpr uint32_t NS = C::STAGES, NR = C::RAW_STAGES;
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bars[2 * (NS + NR) + 5 + 2 * kTmScales];
    __shared__ uint8_t s_scale[F32 ? kTmScales : 1][128];  // the exponents (biased) of what the rows of the last tiles are multiplied by
    __shared__ float2 s_unscale[F32 ? 512 : 1];  // what columns are multiplied by (from memory at a tile's end: V = 30,000, E = 32 22.0 us, so 18.5)
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    __shared__ bool s_mend;
    __shared__ TablesShare s_share;
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
    const uint32_t accfull0 = rempty0 + 8 * NR, accempty0 = accfull0 + 16, sfull0 = accempty0 + 16, sempty0 = sfull0 + 8 * kTmScales;
    const uint32_t loempty = sempty0 + 8 * kTmScales;  // fp32: the small products' accumulator has been emptied
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
        for (uint32_t s = 0; s < kTmScales; ++s) {
            mbar_init(sfull0 + 8 * s, kTmConvWarps / 2);
            mbar_init(sempty0 + 8 * s, kTmEpiWarps + kTmConvWarps);
        }
        mbar_init(loempty, kTmEpiWarps);
        mbar_fence_init();
        s_abort = 0;
        s_mend = false;
    }
    if (tid == 32) tables_shares(p, pair, s_share);
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
        if (F32) {
            for (int c = tid; c < p.m_pad; c += kTmEpiWarps * 32) s_unscale[c] = __ldg(p.unscale + c);
            named_bar_sync(3, kTmEpiWarps * 32);
        }
        for (int i = 0; tables_item(p, s_share, pair, i, it); ++i) {
            const int rt = it.tile / p.n_mb, mb = it.tile - rt * p.n_mb;
            const uint32_t n = (uint32_t)tables_n<F32>(p, mb);
            int row_exp = 127;  // (fp32) the exponent of what this thread's row is multiplied by
            if (F32) {
                const uint32_t slot = (uint32_t)i % kTmScales;
                wait(sfull0 + 8 * slot, ((uint32_t)i / kTmScales) & 1u);
                row_exp = s_scale[slot][quarter * 32 + lane];
                __syncwarp();
                if (lane == 0) mbar_arrive(sempty0 + 8 * slot);
            }
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
                    const uint32_t t0 = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)half * 64u;
                    const uint32_t hi = F32 ? tables_hi(slot, n) : slot * 256u, lo = F32 ? kTmLo : slot * 256u + n;
                    const bool both = !F32 || kb + C::CHUNK >= it.kb1;  // (fp32: the small products' sums at the tile's end)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            if (j == 1 && !both) break;
                            uint32_t d[16];
                            tmem_ld_32x16(t0 + (j ? lo : hi) + 16u * q, d);
                            tmem_wait_ld();
#pragma unroll
                            for (int c = 0; c < 16; ++c) {
                                const float x = __uint_as_float(d[c]);
                                acc[h][16 * q + c] = F32 && j ? fmaf(x, 1.0f / kTmLow, acc[h][16 * q + c]) : acc[h][16 * q + c] + x;
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
                        if (F32 && both) mbar_arrive(loempty);
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
                float2 check = make_float2(0.f, 0.f);  // fp32 embeddings: NaN once a result is not finite
                if (v < rows) {
                    float* dst = base + (size_t)v * ld + half * 64;
                    const float2 row_unscale = tables_unscale(row_exp - 127);
#pragma unroll
                    for (int c = 0; c < 64; c += 8) {
                        if (c >= cols) break;
                        const bool both = c + 4 < cols;
                        if (F32) {
#pragma unroll
                            for (int k = 0; k < 8; ++k) {
                                const float2 f = s_unscale[mb * 128 + half * 64 + c + k];
                                acc[h][c + k] = acc[h][c + k] * (f.x * row_unscale.x) * (f.y * row_unscale.y);
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
                if (F32 && check.x + check.y != 0.f) {
                    p.bad_row[(size_t)it.tile * C::ROWS + v] = 1;
                    s_mend = true;
                }
            }
        }
        if (F32) {  // (nothing waits for these warps any more)
            __syncwarp();
            named_bar_sync(1, (kTmEpiWarps + kTmConvWarps) * 32);  // (the tiles are written, their rows looked at; the rings are done with)
            if (s_mend && !s_abort) {
                TablesMend* const sm = (TablesMend*)(smem_raw + (a_ring - smem_u32(smem_raw)));
                for (int i = 0; tables_item(p, s_share, pair, i, it); ++i) {
                    if (it.q0 != it.q1) continue;  // (pieces: the kernel that adds them up)
                    // the tile's flagged rows, 32 at a time; every warp looks at all flags
                    uint32_t again[C::ROWS / 32];
                    int n = 0;
#pragma unroll
                    for (int j = 0; j < C::ROWS / 32; ++j) {
                        again[j] = __ballot_sync(0xFFFFFFFFu, p.bad_row[(size_t)it.tile * C::ROWS + j * 32 + lane] != 0);
                        n += __popc(again[j]);
                    }
                    for (int first = 0; first < n; first += kTmMendRows) {
                        if (warp == 0) {
                            sm->rows[lane] = -1;
                            __syncwarp();
                            int before = -first;
#pragma unroll
                            for (int j = 0; j < C::ROWS / 32; ++j) {
                                const int at = before + __popc(again[j] & ((1u << lane) - 1u));
                                if ((again[j] >> lane & 1u) != 0u && at >= 0 && at < kTmMendRows)
                                    sm->rows[at] = it.tile / p.n_mb * C::ROWS + j * 32 + lane;
                                before += __popc(again[j]);
                            }
                        }
                        named_bar_sync(3, kTmEpiWarps * 32);
                        tables_mend(p, sm, it.tile % p.n_mb * 128, tid);
                    }
                }
            }
        }
    } else if (warp == 8) {
        // ------------------------------ TMA loads: W, bf16 embeddings ----------------------------
        if (lane == 0) {
            const uint32_t full_even = mapa_u32(full0, 0);
            TablesRing<NS> w(1);
            uint32_t cc = 0;  // chunks ahead of this tile
            for (int i = 0; tables_item(p, s_share, pair, i, it); cc += (uint32_t)(it.kb1 - it.kb0 + C::CHUNK - 1) / C::CHUNK, ++i) {
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
                        const int swap = (int)(cc + (uint32_t)(kb - it.kb0) / C::CHUNK) & 1;  // (tables_hi)
#pragma unroll
                        for (int j = 0; j < 2; ++j)
                            tma_load_2d(dw + (j ^ swap) * part, &p.map_w, x, j * p.m_pad + mb * 128, full0 + 8 * w.st);
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
        if constexpr (F32) {
            // The tensor cores stand still while this warp does anything but issue (few instructions are queued), so a block is a
            // wait, four instructions and a commit with next to nothing around them.  The whole warp goes through the loop, and one
            // lane issues: the operands are the same in all lanes that way, and stay in the registers that the instructions want.
            TablesRing<NS> w(0);
            const uint32_t tm = __shfl_sync(0xFFFFFFFFu, tmem, 0), lead = lane == 0 ? 1u : 0u;
            uint32_t cc = 0;
            for (int i = 0; tables_item(p, s_share, pair, i, it); ++i) {
                const uint32_t n = (uint32_t)p.box_n, idesc2 = umma_idesc(128, 2 * n, false), idesc1 = umma_idesc(128, n, false);
                constexpr uint64_t kHi = umma_desc_sw64(0u);
                const uint32_t wn = n * C::BLK * 2 / 16, lo = tm + kTmLo;
                if (i > 0) wait(loempty, (uint32_t)(i - 1) & 1u);
                for (int kb = it.kb0; kb < it.kb1; kb += C::CHUNK, ++cc) {
                    const uint32_t slot = cc & 1u, hi = tm + tables_hi(slot, n), both = slot ? lo : hi, o_w1 = slot ? wn : 0u;
                    if (cc >= 2) wait(accempty0 + 8 * slot, ((cc >> 1) - 1u) & 1u);
                    const int left = it.kb1 - kb < C::CHUNK ? it.kb1 - kb : C::CHUNK;
#pragma unroll 1
                    for (int k = 0; k < left; k += 2) {  // two blocks at a time: their waits and commits side by side
                        const bool two = k + 1 < left;
                        const TablesRing<NS> w0 = w;
                        w.next();
                        wait(full0 + 8 * w0.st, w0.ph);
                        if (two) wait(full0 + 8 * w.st, w.ph);
                        tc_fence_after();
                        uint32_t e1 = tm + kTmParts + 32u * w0.st;
                        uint64_t b = kHi | ((w_ring + w0.st * C::W_BYTES) >> 4);
                        if (k == 0) {  // the large products' accumulator starts again, the small ones' with the tile
                            umma_ts(hi, e1, b + o_w1, idesc1, false, lead);
                            umma_ts(lo, e1, b + (wn - o_w1), idesc1, kb > it.kb0, lead);
                        } else {
                            umma_ts(both, e1, b, idesc2, true, lead);
                        }
                        umma_ts(lo, e1 + 16u, b + o_w1, idesc1, true, lead);
                        umma_ts(both, e1 + 8u, b + 2, idesc2, true, lead);
                        umma_ts(lo, e1 + 24u, b + o_w1 + 2, idesc1, true, lead);
                        if (two) {
                            e1 = tm + kTmParts + 32u * w.st;
                            b = kHi | ((w_ring + w.st * C::W_BYTES) >> 4);
                            umma_ts(both, e1, b, idesc2, true, lead);
                            umma_ts(lo, e1 + 16u, b + o_w1, idesc1, true, lead);
                            umma_ts(both, e1 + 8u, b + 2, idesc2, true, lead);
                            umma_ts(lo, e1 + 24u, b + o_w1 + 2, idesc1, true, lead);
                        }
                        umma_commit_by(empty0 + 8 * w0.st, lead);
                        if (two) {
                            umma_commit_by(empty0 + 8 * w.st, lead);
                            w.next();
                        }
                    }
                    umma_commit_by(accfull0 + 8 * slot, lead);
                }
            }
        } else if (rank == 0) {
            TablesRing<NS> w(0);
            const uint32_t tm = __shfl_sync(0xFFFFFFFFu, tmem, 0), lead = lane == 0 ? 1u : 0u;
            uint32_t cc = 0;
            for (int i = 0; tables_item(p, s_share, pair, i, it); ++i) {
                const int n = tables_n<F32>(p, it.tile % p.n_mb);
                const uint32_t idesc2 = umma_idesc(256, 2 * n, true), idesc1 = umma_idesc(256, n, true);
                constexpr uint64_t kHi = umma_desc_sw128(0u);
                constexpr uint32_t o_w3 = 2 * (C::W_BYTES / 3) / 16;
                // Two blocks at a time.  An instruction whose accumulator columns the one just ahead of it wrote waits for those, so
                // the two row blocks' instructions alternate, except in the first and the last two blocks of a chunk, where the
                // first row block goes ahead: its accumulators are emptied (or were) while the second's are filled.
                for (int kb = it.kb0; kb < it.kb1; kb += 2) {
                    const bool two = kb + 2 <= it.kb1;
                    const bool first = (kb - it.kb0) % C::CHUNK == 0, last = kb + 2 >= it.kb1 || (kb + 2 - it.kb0) % C::CHUNK == 0;
                    const TablesRing<NS> w0 = w;
                    w.next();
                    wait(full0 + 8 * w0.st, w0.ph);
                    if (two) wait(full0 + 8 * w.st, w.ph);
                    tc_fence_after();
                    const uint64_t a0 = kHi | ((a_ring + w0.st * C::A_BYTES) >> 4), b0 = kHi | ((w_ring + w0.st * C::W_BYTES) >> 4);
                    const uint64_t a1 = kHi | ((a_ring + w.st * C::A_BYTES) >> 4), b1 = kHi | ((w_ring + w.st * C::W_BYTES) >> 4);
                    const auto large = [&](uint64_t a, uint64_t b, int h, int ks, bool more) {
                        umma_by(tm + h * 256u, a + h * (C::PART / 16) + 2 * ks, b + 2 * ks, idesc2, more, lead);
                    };
                    const auto small = [&](uint64_t a, uint64_t b, int h, int ks) {
                        umma_by(tm + h * 256u + (uint32_t)n, a + h * (C::PART / 16) + 2 * ks, b + o_w3 + 2 * ks, idesc1, true, lead);
                    };
                    if (!first && !last) {  // (two blocks)
#pragma unroll
                        for (int ks = 0; ks < 2 * (C::BLK / 16); ++ks) {
                            const int k = ks % (C::BLK / 16);
                            const uint64_t a = ks < C::BLK / 16 ? a0 : a1, b = ks < C::BLK / 16 ? b0 : b1;
                            large(a, b, 0, k, true);
                            large(a, b, 1, k, true);
                            small(a, b, 0, k);
                            small(a, b, 1, k);
                        }
                    } else {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (first && cc >= 1) {
                                wait(accempty0 + 8 * h, (cc - 1u) & 1u);
                                tc_fence_after();
                            }
#pragma unroll
                            for (int ks = 0; ks < C::BLK / 16; ++ks) {
                                large(a0, b0, h, ks, !first || ks > 0);
                                small(a0, b0, h, ks);
                            }
                            if (two) {
#pragma unroll
                                for (int ks = 0; ks < C::BLK / 16; ++ks) {
                                    large(a1, b1, h, ks, true);
                                    small(a1, b1, h, ks);
                                }
                            }
                            if (last) umma_commit_pair_by(accfull0 + 8 * h, lead);
                        }
                    }
                    umma_commit_pair_by(empty0 + 8 * w0.st, lead);
                    if (two) {
                        umma_commit_pair_by(empty0 + 8 * w.st, lead);
                        w.next();
                    }
                    if (last) ++cc;
                }
            }
        }
    } else if (F32 && warp == 10) {
        // ------------------------------ TMA loads: fp32 embeddings -------------------------------
        if (lane == 0) {
            TablesRing<NR> r(1);
            for (int i = 0; tables_item(p, s_share, pair, i, it); ++i) {
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
        // barriers that it waits on: with an even number of stages every stage is always the same half's.
        static_assert(!F32 || (NR % 2 == 0 && NS % 2 == 0), "a stage of either ring belongs to one half of the converting warps");
        // A thread has a row: a warp reaches its quarter of TMEM's lanes (its index modulo four), and a half has all four.
        const int half = (warp - (kTmEpiWarps + 3)) >> 2, row = 32 * (warp & 3) + lane;
        const uint32_t parts = tmem + kTmParts + ((uint32_t)(32 * (warp & 3)) << 16);
        TablesRing<NS> a(1);
        TablesRing<NR> r(0);
        float4 x[8];
        auto load = [&]() {
            wait(rfull0 + 8 * r.st, r.ph);
            const uint32_t src = raw_ring + r.st * C::RAW + (uint32_t)row * 128u;
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = ld_shared_f4(src + (uint32_t)((j ^ (row & 7)) * 16));  // (128-byte rows in the 128-byte swizzle)
            __syncwarp();
            if (lane == 0) mbar_arrive(rempty0 + 8 * r.st);
        };
        auto largest = [&](int j) {  // of columns 8 j .. 8 j + 7
            const float m0 = fmaxf(fmaxf(fabsf(x[2 * j].x), fabsf(x[2 * j].y)), fmaxf(fabsf(x[2 * j].z), fabsf(x[2 * j].w)));
            const float m1 = fmaxf(fmaxf(fabsf(x[2 * j + 1].x), fabsf(x[2 * j + 1].y)), fmaxf(fabsf(x[2 * j + 1].z), fabsf(x[2 * j + 1].w)));
            return fmaxf(m0, m1);
        };
        for (int i = 0; tables_item(p, s_share, pair, i, it); ++i) {
            // the rows' scales, from the half that has the tile's first block, for both halves and for the warps that empty the
            // accumulators (everybody waits for every phase of these barriers, the half that sets the scales too)
            const uint32_t slot = (uint32_t)i % kTmScales, turn = (uint32_t)i / kTmScales;
            const bool lead = (int)(a.t & 1u) == half;
            if (turn > 0) wait(sempty0 + 8 * slot, (turn - 1u) & 1u);
            if (lead) {
                load();
                s_scale[slot][row] = (uint8_t)(__float_as_uint(tables_row_scale(fmaxf(fmaxf(largest(0), largest(1)), fmaxf(largest(2), largest(3))))) >> 23);
                __syncwarp();
                if (lane == 0) mbar_arrive(sfull0 + 8 * slot);
            }
            wait(sfull0 + 8 * slot, turn & 1u);
            const float scale = __uint_as_float((uint32_t)s_scale[slot][row] << 23);
            float most = 0.f, least = INFINITY;  // largest and smallest, but for zero, of eight entries' largest magnitudes
            __syncwarp();
            if (lane == 0) mbar_arrive(sempty0 + 8 * slot);
            for (int kb = it.kb0; kb < it.kb1; ++kb, a.next(), r.next()) {
                if ((int)(a.t & 1u) != half) continue;
                if (kb != it.kb0) load();
                uint32_t b[32];  // columns of TMEM: the 32 numbers' first parts, then their second
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    split2(x[j].x, x[j].y, scale, b[2 * j], b[16 + 2 * j]);
                    split2(x[j].z, x[j].w, scale, b[2 * j + 1], b[16 + 2 * j + 1]);
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float m = largest(j);
                    most = fmaxf(most, m);
                    if (m != 0.f) least = fminf(least, m);
                }
                if (a.t >= NS) {
                    wait(empty0 + 8 * a.st, a.ph);
                    tc_fence_after();
                }
                tmem_st_32x32(parts + 32u * a.st, b);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(full0 + 8 * a.st);
            }
            // rows that the parts do not hold well enough
            const int rt = it.tile / p.n_mb;
            if ((most * scale > kTmMost || least * scale < kTmLeast) && rt * C::ROWS + row < p.V) {
                p.bad_row[(size_t)it.tile * C::ROWS + row] = 1;
                if (it.q0 == it.q1) s_mend = true;
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

// The left-over tiles' pieces, added up in order: four columns of N rows a thread, a warp a row, 8 N rows a block.
template <bool F32, int N, int PER_SM>
__global__ void __launch_bounds__(256, PER_SM) tables_pieces_kernel(const __grid_constant__ TablesParams p) {
    using C = TablesCfg<F32>;
    static_assert(8 * N <= kTmMendRows, "rows that may have to be worked out again");
    __shared__ TablesMend sm;
    pdl_wait();
    const int tile = (int)blockIdx.y, rt = tile / p.n_mb, mb = tile - rt * p.n_mb;
    const int q0 = tables_owner(p, tile * p.n_kb), q1 = tables_owner(p, (tile + 1) * p.n_kb - 1);
    const int v0 = (int)blockIdx.x * 8 * N, warp = threadIdx.x >> 5, c = (threadIdx.x & 31) * 4, col = mb * 128 + c;
    if (q0 == q1 || rt * C::ROWS + v0 >= p.V) return;  // (q0 == q1: written whole; uniform)
    float4 s[N];
#pragma unroll
    for (int i = 0; i < N; ++i) s[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int seg0 = tables_share(p, q0) < tile * p.n_kb ? 1 : 0;  // (the others' shares begin in this tile)
#pragma unroll(PER_SM == 4 ? 8 : 4)
    for (int q = q0; q <= q1; ++q) {
        const int seg = q == q0 ? seg0 : 0;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const float4 x = __ldcs((const float4*)(p.pieces + ((size_t)(q * 2 + seg) * C::ROWS + v0 + 8 * i + warp) * 128 + c));
            s[i].x += x.x, s[i].y += x.y, s[i].z += x.z, s[i].w += x.w;
        }
    }
    float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
    if (p.bias && col < p.m) b = make_float4(p.bias[col], p.bias[col + 1], p.bias[col + 2], p.bias[col + 3]);
    bool any = false;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const int v = v0 + 8 * i + warp, row = rt * C::ROWS + v;
        bool off = false;
        if (row < p.V && col < p.m) {
            s[i].x += b.x, s[i].y += b.y, s[i].z += b.z, s[i].w += b.w;
            *(float4*)(p.out + (size_t)row * p.m + col) = s[i];
            off = F32 && (p.bad_row[(size_t)tile * C::ROWS + v] != 0 || fmaf(0.f, s[i].x, fmaf(0.f, s[i].y, fmaf(0.f, s[i].z, 0.f * s[i].w))) != 0.f);
        }
        if (F32) {
            off = __any_sync(0xFFFFFFFFu, off);
            if (c == 0) sm.rows[8 * i + warp] = off ? row : -1;
            any |= off;
        }
    }
    if (F32 && __syncthreads_or(any)) {
        if (warp == 0) {  // those that are wanted first
            const int r = (c >> 2) < 8 * N ? sm.rows[c >> 2] : -1;
            __syncwarp();
            const uint32_t wanted = __ballot_sync(0xFFFFFFFFu, r >= 0), below = (1u << (c >> 2)) - 1u;
            sm.rows[r >= 0 ? __popc(wanted & below) : __popc(wanted) + __popc(~wanted & below)] = r;
        }
        __syncthreads();
        tables_mend(p, &sm, mb * 128, (int)threadIdx.x);
    }
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
    size_t o_w, o_unscale, o_bad, n_bad, total;  // (fp32 only: from o_unscale on)
};
TablesSizes tables_sizes(int num_sms, int V, int E, int m, bool f32) {
    TablesSizes s;
    s.n_mb = (m + 127) / 128;
    s.m_pad = 128 * s.n_mb;
    s.E_pad = (E + 63) / 64 * 64;
    s.pairs = f32 ? num_sms : num_sms / 2;
    s.o_w = (size_t)s.pairs * 2 * (f32 ? TablesCfg<true>::ROWS : TablesCfg<false>::ROWS) * 128 * sizeof(float);
    s.o_unscale = s.o_w + (size_t)(f32 ? 2 : 3) * s.m_pad * s.E_pad * 2;
    s.o_bad = s.o_unscale + (f32 ? (size_t)s.m_pad * sizeof(float2) : 0);
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
        // fp32: 32 rows a block where that leaves a block an SM or more, else 8 (E = 2048, 32 rows and 8: 102 tiles left, V = 32,000,
        // 73.3 and 77.1 us; 71, V = 28,000, 64.7 and 66.9; 33, V = 42,000, 89.3 and 87.7; 9, V = 20,000, 59.0 and 52.3)
        constexpr int N = F32 ? 4 : 1;
        if (F32 ? p.left * (C::ROWS / (8 * N)) >= p.pairs : p.share_pairs < 6 * p.left)
            e = launch_pdl(tables_pieces_kernel<F32, N, F32 ? 3 : 8>, dim3(C::ROWS / (8 * N), p.left), dim3(256), 0, st, p);
        else  // (few tiles left, many pieces each: bf16 with registers for eight pieces' loads, V = 151,936, one tile: 14 -> 8 us; 9, V =
              // 80,000, E = 4096 183.5 -> 181.9; 24, three pieces each, V = 50,000, E = 2048 stays: 70.7 against 72.3)
            e = launch_pdl(tables_pieces_kernel<F32, 1, F32 ? 3 : 4>, dim3(C::ROWS / 8, p.left), dim3(256), 0, st, p);
        *launches += 1;
    }
    return e;
}

}  // namespace

// Can the tensor cores take this table?  16-byte rows for the loads and stores; anything else goes to the FMA kernel.
bool tables_mma_fits(int num_sms, int V, const void* d_emb, graft_dtype dt, int E, int m, const void* d_out) {
    if (E % (dt == GRAFT_BF16 ? 8 : 4) != 0 || (((uintptr_t)d_emb | (uintptr_t)d_out) & 15) != 0 || encode_tiled() == nullptr) return false;
    // Shares of the tiles that are left are worked out in 32 bits (tables_share, tables_owner), which holds for all that fits in
    // memory: 148 workers share 28 million blocks and more, of 16 KB each, and a few narrow tiles are shared by fewer.
    const int rows = dt == GRAFT_F32 ? TablesCfg<true>::ROWS : TablesCfg<false>::ROWS, blk = dt == GRAFT_F32 ? TablesCfg<true>::BLK : TablesCfg<false>::BLK;
    const TablesSizes s = tables_sizes(num_sms, V, E, m, dt == GRAFT_F32);
    const uint64_t left = (uint64_t)((V + (long long)rows - 1) / rows * s.n_mb % s.pairs);
    const uint64_t share = left * kTmMaxSplit < (uint64_t)s.pairs ? left * kTmMaxSplit : (uint64_t)s.pairs;
    return (share + 1) * left * ((uint64_t)(E + (long long)blk - 1) / blk) <= 0xFFFFFFFFull;
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
        // 4096, with and without a round of whole tiles ahead.  Now, equal and whole, us: V = 16,000, bf16: E = 1024 29.7 and 24.9,
        // E = 4096 54.2 and 52.2; V = 32,000, E = 1024: bf16 43.1 and 30.1, fp32 48.1 and 45.0; fp32, E = 2048 73.3 and 74.9, V = 50,000
        // 105.1 and 109.1, which keep equal shares.  Of 54 sizes two are on the slower side: fp32, E = 1536, V = 32,000 61.1 and 59.7,
        // 64,000 104.0 and 100.4.)
        const long long q = sp / p.left;
        const double longer = (1.0 / (double)q - (double)p.left / (double)sp) * E;
        if (longer <= (f32 ? (q == 1 ? 380 : 130) : (q == 1 ? 850 : 350))) sp = q * p.left;
    }
    p.share_pairs = (int)(sp < p.left ? p.left : sp);
    p.wide = m % 8 == 0 && ((uintptr_t)d_out & 31) == 0;
    SplitParams split;
    split.W = d_W;
    split.m = m;
    split.E = E;
    split.m_pad = s.m_pad;
    split.E_pad = s.E_pad;
    split.w = w;
    split.unscale = (float2*)((char*)scratch + s.o_unscale);
    split.flags = (uint32_t*)p.bad_row;
    split.n_flags = (int)(s.n_bad / 4);
    cudaError_t e = f32 ? launch_pdl(weight_split16_kernel, dim3(s.m_pad), dim3(256), 0, st, split)
                        : launch_pdl(weight_split_kernel, dim3((s.E_pad + 511) / 512, s.m_pad), dim3(256), 0, st, split);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    int launches = 1;
    e = f32 ? tables_run<true>(p, st, &launches) : tables_run<false>(p, st, &launches);
    ctx->launches += (uint64_t)launches;
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace graft

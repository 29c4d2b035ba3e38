// Table precompute on the tensor cores: out[v] = W e_v + b (text after Eq. 6: the projections depend only on the token
// id and are computed once).  This is the one dense contraction of the method, [V, E] x [E, m].
//
// Operands are bf16 parts of the inputs: an fp32 number is the sum of three bf16 ones (8 + 8 + 8 mantissa bits), and a
// product of two bf16 numbers is exact in the fp32 accumulator.
//   bf16 embeddings: out = e W1 + e W2 + e W3               (three products a step, all exact)
//   fp32 embeddings: out = (e1 + e2 + e3) W1 + ((e1 + e2 + e3) W2 + e1 W3)   (what is dropped is below 2^-26 of a term)
// so the result differs from an fp32 GEMM by the order and the rounding of the additions.  The accumulators of the tensor
// cores round less carefully than an FMA chain: they are emptied into fp32 registers after 32 (bf16) or 24 (fp32
// embeddings) additions to the large products' accumulators, which W2's and W3's do not share.
//
// One persistent kernel.  A worker -- a pair of CTAs (cluster of two, tcgen05 cta_group::2) for bf16 embeddings, one CTA
// for fp32 -- owns a tile of 512 (fp32: 128) rows of V times up to 128 columns of m, and streams E in blocks of 64 (32)
// columns through shared-memory rings.
//   warps 0-7    empty the accumulators (TMEM, two sets of 2 x 128 columns), keep the running sums and write the tile
//   warp 8       TMA loads: W's parts (split once per call into scratch by weight_split_kernel), bf16 embeddings
//   warp 9       issues the matrix instructions
//   warp 10      fp32 only: TMA loads of the raw rows;  warps 11-18  raw rows -> bf16 parts in the operands' layout
// W1 and W2 stand side by side as one operand of N = 256, W3 is an N = 128 of its own (three of N = 128 in a row on one
// accumulator took 122 cycles each: an instruction waits for the one ahead of it on the same columns).  Tiles of 512
// rows halve the passes over W, which comes from L2 every time.  The fp32 kernel works on single CTAs because its rows
// go through threads: telling the other CTA of a pair about every block cost more (136 - 160 us at V = 32,000, E = 2048)
// than the second CTA's half of W saves (120 us).  The embeddings are read from memory once; nothing but the tables is
// written.  What is left when the tiles do not divide by the workers is dealt out along E in shares, whose sums a
// small kernel adds up in order (summing them inside, by the warp that came last, stalled its tile: 462 against 370 us).
//
// Measured (one tower, back to back, B200): V = 151,936, E = 4096, m = 128, bf16: 373 us (798 us with the library
// template's GEMMs, whose partial sums went through memory); its products take 287 us at the measured dense rate, the
// loads alone 258 us.  V = 32,000, E = 2048, fp32: 120 us (1180 us by the FMA kernel; the loads and the splitting 82 us).
// Largest error against fp64 products at those sizes: 3.2e-6 and 3.0e-6 (library template 6.3e-6, FMA kernel 1.2e-5).
#include <cuda.h>
#include <cuda_bf16.h>
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
    static constexpr int CHUNK = F32 ? 4 : 8;  // blocks between two emptyings of an accumulator
    static constexpr int PART = 128 * BLK * 2;                // bytes of 128 rows of bf16
    static constexpr int A_BYTES = (F32 ? 3 : MT) * PART;     // a block's embeddings
    static constexpr int W_BYTES = (F32 ? 384 : 192) * BLK * 2;  // a block's W; a pair: W1 (even CTA) or W2 (odd), half of W3
    static constexpr int RAW = 128 * BLK * 4;                 // a block's fp32 embeddings
    static constexpr int A_STAGES = F32 ? 3 : 4, W_STAGES = F32 ? 3 : 4, RAW_STAGES = F32 ? 4 : 1;
    static constexpr int THREADS = (kTmEpiWarps + 2 + (F32 ? 1 + kTmConvWarps : 0)) * 32;
    // (the rings start on a 1024-byte boundary)
    static constexpr size_t SMEM = (size_t)A_STAGES * A_BYTES + (size_t)W_STAGES * W_BYTES + (F32 ? (size_t)RAW_STAGES * RAW : 0) + 1024;
    static __device__ __forceinline__ uint64_t desc(uint32_t addr) { return F32 ? umma_desc_sw64(addr) : umma_desc_sw128(addr); }
};

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
    CUtensorMap map_w;  // [3 * m_pad, E_pad] bf16
    CUtensorMap map_e;  // [V, E] embeddings
    const void* emb;    // [V, E]
    const float* W;     // [m, E]
    const float* bias;  // [m] or NULL
    float* out;         // [V, m]
    float* pieces;      // [pairs][2 pieces][ROWS][128]
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

// two fp32 numbers -> their three bf16 parts, packed
__device__ __forceinline__ void split3(float x0, float x1, uint32_t& a, uint32_t& b, uint32_t& c) {
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(a) : "f"(x1), "f"(x0));
    x0 -= __uint_as_float(a << 16);
    x1 -= __uint_as_float(a & 0xFFFF0000u);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(b) : "f"(x1), "f"(x0));
    x0 -= __uint_as_float(b << 16);
    x1 -= __uint_as_float(b & 0xFFFF0000u);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(c) : "f"(x1), "f"(x0));
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

// fp32 embeddings: an entry whose bf16 parts are not all finite -- an infinity, a value that rounds past the largest bf16 --
// turns every result it has a part in into a NaN or an infinity.  Results that are not finite are worked out again as one
// chain of fp32 multiply-adds, which gives what fp32 arithmetic gives; such entries are rare, so the time does not matter.
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
    constexpr uint32_t NA = C::A_STAGES, NW = C::W_STAGES, NR = C::RAW_STAGES;
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bars[2 * (NA + NW + NR) + 4];
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
    const uint32_t w_ring = a_ring + NA * C::A_BYTES, raw_ring = w_ring + NW * C::W_BYTES;
    // afull / wfull: a block's rows, its W are there (a pair: in both CTAs; the even CTA's barriers), aempty / wempty: the
    // instructions that read them are done, rfull / rempty: fp32 rows as loaded
    const uint32_t afull0 = smem_u32(bars), aempty0 = afull0 + 8 * NA, wfull0 = aempty0 + 8 * NA, wempty0 = wfull0 + 8 * NW;
    const uint32_t rfull0 = wempty0 + 8 * NW, rempty0 = rfull0 + 8 * NR;
    const uint32_t accfull0 = rempty0 + 8 * NR, accempty0 = accfull0 + 16;
    if (tid == 0) {
        for (uint32_t s = 0; s < NA; ++s) {
            mbar_init(afull0 + 8 * s, F32 ? kTmConvWarps : 1);
            mbar_init(aempty0 + 8 * s, 1);
        }
        for (uint32_t s = 0; s < NW; ++s) {
            mbar_init(wfull0 + 8 * s, 1);
            mbar_init(wempty0 + 8 * s, 1);
        }
        for (uint32_t s = 0; s < NR; ++s) {
            mbar_init(rfull0 + 8 * s, 1);
            mbar_init(rempty0 + 8 * s, kTmConvWarps);
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
                            for (int c = 0; c < 16; ++c) acc[h][16 * q + c] += __uint_as_float(d[c]);
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
            named_bar_sync(1, kTmEpiWarps * 32);  // (the tiles are written for every thread of these warps)
            if (s_mend && !s_abort) {
                for (int i = 0; tables_item(p, pair, i, it); ++i) {
                    if (it.q0 != it.q1) continue;  // (pieces: the kernel that adds them up)
                    const int rt = it.tile / p.n_mb, c0 = (it.tile - rt * p.n_mb) * 128;
                    for (int v = rt * C::ROWS + warp; v < p.V && v < (rt + 1) * C::ROWS; v += kTmEpiWarps)
                        for (int c = c0 + lane; c < p.m && c < c0 + 128; c += 32) {
                            float* o = p.out + (size_t)v * p.m + c;
                            if (!tables_finite(*o)) *o = tables_fp32(p, v, c);
                        }
                }
            }
        }
    } else if (warp == 8) {
        // ------------------------------ TMA loads: W, bf16 embeddings ----------------------------
        if (lane == 0) {
            const uint32_t afull_even = mapa_u32(afull0, 0), wfull_even = mapa_u32(wfull0, 0);
            TablesRing<NA> a(1);
            TablesRing<NW> w(1);
            for (int i = 0; tables_item(p, pair, i, it); ++i) {
                const int rt = it.tile / p.n_mb, mb = it.tile - rt * p.n_mb;
                const int n = tables_n<F32>(p, mb);
                const int w12 = (int)rank * p.m_pad + mb * 128, w3 = 2 * p.m_pad + mb * 128 + (int)rank * (n >> 1);
                for (int kb = it.kb0; kb < it.kb1; ++kb) {
                    const int x = kb * C::BLK;
                    if (!F32) {
                        if (a.t >= NA) wait(aempty0 + 8 * a.st, a.ph);
                        if (s_abort) break;  // (no copy is started any more)
                        if (rank == 0) mbar_arrive_expect_tx(afull0 + 8 * a.st, 2u * C::A_BYTES);
#pragma unroll
                        for (int h = 0; h < C::MT; ++h)
                            tma_load_2d_pair(a_ring + a.st * C::A_BYTES + h * C::PART, &p.map_e, x,
                                             rt * C::ROWS + h * 256 + (int)rank * 128, afull_even + 8 * a.st);
                        a.next();
                    }
                    if (w.t >= NW) wait(wempty0 + 8 * w.st, w.ph);
                    if (s_abort) break;
                    const uint32_t dw = w_ring + w.st * C::W_BYTES, fb = wfull_even + 8 * w.st;
                    if (C::PAIR) {
                        if (rank == 0) mbar_arrive_expect_tx(wfull0 + 8 * w.st, 2u * C::W_BYTES);
                        tma_load_2d_pair(dw, &p.map_w, x, w12, fb);
                        tma_load_2d_pair(dw + C::W_BYTES / 3, &p.map_w, x, w12 + 64, fb);
                        tma_load_2d_pair(dw + 2 * (C::W_BYTES / 3), &p.map_w, x, w3, fb);
                    } else {
                        const uint32_t part = (uint32_t)n * C::BLK * 2;
                        mbar_arrive_expect_tx(wfull0 + 8 * w.st, 3u * part);
#pragma unroll
                        for (int j = 0; j < 3; ++j)
                            tma_load_2d(dw + j * part, &p.map_w, x, j * p.m_pad + mb * 128, wfull0 + 8 * w.st);
                    }
                    w.next();
                }
            }
            // the last arrivals from the other CTA have come before this CTA retires; after an abort: no copy of the pair
            // is in flight any more
            if (!F32) a.drain(aempty0, rank == 0 ? afull0 : 0u, &s_abort);
            w.drain(wempty0, rank == 0 ? wfull0 : 0u, &s_abort);
        }
    } else if (warp == 9) {
        // ------------------------------ matrix instructions --------------------------------------
        if (rank == 0 && lane == 0) {
            TablesRing<NA> a(0);
            TablesRing<NW> w(0);
            uint32_t cc = 0;
            for (int i = 0; tables_item(p, pair, i, it); ++i) {
                const int mb = it.tile % p.n_mb;
                const int n = tables_n<F32>(p, mb);
                constexpr int M = C::PAIR ? 256 : 128;
                const uint32_t idesc2 = umma_idesc_bf16(M, 2 * n), idesc1 = umma_idesc_bf16(M, n);
                const uint32_t o_w3 = C::PAIR ? 2 * (C::W_BYTES / 3) : (uint32_t)n * (2 * C::BLK * 2);
                for (int kb = it.kb0; kb < it.kb1; ++kb) {
                    const bool first = (kb - it.kb0) % C::CHUNK == 0;
                    const bool last = kb + 1 == it.kb1 || (kb + 1 - it.kb0) % C::CHUNK == 0;
                    wait(wfull0 + 8 * w.st, w.ph);
                    wait(afull0 + 8 * a.st, a.ph);
                    tc_fence_after();
                    const uint32_t a0 = a_ring + a.st * C::A_BYTES, b0 = w_ring + w.st * C::W_BYTES;
                    // An instruction whose accumulator columns the one just ahead of it wrote waits for those; with two row
                    // blocks their instructions alternate, except in the first and the last block of a chunk, where the
                    // first row block goes ahead (its accumulators are emptied, or were, while the second's are filled).
                    auto mma = [&](int h, int ks, bool w3) {
                        const uint32_t d = tmem + (C::MT == 1 ? (cc & 1u) : (uint32_t)h) * 256u;
                        const uint64_t a1 = C::desc(a0 + h * C::PART + 32 * ks);
                        if (w3) {
                            umma<C::PAIR>(d + (uint32_t)n, a1, C::desc(b0 + o_w3 + 32 * ks), idesc1, true);
                        } else {
                            const uint64_t w12 = C::desc(b0 + 32 * ks);
                            umma<C::PAIR>(d, a1, w12, idesc2, !first || ks > 0);
                            if (F32) {
                                umma<C::PAIR>(d, C::desc(a0 + C::PART + 32 * ks), w12, idesc2, true);
                                umma<C::PAIR>(d, C::desc(a0 + 2 * C::PART + 32 * ks), w12, idesc2, true);
                            }
                        }
                    };
                    if (C::MT == 2 && !first && !last) {
                        if (!s_abort) {
#pragma unroll
                            for (int ks = 0; ks < C::BLK / 16; ++ks) {
                                mma(0, ks, false);
                                mma(1, ks, false);
                                mma(0, ks, true);
                                mma(1, ks, true);
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
                                for (int ks = 0; ks < C::BLK / 16; ++ks) {
                                    mma(h, ks, false);
                                    mma(h, ks, true);
                                }
                            }
                            if (last) umma_commit<C::PAIR>(accfull0 + 8 * slot);
                        }
                    }
                    umma_commit<C::PAIR>(aempty0 + 8 * a.st);
                    umma_commit<C::PAIR>(wempty0 + 8 * w.st);
                    if (last) ++cc;
                    a.next();
                    w.next();
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
        // ------------------------------ fp32 embeddings -> bf16 parts ----------------------------
        const int ct = tid - (kTmEpiWarps + 3) * 32;
        const int c8 = ct & 3, r0 = ct >> 2;  // columns 8 c8 .. 8 c8 + 7 of rows r0 and r0 + 64
        TablesRing<NA> a(1);
        TablesRing<NR> r(0);
        for (int i = 0; tables_item(p, pair, i, it); ++i) {
            for (int kb = it.kb0; kb < it.kb1; ++kb) {
                wait(rfull0 + 8 * r.st, r.ph);
                const uint32_t src = raw_ring + r.st * C::RAW;
                float4 x[2][2];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int row = r0 + 64 * q;
#pragma unroll
                    for (int h = 0; h < 2; ++h)  // (128-byte rows in the 128-byte swizzle)
                        x[q][h] = ld_shared_f4(src + (uint32_t)row * 128u + (uint32_t)(((2 * c8 + h) ^ (row & 7)) * 16));
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(rempty0 + 8 * r.st);
                r.next();
                if (a.t >= NA) wait(aempty0 + 8 * a.st, a.ph);
                const uint32_t dst = a_ring + a.st * C::A_BYTES;
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int row = r0 + 64 * q;  // (64-byte rows in the 64-byte swizzle)
                    const uint32_t at = dst + (uint32_t)row * 64u + (uint32_t)((c8 ^ ((row >> 1) & 3)) * 16);
                    uint32_t b1[4], b2[4], b3[4];
                    split3(x[q][0].x, x[q][0].y, b1[0], b2[0], b3[0]);
                    split3(x[q][0].z, x[q][0].w, b1[1], b2[1], b3[1]);
                    split3(x[q][1].x, x[q][1].y, b1[2], b2[2], b3[2]);
                    split3(x[q][1].z, x[q][1].w, b1[3], b2[3], b3[3]);
                    st_shared_v4(at, b1);
                    st_shared_v4(at + C::PART, b2);
                    st_shared_v4(at + 2 * C::PART, b3);
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(afull0 + 8 * a.st);
                a.next();
            }
        }
        a.drain(aempty0, 0u, &s_abort);
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
    if (F32 && fmaf(0.f, s.x, fmaf(0.f, s.y, fmaf(0.f, s.z, 0.f * s.w))) != 0.f) {
        if (!tables_finite(s.x)) s.x = tables_fp32(p, row, col);
        if (!tables_finite(s.y)) s.y = tables_fp32(p, row, col + 1);
        if (!tables_finite(s.z)) s.z = tables_fp32(p, row, col + 2);
        if (!tables_finite(s.w)) s.w = tables_fp32(p, row, col + 3);
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
bool encode_map(CUtensorMap* map, const void* base, bool f32, uint64_t rows, uint64_t cols, uint32_t box_rows, uint32_t box_bytes) {
    const uint32_t esz = f32 ? 4 : 2;
    const cuuint64_t dims[2] = {cols, rows}, strides[1] = {cols * esz};
    const cuuint32_t box[2] = {box_bytes / esz, box_rows}, step[2] = {1, 1};
    return encode_tiled()(map, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                          const_cast<void*>(base), dims, strides, box, step, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          box_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct TablesSizes {
    int n_mb, m_pad, E_pad, pairs;
    size_t o_w, total;
};
TablesSizes tables_sizes(int num_sms, int E, int m, bool f32) {
    TablesSizes s;
    s.n_mb = (m + 127) / 128;
    s.m_pad = 128 * s.n_mb;
    s.E_pad = (E + 63) / 64 * 64;
    s.pairs = f32 ? num_sms : num_sms / 2;
    s.o_w = (size_t)s.pairs * 2 * (f32 ? TablesCfg<true>::ROWS : TablesCfg<false>::ROWS) * 128 * sizeof(float);
    s.total = s.o_w + (size_t)3 * s.m_pad * s.E_pad * 2;
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
size_t tables_mma_scratch_bytes(int num_sms, int E, int m, graft_dtype dt) {
    return tables_sizes(num_sms, E, m, dt == GRAFT_F32).total;
}

// out [V, m] = emb [V, E] . W^T + bias.  scratch: tables_mma_scratch_bytes, 256-byte aligned.
cudaError_t tables_mma_launch(graft_ctx* ctx, const void* d_emb, graft_dtype dt, int E, const float* d_W, const float* d_b,
                              float* d_out, void* scratch, cudaStream_t st) {
    const int V = ctx->cfg.V, m = ctx->cfg.m;
    const bool f32 = dt == GRAFT_F32;
    const TablesSizes s = tables_sizes(ctx->num_sms, E, m, f32);
    __nv_bfloat16* w = (__nv_bfloat16*)((char*)scratch + s.o_w);
    TablesParams p;
    const int blk = f32 ? TablesCfg<true>::BLK : TablesCfg<false>::BLK;
    p.box_n = s.n_mb > 1 ? 128 : (m + 31) / 32 * 32;
    if (!encode_map(&p.map_w, w, false, (uint64_t)3 * s.m_pad, s.E_pad, f32 ? p.box_n : 64, 2 * blk) ||
        !encode_map(&p.map_e, d_emb, f32, V, E, 128, 128))
        return cudaErrorUnknown;
    p.emb = d_emb;
    p.W = d_W;
    p.bias = d_b;
    p.out = d_out;
    p.pieces = (float*)scratch;
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
    weight_split_kernel<<<dim3((s.E_pad + 511) / 512, s.m_pad), 256, 0, st>>>(d_W, m, E, s.m_pad, s.E_pad, w);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    int launches = 1;
    e = f32 ? tables_run<true>(p, st, &launches) : tables_run<false>(p, st, &launches);
    ctx->launches += (uint64_t)launches;
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace graft

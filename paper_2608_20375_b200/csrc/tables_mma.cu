// Table precompute on the tensor cores: out[v] = W e_v + b (text after Eq. 6: the projections depend only on the token
// id and are computed once).  This is the one dense contraction of the method, [V, E] x [E, m].
//
// Operands are bf16 parts of the inputs: an fp32 number is the sum of three bf16 ones (8 + 8 + 8 mantissa bits), and a
// product of two bf16 numbers is exact in the fp32 accumulator.
//   bf16 embeddings: out = e W1 + e W2 + e W3               (three products a step, all exact)
//   fp32 embeddings: out = e1 W1 + (e1 W2 + e1 W3 + e2 W1 + e2 W2 + e3 W1)   (what is dropped is below 2^-23 of a term)
// so the result differs from an fp32 GEMM only by the order of the additions.  The accumulators of the tensor cores
// round less carefully than an FMA chain: they are emptied into fp32 registers after 32 (bf16) or 24 (fp32
// embeddings) additions to the large products' accumulators, which W2's and W3's do not share.
//
// One kernel, persistent, a cluster of two CTAs per pair of SMs (tcgen05, cta_group::2): a pair owns a tile of 512 rows
// of V (fp32 embeddings: 256) times up to 128 columns of m, and streams E in blocks of 64 through a shared-memory ring.
//   warps 0-7   empty the accumulators (TMEM, two sets of 2 x 128 columns), keep the running sums and write the tile
//   warp 8      TMA loads: W's parts (split once per call into scratch by weight_split_kernel) and the embeddings
//   warp 9      issues the matrix instructions (even CTA only)
//   warps 10-17 fp32 embeddings only: raw rows -> bf16 parts in the operands' layout
// W1 and W2 stand side by side as one operand of N = 256 (M = 256, N = 128 takes as long as N = 256: 128 cycles measured),
// W3 is an N = 128 of its own.  Tiles of 512 rows halve the passes over W, which comes from L2 every time.  The
// embeddings are read from memory once; nothing but the tables is written.  What is left when the tiles do not divide
// by the pairs is dealt out along E in equal shares, and the pair that finishes a tile's last piece adds them up in order.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "internal.h"
#include "umma.cuh"

namespace graft {
namespace {

constexpr int kTmBlk = 64;            // columns of E per ring stage: one 128-byte row of bf16
constexpr int kTmPart = 128 * 128;    // bytes of 128 rows of bf16 in a stage
constexpr int kTmW = 3 * 64 * 128;    // bytes of W in a stage: W1 (even CTA) or W2 (odd CTA), and half of W3
constexpr int kTmEpiWarps = 8;
constexpr int kTmConvWarps = 8;
constexpr int kTmMaxSplit = 8;        // pairs that share a left-over tile, about

template <bool F32>
struct TablesCfg {
    static constexpr int MT = F32 ? 1 : 2;          // row blocks of 128 a CTA works on at a time
    static constexpr int ROWS = 256 * MT;           // rows of V per tile
    static constexpr int CHUNK = F32 ? 2 : 8;       // ring stages between two emptyings of an accumulator
    static constexpr int STAGES = F32 ? 2 : 4;
    static constexpr int A_BYTES = (F32 ? 3 : MT) * kTmPart;
    static constexpr int STAGE = A_BYTES + kTmW;
    static constexpr int RAW_STAGES = F32 ? 2 : 0;  // blocks of fp32 embeddings on their way
    static constexpr int RAW = 2 * kTmPart;
    static constexpr int THREADS = (kTmEpiWarps + 2 + (F32 ? kTmConvWarps : 0)) * 32;
    static constexpr int SLOT = 32 * 64 * MT;       // running sums of one epilogue warp
    static constexpr size_t SMEM = (size_t)STAGES * STAGE + (size_t)RAW_STAGES * RAW + 1024;  // (ring on a 1024-byte boundary)
};

struct __align__(64) TablesParams {
    CUtensorMap map_w;  // [3 * m_pad, E_pad] bf16
    CUtensorMap map_e;  // [V, E] embeddings
    const float* bias;  // [m] or NULL
    float* out;         // [V, m]
    float* pieces;      // [pairs][2 pieces][2 CTAs][kTmEpiWarps][SLOT]
    int* counters;      // [pairs][2 CTAs][kTmEpiWarps], zero between calls
    int32_t* errflag;
    int V, m, m_pad, n_mb, n_kb;
    int pairs, full_rounds;
    int left, share_pairs;  // left-over tiles, pairs that share them
};

// What a pair works on: whole tiles, one in every round, then its share of the left-over tiles' blocks (the share is no
// longer than a tile, so it lies in two tiles at most).
struct TablesItem {
    int tile, kb0, kb1;
    int q0, q1;  // a piece: the first and the last pair that work on the tile (q0 == q1: the whole tile)
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
    if (i < p.full_rounds) {
        it.tile = pair + i * p.pairs;
        it.kb0 = 0;
        it.kb1 = p.n_kb;
        it.q0 = it.q1 = pair;
        return true;
    }
    if (p.left == 0 || pair >= p.share_pairs) return false;
    const int x0 = tables_share(p, pair), x1 = tables_share(p, pair + 1);
    const int t = x0 / p.n_kb + (i - p.full_rounds);
    const int b0 = t * p.n_kb, b1 = b0 + p.n_kb;
    if (b0 >= x1) return false;
    it.tile = p.full_rounds * p.pairs + t;
    it.kb0 = x0 > b0 ? x0 - b0 : 0;
    it.kb1 = x1 < b1 ? x1 - b0 : p.n_kb;
    it.seg = i - p.full_rounds;
    it.q0 = tables_owner(p, b0);
    it.q1 = tables_owner(p, b1 - 1);
    return true;
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
__device__ __forceinline__ void st_shared_v4(uint32_t at, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ float4 ld_shared_f4(uint32_t at) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(at));
    return v;
}

template <bool F32>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TablesCfg<F32>::THREADS, 1)
    tables_mma_kernel(const __grid_constant__ TablesParams p) {
    using C = TablesCfg<F32>;
    constexpr uint32_t NST = C::STAGES, NRAW = F32 ? C::RAW_STAGES : 1;
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bars[3 * NST + 2 * NRAW + 4];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_ctarank();
    const int pair = (int)blockIdx.x >> 1;
    const uint32_t ring = (smem_u32(smem_raw) + 1023u) & ~1023u, raw_ring = ring + NST * C::STAGE;
    // full: a stage's copies have landed in both CTAs (fp32: and the odd CTA's parts are written) -- the even CTA's;
    // empty: its matrix instructions are done; conv: this CTA's parts of a stage are written (fp32)
    const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * NST, conv0 = empty0 + 8 * NST;
    const uint32_t rawfull0 = conv0 + 8 * NST, rawempty0 = rawfull0 + 8 * NRAW;
    const uint32_t accfull0 = rawempty0 + 8 * NRAW, accempty0 = accfull0 + 16;
    if (tid == 0) {
        for (uint32_t s = 0; s < NST; ++s) {
            mbar_init(full0 + 8 * s, F32 ? 2 : 1);
            mbar_init(empty0 + 8 * s, 1);
            mbar_init(conv0 + 8 * s, kTmConvWarps);
        }
        for (uint32_t s = 0; s < NRAW; ++s) {
            mbar_init(rawfull0 + 8 * s, 1);
            mbar_init(rawempty0 + 8 * s, kTmConvWarps);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(accfull0 + 8 * s, 1);
            mbar_init(accempty0 + 8 * s, 2 * kTmEpiWarps);  // (the even CTA's)
        }
        mbar_fence_init();
        s_abort = 0;
    }
    if (warp == 9) tmem_alloc_pair(smem_u32(&s_tmem), 512);
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
        for (int i = 0; tables_item(p, pair, i, it); ++i) {
            const int rt = it.tile / p.n_mb, mb = it.tile - rt * p.n_mb;
            const uint32_t n = (uint32_t)((p.m - mb * 128 < 128 ? p.m - mb * 128 : 128) + 31) & ~31u;
            float acc[C::MT][64];
#pragma unroll
            for (int h = 0; h < C::MT; ++h)
#pragma unroll
                for (int c = 0; c < 64; ++c) acc[h][c] = 0.f;
            for (int kb = it.kb0; kb < it.kb1; kb += C::CHUNK, ++cc) {
#pragma unroll
                for (int h = 0; h < C::MT; ++h) {
                    const uint32_t slot = C::MT == 1 ? (cc & 1u) : (uint32_t)h;
                    mbar_wait_cluster(accfull0 + 8 * slot, (C::MT == 1 ? cc >> 1 : cc) & 1u, &s_abort);
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
                    if (lane == 0) mbar_arrive_cluster(accempty_even + 8 * slot);
                }
            }
            bool write = true;
            if (it.q0 != it.q1) {  // a piece of a left-over tile: the warp that arrives last adds the pieces up
                auto piece = [&](int q, int seg) {
                    return p.pieces + ((size_t)((q * 2 + seg) * 2 + (int)rank) * kTmEpiWarps + warp) * C::SLOT + lane;
                };
                float* mine = piece(pair, it.seg);
#pragma unroll
                for (int h = 0; h < C::MT; ++h)
#pragma unroll
                    for (int c = 0; c < 64; ++c) mine[(h * 64 + c) * 32] = acc[h][c];
                __threadfence();
                __syncwarp();
                int* cnt = p.counters + ((it.tile - p.full_rounds * p.pairs) * 2 + (int)rank) * kTmEpiWarps + warp;
                int old = 0;
                if (lane == 0) old = atomicAdd(cnt, 1);
                old = __shfl_sync(0xFFFFFFFFu, old, 0);
                write = old == it.q1 - it.q0;
                if (write) {
                    __threadfence();
                    if (lane == 0) *cnt = 0;  // ready for the next call
                    const int b0 = (it.tile - p.full_rounds * p.pairs) * p.n_kb;
#pragma unroll
                    for (int h = 0; h < C::MT; ++h)
#pragma unroll
                        for (int c = 0; c < 64; ++c) acc[h][c] = 0.f;
                    for (int q = it.q0; q <= it.q1; ++q) {
                        const float* src = piece(q, tables_share(p, q) < b0 ? 1 : 0);
#pragma unroll
                        for (int h = 0; h < C::MT; ++h)
#pragma unroll
                            for (int c = 0; c < 64; ++c) acc[h][c] += __ldcg(src + (h * 64 + c) * 32);
                    }
                }
            }
#pragma unroll
            for (int h = 0; h < C::MT; ++h) {
                const int v = rt * C::ROWS + h * 256 + (int)rank * 128 + quarter * 32 + lane;
                if (write && v < p.V) {
                    const int col0 = mb * 128 + half * 64;
                    float* dst = p.out + (size_t)v * p.m + col0;
#pragma unroll
                    for (int c = 0; c < 64; c += 4) {
                        if (col0 + c < p.m) {
                            float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (p.bias)
                                b = make_float4(__ldg(p.bias + col0 + c), __ldg(p.bias + col0 + c + 1),
                                                __ldg(p.bias + col0 + c + 2), __ldg(p.bias + col0 + c + 3));
                            *(float4*)(dst + c) = make_float4(acc[h][c] + b.x, acc[h][c + 1] + b.y, acc[h][c + 2] + b.z,
                                                              acc[h][c + 3] + b.w);
                        }
                    }
                }
            }
        }
    } else if (warp == 8) {
        // ------------------------------ TMA loads ------------------------------------------------
        if (lane == 0) {
            const uint32_t full_even = mapa_u32(full0, 0);
            uint32_t t = 0, st = 0, ph = 1, rst = 0, rph = 1;
            // fp32: an iterator of the raw blocks, which run ahead of W's
            int ri = 0, rkb = 0;
            uint32_t rt_ = 0;
            TablesItem rit;
            bool rvalid = F32 && tables_item(p, pair, 0, rit);
            if (rvalid) rkb = rit.kb0;
            auto raw_load = [&]() {
                if (!rvalid || s_abort) return;
                if (rt_ >= NRAW) mbar_wait_bounded(rawempty0 + 8 * rst, rph, &s_abort);
                if (s_abort) return;
                const int row = rit.tile / p.n_mb * C::ROWS + (int)rank * 128;
                mbar_arrive_expect_tx(rawfull0 + 8 * rst, C::RAW);
                tma_load_2d(raw_ring + rst * C::RAW, &p.map_e, rkb * kTmBlk, row, rawfull0 + 8 * rst);
                tma_load_2d(raw_ring + rst * C::RAW + kTmPart, &p.map_e, rkb * kTmBlk + 32, row, rawfull0 + 8 * rst);
                ++rt_;
                if (++rst == NRAW) {
                    rst = 0;
                    rph ^= 1;
                }
                if (++rkb == rit.kb1) {
                    rvalid = tables_item(p, pair, ++ri, rit);
                    if (rvalid) rkb = rit.kb0;
                }
            };
            if (F32) raw_load();
            for (int i = 0; tables_item(p, pair, i, it); ++i) {
                const int rt = it.tile / p.n_mb, mb = it.tile - rt * p.n_mb;
                const int n = ((p.m - mb * 128 < 128 ? p.m - mb * 128 : 128) + 31) & ~31;
                const int w12 = (int)rank * p.m_pad + mb * 128, w3 = 2 * p.m_pad + mb * 128 + (int)rank * (n >> 1);
                for (int kb = it.kb0; kb < it.kb1; ++kb, ++t) {
                    if (F32) raw_load();
                    if (t >= NST) mbar_wait_cluster(empty0 + 8 * st, ph, &s_abort);
                    if (s_abort) break;  // (no copy is started any more)
                    const uint32_t dst = ring + st * C::STAGE, dw = dst + C::A_BYTES, fb = full_even + 8 * st;
                    const int x = kb * kTmBlk;
                    if (rank == 0) mbar_arrive_expect_tx(full0 + 8 * st, 2u * (F32 ? kTmW : C::STAGE));
                    if (!F32) {
#pragma unroll
                        for (int h = 0; h < C::MT; ++h)
                            tma_load_2d_pair(dst + h * kTmPart, &p.map_e, x, rt * C::ROWS + h * 256 + (int)rank * 128, fb);
                    }
                    tma_load_2d_pair(dw, &p.map_w, x, w12, fb);
                    tma_load_2d_pair(dw + 8192, &p.map_w, x, w12 + 64, fb);
                    tma_load_2d_pair(dw + 16384, &p.map_w, x, w3, fb);
                    if (++st == NST) {
                        st = 0;
                        ph ^= 1;
                    }
                }
            }
            // every stage has been read before the CTA retires (its barriers are arrived at from the other CTA); after
            // an abort: no copy of this pair may still be in flight
            const uint32_t back = t < NST ? t : NST;
            for (uint32_t b = 0; b < back; ++b) {
                const uint32_t tt = t - back + b;
                uint32_t tries = 0;
                while (!mbar_try_wait_cluster(empty0 + 8 * (tt % NST), (tt / NST) & 1) && ++tries < GRAFT_SPIN_LIMIT) {
                    if (s_abort && tries > 4096u) break;
                }
                if (s_abort && rank == 0) {
                    tries = 0;
                    while (!mbar_try_wait_cluster(full0 + 8 * (tt % NST), (tt / NST) & 1) && ++tries < 65536u) {
                    }
                }
            }
            if (F32 && s_abort) {
                const uint32_t rback = rt_ < NRAW ? rt_ : NRAW;
                for (uint32_t b = 0; b < rback; ++b) {
                    const uint32_t tt = rt_ - rback + b;
                    uint32_t tries = 0;
                    while (!mbar_try_wait(rawfull0 + 8 * (tt % NRAW), (tt / NRAW) & 1) && ++tries < 65536u) {
                    }
                }
            }
        }
    } else if (warp == 9) {
        // ------------------------------ matrix instructions --------------------------------------
        if (rank == 0 && lane == 0) {
            uint32_t st = 0, ph = 0, cc = 0;
            for (int i = 0; tables_item(p, pair, i, it); ++i) {
                const int mb = it.tile % p.n_mb;
                const int n = ((p.m - mb * 128 < 128 ? p.m - mb * 128 : 128) + 31) & ~31;
                const uint32_t idesc2 = umma_idesc_bf16(256, 2 * n), idesc1 = umma_idesc_bf16(256, n);
                for (int kb = it.kb0; kb < it.kb1; ++kb) {
                    const bool first = (kb - it.kb0) % C::CHUNK == 0;
                    const bool last = kb + 1 == it.kb1 || (kb + 1 - it.kb0) % C::CHUNK == 0;
                    mbar_wait_cluster(full0 + 8 * st, ph, &s_abort);
                    if (F32) mbar_wait_cluster(conv0 + 8 * st, ph, &s_abort);
                    tc_fence_after();
                    const uint32_t a0 = ring + st * C::STAGE, b0 = a0 + C::A_BYTES;
                    // An instruction whose accumulator columns the one just ahead of it wrote waits for those; with two row
                    // blocks their instructions alternate, except in the first and the last block of a chunk, where the
                    // first row block goes ahead (its accumulators are emptied, or were, while the second's are filled).
                    const bool alternate = C::MT == 2 && !first && !last;
                    auto mma = [&](int h, int ks, bool w3) {
                        const uint32_t d = tmem + (C::MT == 1 ? (cc & 1u) : (uint32_t)h) * 256u;
                        const uint64_t a1 = umma_desc_sw128(a0 + h * kTmPart + 32 * ks);
                        if (w3) {
                            umma_pair(d + (uint32_t)n, a1, umma_desc_sw128(b0 + 16384 + 32 * ks), idesc1, true);
                        } else {
                            const uint64_t w12 = umma_desc_sw128(b0 + 32 * ks);
                            umma_pair(d, a1, w12, idesc2, !first || ks > 0);
                            if (F32) {
                                umma_pair(d, umma_desc_sw128(a0 + kTmPart + 32 * ks), w12, idesc2, true);
                                umma_pair(d, umma_desc_sw128(a0 + 2 * kTmPart + 32 * ks), w12, idesc2, true);
                            }
                        }
                    };
                    if (alternate) {
                        if (!s_abort) {
#pragma unroll
                            for (int ks = 0; ks < 4; ++ks) {
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
                                mbar_wait_cluster(accempty0 + 8 * slot, (turn - 1u) & 1u, &s_abort);
                                tc_fence_after();
                            }
                            if (!s_abort) {
#pragma unroll
                                for (int ks = 0; ks < 4; ++ks) {
                                    mma(h, ks, false);
                                    mma(h, ks, true);
                                }
                            }
                            if (last) umma_commit_pair(accfull0 + 8 * slot);
                        }
                    }
                    umma_commit_pair(empty0 + 8 * st);
                    if (last) ++cc;
                    if (++st == NST) {
                        st = 0;
                        ph ^= 1;
                    }
                }
            }
        } else if (F32 && rank == 1 && lane == 0) {
            // the odd CTA's parts of a stage are written: tell the even CTA
            const uint32_t full_even = mapa_u32(full0, 0);
            uint32_t st = 0, ph = 0;
            for (int i = 0; tables_item(p, pair, i, it); ++i)
                for (int kb = it.kb0; kb < it.kb1; ++kb) {
                    mbar_wait_cluster(conv0 + 8 * st, ph, &s_abort);
                    mbar_arrive_cluster(full_even + 8 * st);
                    if (++st == NST) {
                        st = 0;
                        ph ^= 1;
                    }
                }
        }
    } else if (F32) {
        // ------------------------------ fp32 embeddings -> bf16 parts ----------------------------
        const int ct = tid - (kTmEpiWarps + 2) * 32;
        const int c8 = ct & 7, r0 = ct >> 3;  // columns 8 c8 .. 8 c8 + 7 of rows r0, r0 + 32, ...
        uint32_t t = 0, st = 0, ph = 1, rst = 0, rph = 0;
        for (int i = 0; tables_item(p, pair, i, it); ++i) {
            for (int kb = it.kb0; kb < it.kb1; ++kb, ++t) {
                mbar_wait_bounded(rawfull0 + 8 * rst, rph, &s_abort);
                // a block is two boxes of 32 columns; the lanes of the second read their halves in the other order, so
                // that the eight lanes of a row touch every bank once
                const uint32_t src = raw_ring + rst * C::RAW + (uint32_t)(c8 >> 2) * kTmPart;
                float x[4][8];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int row = r0 + 32 * q;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int hh = h ^ (c8 >> 2);
                        const float4 v = ld_shared_f4(src + (uint32_t)row * 128u + (uint32_t)(((2 * (c8 & 3) + hh) ^ (row & 7)) * 16));
                        x[q][4 * h] = v.x, x[q][4 * h + 1] = v.y, x[q][4 * h + 2] = v.z, x[q][4 * h + 3] = v.w;
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(rawempty0 + 8 * rst);
                if (++rst == NRAW) {
                    rst = 0;
                    rph ^= 1;
                }
                if (t >= NST) mbar_wait_bounded(empty0 + 8 * st, ph, &s_abort);
                const uint32_t dst = ring + st * C::STAGE;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int row = r0 + 32 * q;
                    const uint32_t at = dst + (uint32_t)row * 128u + (uint32_t)((c8 ^ (row & 7)) * 16);
                    uint32_t a[4], b[4], c[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) split3(x[q][2 * k], x[q][2 * k + 1], a[k], b[k], c[k]);
                    if (c8 >> 2) {  // (the halves were read in the other order)
                        st_shared_v4(at, a[2], a[3], a[0], a[1]);
                        st_shared_v4(at + kTmPart, b[2], b[3], b[0], b[1]);
                        st_shared_v4(at + 2 * kTmPart, c[2], c[3], c[0], c[1]);
                    } else {
                        st_shared_v4(at, a[0], a[1], a[2], a[3]);
                        st_shared_v4(at + kTmPart, b[0], b[1], b[2], b[3]);
                        st_shared_v4(at + 2 * kTmPart, c[0], c[1], c[2], c[3]);
                    }
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(conv0 + 8 * st);
                if (++st == NST) {
                    st = 0;
                    ph ^= 1;
                }
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    cluster_sync();  // (the other CTA's last arrivals on this CTA's barriers, and its reads of this CTA's memory, are done)
    tc_fence_after();
    if (warp == 9) tmem_free_pair(tmem, 512);
    if (tid == 0 && s_abort) atomicOr(p.errflag, 1);
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
// [rows, cols], boxes of box_rows rows of 128 bytes, 128-byte swizzle, zeros outside
bool encode_map(CUtensorMap* map, const void* base, bool f32, uint64_t rows, uint64_t cols, uint32_t box_rows) {
    const cuuint64_t dims[2] = {cols, rows}, strides[1] = {cols * (f32 ? 4 : 2)};
    const cuuint32_t box[2] = {f32 ? 32u : 64u, box_rows}, step[2] = {1, 1};
    return encode_tiled()(map, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, step,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct TablesSizes {
    int n_mb, m_pad, E_pad, pairs;
    size_t o_pieces, o_w, total;  // (the counters stand first: their place does not depend on E)
};
TablesSizes tables_sizes(int num_sms, int E, int m) {
    TablesSizes s;
    s.n_mb = (m + 127) / 128;
    s.m_pad = 128 * s.n_mb;
    s.E_pad = (E + kTmBlk - 1) / kTmBlk * kTmBlk;
    s.pairs = num_sms / 2;
    s.o_pieces = ((size_t)s.pairs * 2 * kTmEpiWarps * sizeof(int) + 255) & ~(size_t)255;
    s.o_w = s.o_pieces + (size_t)s.pairs * 2 * 2 * kTmEpiWarps * TablesCfg<false>::SLOT * sizeof(float);
    s.total = s.o_w + (size_t)3 * s.m_pad * s.E_pad * 2;
    return s;
}

}  // namespace

// Can the tensor cores take this table?  16-byte rows for the loads and stores; anything else goes to the FMA kernel.
bool tables_mma_fits(const void* d_emb, graft_dtype dt, int E, const void* d_out) {
    return E % (dt == GRAFT_BF16 ? 8 : 4) == 0 && (((uintptr_t)d_emb | (uintptr_t)d_out) & 15) == 0 && encode_tiled() != nullptr;
}
size_t tables_mma_counter_bytes(int num_sms) { return tables_sizes(num_sms, 1, 1).o_pieces; }
size_t tables_mma_scratch_bytes(int num_sms, int E, int m) { return tables_sizes(num_sms, E, m).total; }

// out [V, m] = emb [V, E] . W^T + bias.  scratch: tables_mma_scratch_bytes, 256-byte aligned; its first
// tables_mma_counter_bytes are zero when it is first used.
cudaError_t tables_mma_launch(graft_ctx* ctx, const void* d_emb, graft_dtype dt, int E, const float* d_W, const float* d_b,
                              float* d_out, void* scratch, cudaStream_t st) {
    const int V = ctx->cfg.V, m = ctx->cfg.m;
    const TablesSizes s = tables_sizes(ctx->num_sms, E, m);
    const bool f32 = dt == GRAFT_F32;
    __nv_bfloat16* w = (__nv_bfloat16*)((char*)scratch + s.o_w);
    TablesParams p;
    if (!encode_map(&p.map_w, w, false, (uint64_t)3 * s.m_pad, s.E_pad, 64) || !encode_map(&p.map_e, d_emb, f32, V, E, 128))
        return cudaErrorUnknown;
    p.bias = d_b;
    p.out = d_out;
    p.pieces = (float*)((char*)scratch + s.o_pieces);
    p.counters = (int*)scratch;
    p.errflag = ctx->w_errflag;
    p.V = V;
    p.m = m;
    p.m_pad = s.m_pad;
    p.n_mb = s.n_mb;
    p.n_kb = s.E_pad / kTmBlk;
    p.pairs = s.pairs;
    const int rows = f32 ? TablesCfg<true>::ROWS : TablesCfg<false>::ROWS;
    const int tiles = (V + rows - 1) / rows * s.n_mb;
    p.full_rounds = tiles / s.pairs;
    p.left = tiles - p.full_rounds * s.pairs;
    // a share of the left-over tiles: at least an eighth of a tile and four ring stages, at most a tile
    long long sp = s.pairs;
    if (sp > (long long)p.left * kTmMaxSplit) sp = (long long)p.left * kTmMaxSplit;
    if (sp > (long long)p.left * p.n_kb / 4) sp = (long long)p.left * p.n_kb / 4;
    p.share_pairs = (int)(sp < p.left ? p.left : sp);
    if (p.left == 0) p.share_pairs = 1;
    weight_split_kernel<<<dim3((s.E_pad + 511) / 512, s.m_pad), 256, 0, st>>>(d_W, m, E, s.m_pad, s.E_pad, w);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (f32) {
        e = cudaFuncSetAttribute(tables_mma_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TablesCfg<true>::SMEM);
        if (e == cudaSuccess)
            e = launch_pdl(tables_mma_kernel<true>, dim3(2 * s.pairs), dim3(TablesCfg<true>::THREADS), TablesCfg<true>::SMEM, st, p);
    } else {
        e = cudaFuncSetAttribute(tables_mma_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TablesCfg<false>::SMEM);
        if (e == cudaSuccess)
            e = launch_pdl(tables_mma_kernel<false>, dim3(2 * s.pairs), dim3(TablesCfg<false>::THREADS), TablesCfg<false>::SMEM, st, p);
    }
    ctx->launches += 2;
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace graft

// Table precompute on the tensor cores: out[v] = W e_v + b (text after Eq. 6: the projections depend only on the token
// id and are computed once).  This is the one dense contraction of the method, [V, E] x [E, m].
//
// Operands are bf16 parts of the inputs: an fp32 number is the sum of three bf16 ones (8 + 8 + 8 mantissa bits), and a
// product of two bf16 numbers is exact in the fp32 accumulator.
//   bf16 embeddings: out = e W1 + e W2 + e W3               (three products a step, all exact)
//   fp32 embeddings: out = e1 W1 + (e1 W2 + e1 W3 + e2 W1 + e2 W2 + e3 W1)   (what is dropped is below 2^-23 of a term)
// so the result differs from an fp32 GEMM only by the order of the additions.  The accumulators of the tensor cores
// round less carefully than an FMA chain: they are emptied into fp32 registers every 512 columns of E, and the large
// products (e1 W1) have accumulators of their own.
//
// One kernel, persistent, a cluster of two CTAs per pair of SMs (tcgen05, cta_group::2): a pair owns a tile of 256 rows
// of V times up to 128 columns of m, and streams E in blocks of 64 through a shared-memory ring.
//   warps 0-7   empty the accumulators (TMEM, two sets of 2 x 128 columns: one is filled while the other is emptied),
//               keep the running sums (64 a thread) and write the tile
//   warp 8      TMA loads: W's parts (split once per call into scratch by weight_split_kernel), bf16 embeddings
//   warp 9      issues the matrix instructions (M = 256, N = 128: even CTA only)
//   warps 10-17 fp32 embeddings only: split them on the way from global memory to the ring, two blocks of loads in flight
// The embeddings are read from memory once; nothing but the tables is written.  What is left when the tiles do not
// divide by the pairs is split along E, and the pair that finishes a tile's last piece adds the pieces up in order.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "internal.h"
#include "umma.cuh"

namespace graft {
namespace {

constexpr int kTmTileRows = 256;      // rows of V per tile (128 per CTA)
constexpr int kTmBlk = 64;            // columns of E per ring stage: one 128-byte row of bf16
constexpr int kTmPart = 128 * 128;    // bytes of one part of the embeddings in a stage (128 rows of 128 bytes)
constexpr int kTmW = 3 * 64 * 128;    // bytes of W in a stage: this CTA's 64 rows of each part
constexpr int kTmChunk = 8;           // ring stages between two emptyings of an accumulator
constexpr int kTmEpiWarps = 8;
constexpr int kTmConvWarps = 8;
constexpr int kTmMaxSplit = 8;        // pieces a left-over tile is cut into at most
constexpr int kTmSlot = 32 * 64;      // running sums of one epilogue warp

struct __align__(64) TablesParams {
    CUtensorMap map_w;  // [3 * m_pad, E_pad] bf16
    CUtensorMap map_e;  // [V, E] bf16 (bf16 embeddings only)
    const float* emb;   // [V, E] fp32 (fp32 embeddings only)
    const float* bias;  // [m] or NULL
    float* out;         // [V, m]
    float* pieces;      // [pairs][2][kTmEpiWarps][kTmSlot]
    int* counters;      // [pairs][2][kTmEpiWarps], zero between calls
    int32_t* errflag;
    int V, E, m, m_pad, n_mb, n_kb;
    int pairs, full_rounds, left, split;  // left-over tiles, pieces of each
};

struct TablesItem {
    int tile, kb0, kb1, piece;
};
__device__ __forceinline__ bool tables_item(const TablesParams& p, int pair, int i, TablesItem& it) {
    it.piece = -1;
    it.kb0 = 0;
    it.kb1 = p.n_kb;
    if (i < p.full_rounds) {
        it.tile = pair + i * p.pairs;
        return true;
    }
    if (i > p.full_rounds || pair >= p.left * p.split) return false;
    const int q = pair / p.split, r = pair - q * p.split;
    it.tile = p.full_rounds * p.pairs + q;
    if (p.split > 1) {
        it.piece = r;
        it.kb0 = (int)((long long)r * p.n_kb / p.split);
        it.kb1 = (int)((long long)(r + 1) * p.n_kb / p.split);
    }
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
__device__ __forceinline__ void st_shared_v4(uint32_t at, const uint32_t (&v)[4]) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}

template <bool F32>
struct TablesCfg {
    static constexpr int STAGES = F32 ? 3 : 5;
    static constexpr int A_BYTES = (F32 ? 3 : 1) * kTmPart;
    static constexpr int STAGE = A_BYTES + kTmW;
    static constexpr int THREADS = (kTmEpiWarps + 2 + (F32 ? kTmConvWarps : 0)) * 32;
    static constexpr size_t SMEM = (size_t)STAGES * STAGE + 1024;  // (the ring starts on a 1024-byte boundary)
};

// Eight consecutive columns of four rows (32 apart) of a block: the share of one of the 256 splitting threads.
struct ConvRegs {
    float4 v[4][2];
};

template <bool F32>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TablesCfg<F32>::THREADS, 1)
    tables_mma_kernel(const __grid_constant__ TablesParams p) {
    using C = TablesCfg<F32>;
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bars[2 * C::STAGES + 4];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_ctarank();
    const int pair = (int)blockIdx.x >> 1;
    const uint32_t ring = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * C::STAGES;
    const uint32_t accfull0 = empty0 + 8 * C::STAGES, accempty0 = accfull0 + 16;
    if (tid == 0) {
        for (int s = 0; s < C::STAGES; ++s) {
            mbar_init(full0 + 8 * s, F32 ? 1 + 2 * kTmConvWarps : 1);  // (the even CTA's is the one that is used)
            mbar_init(empty0 + 8 * s, 1);
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
        const int half = warp >> 2, quarter = warp & 3;
        const uint32_t accempty_even = mapa_u32(accempty0, 0);
        uint32_t cc = 0;  // chunks emptied so far
        for (int i = 0; tables_item(p, pair, i, it); ++i) {
            float acc[64];
#pragma unroll
            for (int c = 0; c < 64; ++c) acc[c] = 0.f;
            for (int kb = it.kb0; kb < it.kb1; kb += kTmChunk, ++cc) {
                const uint32_t slot = cc & 1u;
                mbar_wait_cluster(accfull0 + 8 * slot, (cc >> 1) & 1u, &s_abort);
                tc_fence_after();
                const uint32_t t0 = tmem + ((uint32_t)(32 * quarter) << 16) + slot * 256u + (uint32_t)half * 64u;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
#pragma unroll
                    for (int lo = 0; lo < 2; ++lo) {
                        uint32_t d[16];
                        tmem_ld_32x16(t0 + 128u * lo + 16u * q, d);
                        tmem_wait_ld();
#pragma unroll
                        for (int c = 0; c < 16; ++c) acc[16 * q + c] += __uint_as_float(d[c]);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(accempty_even + 8 * slot);
            }
            bool write = true;
            if (it.piece >= 0) {  // a piece of a left-over tile: the warp that arrives last adds the pieces up
                const int first = (pair / p.split) * p.split;
                const size_t stride = (size_t)2 * kTmEpiWarps * kTmSlot;
                float* base = p.pieces + ((size_t)(first * 2 + (int)rank) * kTmEpiWarps + warp) * kTmSlot;
                float* mine = base + (size_t)it.piece * stride;
#pragma unroll
                for (int c = 0; c < 64; ++c) mine[c * 32 + lane] = acc[c];
                __threadfence();
                __syncwarp();
                int* cnt = p.counters + ((first * 2 + (int)rank) * kTmEpiWarps + warp);
                int old = 0;
                if (lane == 0) old = atomicAdd(cnt, 1);
                old = __shfl_sync(0xFFFFFFFFu, old, 0);
                write = old == p.split - 1;
                if (write) {
                    __threadfence();
                    if (lane == 0) *cnt = 0;  // ready for the next call
#pragma unroll
                    for (int c = 0; c < 64; ++c) acc[c] = 0.f;
                    for (int s = 0; s < p.split; ++s)
#pragma unroll
                        for (int c = 0; c < 64; ++c) acc[c] += __ldcg(base + (size_t)s * stride + c * 32 + lane);
                }
            }
            const int rt = it.tile / p.n_mb, mb = it.tile - rt * p.n_mb;
            const int v = rt * kTmTileRows + (int)rank * 128 + quarter * 32 + lane;
            if (write && v < p.V) {
                const int col0 = mb * 128 + half * 64;
                float* dst = p.out + (size_t)v * p.m + col0;
#pragma unroll
                for (int c = 0; c < 64; c += 4) {
                    if (col0 + c < p.m) {
                        float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (p.bias)
                            b = make_float4(__ldg(p.bias + col0 + c), __ldg(p.bias + col0 + c + 1), __ldg(p.bias + col0 + c + 2),
                                            __ldg(p.bias + col0 + c + 3));
                        *(float4*)(dst + c) = make_float4(acc[c] + b.x, acc[c + 1] + b.y, acc[c + 2] + b.z, acc[c + 3] + b.w);
                    }
                }
            }
        }
    } else if (warp == 8) {
        // ------------------------------ TMA loads ------------------------------------------------
        if (lane == 0) {
            const uint32_t full_even = mapa_u32(full0, 0);
            uint32_t t = 0, st = 0, ph = 1;
            for (int i = 0; tables_item(p, pair, i, it); ++i) {
                const int rt = it.tile / p.n_mb, mb = it.tile - rt * p.n_mb;
                const int mrem = p.m - mb * 128 < 128 ? p.m - mb * 128 : 128;
                const int w_row = mb * 128 + (int)rank * (((mrem + 31) & ~31) >> 1);
                for (int kb = it.kb0; kb < it.kb1; ++kb, ++t) {
                    if (t >= (uint32_t)C::STAGES) mbar_wait_cluster(empty0 + 8 * st, ph, &s_abort);
                    if (s_abort) break;  // (no copy is started any more)
                    const uint32_t dst = ring + st * C::STAGE;
                    if (rank == 0) mbar_arrive_expect_tx(full0 + 8 * st, 2u * (F32 ? kTmW : C::STAGE));
                    if (!F32) tma_load_2d_pair(dst, &p.map_e, kb * kTmBlk, rt * kTmTileRows + (int)rank * 128, full_even + 8 * st);
#pragma unroll
                    for (int j = 0; j < 3; ++j)
                        tma_load_2d_pair(dst + C::A_BYTES + j * (64 * 128), &p.map_w, kb * kTmBlk, j * p.m_pad + w_row,
                                         full_even + 8 * st);
                    if (++st == (uint32_t)C::STAGES) {
                        st = 0;
                        ph ^= 1;
                    }
                }
            }
            // every stage has been read before the CTA retires (its barriers are arrived at from the other CTA); after
            // an abort: no copy of this pair may still be in flight
            const uint32_t back = t < (uint32_t)C::STAGES ? t : (uint32_t)C::STAGES;
            for (uint32_t b = 0; b < back; ++b) {
                const uint32_t tt = t - back + b;
                uint32_t tries = 0;
                while (!mbar_try_wait_cluster(empty0 + 8 * (tt % C::STAGES), (tt / C::STAGES) & 1) && ++tries < GRAFT_SPIN_LIMIT) {
                    if (s_abort && tries > 4096u) break;
                }
                if (s_abort && rank == 0) {
                    tries = 0;
                    while (!mbar_try_wait_cluster(full0 + 8 * (tt % C::STAGES), (tt / C::STAGES) & 1) && ++tries < 65536u) {
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
                const int mrem = p.m - mb * 128 < 128 ? p.m - mb * 128 : 128;
                const uint32_t idesc = umma_idesc_bf16(256, (mrem + 31) & ~31);
                for (int kb = it.kb0; kb < it.kb1; ++kb) {
                    const uint32_t slot = cc & 1u;
                    const bool first = (kb - it.kb0) % kTmChunk == 0;
                    if (first && cc >= 2) mbar_wait_cluster(accempty0 + 8 * slot, ((cc >> 1) - 1u) & 1u, &s_abort);
                    mbar_wait_cluster(full0 + 8 * st, ph, &s_abort);
                    tc_fence_after();
                    const uint32_t a0 = ring + st * C::STAGE, b0 = a0 + C::A_BYTES;
                    const uint32_t d_hi = tmem + slot * 256u, d_lo = d_hi + 128u;
                    if (!s_abort) {
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks) {
                            const bool acc = !first || ks > 0;
                            const uint64_t a1 = umma_desc_sw128(a0 + 32 * ks), w1 = umma_desc_sw128(b0 + 32 * ks);
                            const uint64_t w2 = umma_desc_sw128(b0 + 64 * 128 + 32 * ks), w3 = umma_desc_sw128(b0 + 2 * 64 * 128 + 32 * ks);
                            umma_pair(d_hi, a1, w1, idesc, acc);
                            umma_pair(d_lo, a1, w2, idesc, acc);
                            umma_pair(d_lo, a1, w3, idesc, true);
                            if (F32) {
                                const uint64_t a2 = umma_desc_sw128(a0 + kTmPart + 32 * ks), a3 = umma_desc_sw128(a0 + 2 * kTmPart + 32 * ks);
                                umma_pair(d_lo, a2, w1, idesc, true);
                                umma_pair(d_lo, a2, w2, idesc, true);
                                umma_pair(d_lo, a3, w1, idesc, true);
                            }
                        }
                    }
                    umma_commit_pair(empty0 + 8 * st);
                    if (kb + 1 == it.kb1 || (kb + 1 - it.kb0) % kTmChunk == 0) {
                        umma_commit_pair(accfull0 + 8 * slot);
                        ++cc;
                    }
                    if (++st == (uint32_t)C::STAGES) {
                        st = 0;
                        ph ^= 1;
                    }
                }
            }
        }
    } else if (F32) {
        // ------------------------------ fp32 embeddings -> bf16 parts ----------------------------
        const int ct = tid - (kTmEpiWarps + 2) * 32;
        const int c8 = ct & 7, r0 = ct >> 3;  // columns 8 c8 .. 8 c8 + 7 of rows r0, r0 + 32, ...
        const uint32_t full_even = mapa_u32(full0, 0);
        // an iterator over (item, block) that runs two blocks ahead of the one being split
        int li = 0, lkb = 0;
        TablesItem lit;
        bool lvalid = tables_item(p, pair, 0, lit);
        if (lvalid) lkb = lit.kb0;
        auto load = [&](ConvRegs& r) {
            const int rt = lvalid ? lit.tile / p.n_mb : 0;
            const int e = lkb * kTmBlk + 8 * c8;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int v = rt * kTmTileRows + (int)rank * 128 + r0 + 32 * q;
                const float* src = p.emb + (size_t)v * p.E + e;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    r.v[q][h] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (lvalid && v < p.V && e + 4 * h < p.E) r.v[q][h] = __ldcs((const float4*)(src + 4 * h));
                }
            }
            if (lvalid && ++lkb == lit.kb1) {
                lvalid = tables_item(p, pair, ++li, lit);
                if (lvalid) lkb = lit.kb0;
            }
        };
        uint32_t t = 0, st = 0, ph = 1;
        auto split_store = [&](const ConvRegs& r) {
            if (t >= (uint32_t)C::STAGES) mbar_wait_cluster(empty0 + 8 * st, ph, &s_abort);
            const uint32_t dst = ring + st * C::STAGE;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int row = r0 + 32 * q;
                const uint32_t at = dst + (uint32_t)row * 128u + (uint32_t)((c8 ^ (row & 7)) * 16);
                uint32_t a[4], b[4], c[4];
                split3(r.v[q][0].x, r.v[q][0].y, a[0], b[0], c[0]);
                split3(r.v[q][0].z, r.v[q][0].w, a[1], b[1], c[1]);
                split3(r.v[q][1].x, r.v[q][1].y, a[2], b[2], c[2]);
                split3(r.v[q][1].z, r.v[q][1].w, a[3], b[3], c[3]);
                st_shared_v4(at, a);
                st_shared_v4(at + kTmPart, b);
                st_shared_v4(at + 2 * kTmPart, c);
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(full_even + 8 * st);
            ++t;
            if (++st == (uint32_t)C::STAGES) {
                st = 0;
                ph ^= 1;
            }
        };
        int total = 0;  // blocks of this pair
        for (int i = 0; tables_item(p, pair, i, it); ++i) total += it.kb1 - it.kb0;
        ConvRegs x, y;
        load(x);
        load(y);
        for (int n = 0; n < total; n += 2) {
            split_store(x);
            load(x);
            if (n + 1 < total) {
                split_store(y);
                load(y);
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
// [rows, cols] bf16, boxes of 64 columns x box_rows, 128-byte swizzle, zeros outside
bool encode_map(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
    const cuuint64_t dims[2] = {cols, rows}, strides[1] = {cols * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kTmBlk, box_rows}, step[2] = {1, 1};
    return encode_tiled()(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, step,
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
    s.o_w = s.o_pieces + (size_t)s.pairs * 2 * kTmEpiWarps * kTmSlot * sizeof(float);
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
    if (!encode_map(&p.map_w, w, (uint64_t)3 * s.m_pad, s.E_pad, 64)) return cudaErrorUnknown;
    p.map_e = p.map_w;
    if (!f32 && !encode_map(&p.map_e, d_emb, V, E, 128)) return cudaErrorUnknown;
    p.emb = f32 ? (const float*)d_emb : nullptr;
    p.bias = d_b;
    p.out = d_out;
    p.pieces = (float*)((char*)scratch + s.o_pieces);
    p.counters = (int*)scratch;
    p.errflag = ctx->w_errflag;
    p.V = V;
    p.E = E;
    p.m = m;
    p.m_pad = s.m_pad;
    p.n_mb = s.n_mb;
    p.n_kb = s.E_pad / kTmBlk;
    p.pairs = s.pairs;
    const int tiles = (V + kTmTileRows - 1) / kTmTileRows * s.n_mb;
    p.full_rounds = tiles / s.pairs;
    p.left = tiles - p.full_rounds * s.pairs;
    // pieces of a left-over tile: as many as there are pairs for, at least four ring stages each
    p.split = 1;
    if (p.left > 0) {
        p.split = s.pairs / p.left < kTmMaxSplit ? s.pairs / p.left : kTmMaxSplit;
        if (p.split > p.n_kb / 4) p.split = p.n_kb / 4;
        if (p.split < 1) p.split = 1;
    }
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

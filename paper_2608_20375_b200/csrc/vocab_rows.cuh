// Vocab pass, rows held in shared memory: a row of logits is loaded once, whole by one CTA or in equal pieces by a cluster
// of four, and everything else -- log-sum-exp, the bound on the K-th largest logit, the candidates above it, their ranks -- is
// worked out from shared memory.  One row a cluster; the hardware deals the rows out.
//
// The streaming kernel keeps one CTA per SM busy with a ring of tiles and finishes a segment by re-reading the chunks that
// hold its largest logits from L2, beside the stream: 4 us a segment, 3.5 more where the pieces of a row meet through global
// memory.  That is the whole time of a small input, and short rows queue for it.  Here
//   * several CTAs share an SM, so that one loads while another finishes;
//   * the vectors are still in shared memory when the bound T is known: one list of the steps of threads that reach T, one
//     look at their elements, a vector a thread (1.9 k cycles from T to the candidates; every warp on its own took 5 k, a
//     thread on its own 12 k);
//   * the pieces of a row exchange the 64 group maxima behind T (st.async into every CTA of the cluster), so that T is the
//     row's and about K + 12 candidates in all go to the first CTA, which ranks them: two exchanges of 1.3 k cycles, no global
//     memory, no counters;
//   * rows whose candidates overflow the list take what lies above the bound and then the elements equal to it in the order of their ids
//     (masked tokens, ties in bulk: V = 16,000 bf16, batch 16, 8.2 us; 6.2 without masks); where that overflows too (sorted rows) the
//     logits' bits are bisected in shared memory.
// What bounds it: batch 1 at V = 151,936 is a chain -- load 3.9 k cycles (the arithmetic of 38 k logits an SM among them), sums and
// T 1.7 k, candidates 1.6 k, second exchange 1.3 k, ranks and outputs 1.4 k -- 8.0 us a launch (12.7 by the streaming kernel).
// Many short rows: the issue slots (72 % taken by the four CTAs of an SM), 41.2 us for 131 MB at V = 16,000 (63.5).
// References of the sums are whole numbers, so that sums are brought together exactly.
#pragma once
#include "umma.cuh"
#include "vocab_common.cuh"
#include "cosine.cuh"

#ifndef GRAFT_TEST_WITHHOLD_CTA
#define GRAFT_TEST_WITHHOLD_CTA 0  // (test builds: the thread block one of whose copies is never issued)
#endif

namespace graft {

namespace {

// NT threads work on a row (or a piece of it), four 16-byte vectors each a step; one warp more: copies, cosines.
constexpr int rows_tile_vecs(int nt) { return nt * VEC_PER_LANE; }
constexpr int kRowsMaxBytes = 224 * 1024;       // the longest piece, the vectors of its ragged ends among it

constexpr int kRowsHits = 512;                  // steps of threads that can reach T before the exact selection takes over

// Candidates of a CTA at most.  A good bound leaves about K + 12 a row.
constexpr int rows_cap(int cl) { return cl == 1 ? 256 : 512 / cl; }

struct RowsParams {
    const char* logits;
    int rows, V, K;
    int32_t* topk_id;
    float* topk_lp;
    float* lse;
    int32_t* row_status;
    int32_t* errflag;
    graft_vocab_partial* partial_out;
    const void* hidden;
    int hidden_bf16, hidden_dim, L;
    double* cos_out;  // [rows / L, L], or nullptr
    int vecs;         // room for a piece: vectors of shared memory
};

template <int CL, int NT>
struct __align__(16) RowsShared {
    static constexpr int CAP = rows_cap(CL);
    static constexpr int WARPS = NT / 32, TILE = rows_tile_vecs(NT), MAX_TILES = kRowsMaxBytes / (16 * TILE);
    static_assert(kRowsMaxBytes % (16 * TILE) == 0 && MAX_TILES <= 32, "a barrier a tile, a bit a tile");
    uint64_t cand[CL * CAP];   // this CTA's candidates; in the end, in the first CTA, the row's
    uint64_t in[CL > 1 ? CL : 1][CL > 1 ? CAP : 1];  // the first CTA's: every CTA's candidates
    uint64_t outk[kMaxK];
    uint64_t full[MAX_TILES];
    uint64_t x1, x2, x3;       // the group maxima are here; the lists' first 32 candidates are; the rest of long lists is
    uint32_t gmax[kVpGroups];  // maxima of this CTA's groups of threads
    uint32_t gall[CL][kVpGroups];
    __align__(16) uint32_t gc[kVpGroups];  // the row's group maxima; the group in the low bits, so that no two are equal
    float2 lse[CL][WARPS];  // the first CTA's: reference exponent and sum of every warp
    double lse_d, C, S;        // the first CTA's: the row's log-sum-exp, its pieces
    uint32_t vmax;
    uint32_t T;
    uint32_t gmost;            // the largest group maximum, its low bits set
    uint32_t gleast;           // the least, its low bits cut off
    uint2 cnt[CL];             // the first CTA's: candidates of every CTA; has a bounded wait run out there?
    int ncand, nhits;
    uint16_t hits[kRowsHits];  // (step, thread) whose maximum reaches T
    int count[2];              // the exact selection's
    int scan[WARPS];
    volatile int abort_flag;
};

template <int NT>
__device__ __forceinline__ void rows_bar() { named_bar_sync(1, NT); }
__device__ __forceinline__ void st_async_v2(uint32_t dst, uint32_t a, uint32_t b, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.u32 [%0], {%1, %2}, [%3];" ::"r"(dst), "r"(a), "r"(b),
                 "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void st_cluster_u64(uint32_t dst, uint64_t v) {
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(dst), "l"(v) : "memory");
}

// What a CTA holds: vector 0 the elements ahead of the first 16-byte boundary, then the bulk copies, then the rest; places
// outside [e0, e1) hold -inf and are nobody's candidates.
struct RowsPiece {
    int nvec;      // vectors in all
    int e_vec0;    // the element at the beginning of vector 0 (may lie before e0)
    int e0, e1;
};

// Calls f(order-preserving image, element, whether it reaches `least`) for this thread's elements (vectors t, t + NT, ...);
// a whole warp together, so that f may count.
template <bool BF16, int NT, typename F>
__device__ __forceinline__ void rows_each(const uint4* vec, const RowsPiece& pc, uint32_t least, int tid, F f) {
    using T = VT<BF16>;
#pragma unroll 2
    for (int s0 = 0; s0 < pc.nvec; s0 += NT) {  // (uniform)
        const int s = s0 + tid;
        uint4 x = make_uint4(T::NEG_INF_WORD, T::NEG_INF_WORD, T::NEG_INF_WORD, T::NEG_INF_WORD);
        if (s < pc.nvec) x = vec[s];
        const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int j = 0; j < T::EPV; ++j) {
            const uint32_t xb = !BF16 ? w[j] : (j & 1) ? (w[j >> 1] & 0xFFFF0000u) : (w[j >> 1] << 16);
            const uint32_t o = ord_from_bits(xb);
            const int e = pc.e_vec0 + s * T::EPV + j;
            f(o, e, o >= least && e >= pc.e0 && e < pc.e1);
        }
    }
}
// A step of a streaming thread: N of its vectors into the sum and the maxima, the largest of them to *slot (fp32: rounded up to
// bf16) or returned.
template <bool BF16, int N>
__device__ __forceinline__ float rows_step(const uint4 (&v)[N], Acc& a, uint16_t* slot) {
    float m;
    if (BF16) {
        uint32_t cm = hmax2_bf16(hmax2_bf16(v[0].x, v[0].y), hmax2_bf16(v[0].z, v[0].w));
#pragma unroll
        for (int i = 1; i < N; ++i) cm = hmax2_bf16(cm, hmax2_bf16(hmax2_bf16(v[i].x, v[i].y), hmax2_bf16(v[i].z, v[i].w)));
        a.rmax = hmax2_bf16(a.rmax, cm);
        if (slot) {
            uint32_t sw;
            asm("prmt.b32 %0, %1, %1, 0x1032;" : "=r"(sw) : "r"(cm));
            *slot = (uint16_t)hmax2_bf16(cm, sw);
        }
        m = pair_max_bf16(cm);
        if (hmax2_bf16(cm, a.thr) != a.thr) acc_raise<BF16, true>(a, m);
    } else {
        m = -INFINITY;
#pragma unroll
        for (int i = 0; i < N; ++i)
            m = fmaxf(m, fmaxf(fmaxf(__uint_as_float(v[i].x), __uint_as_float(v[i].y)),
                               fmaxf(__uint_as_float(v[i].z), __uint_as_float(v[i].w))));
        a.rmax = __float_as_uint(fmaxf(__uint_as_float(a.rmax), m));
        if (slot) {
            const uint32_t mb = __float_as_uint(m);
            *slot = (uint16_t)((mb >> 31) ? (mb >> 16) : ((mb + 0xFFFFu) >> 16));
        }
        if (m > __uint_as_float(a.thr)) acc_raise<BF16, true>(a, m);
    }
    acc_add<BF16>(v, a);
    return m;
}
__device__ __forceinline__ uint64_t rows_key(uint32_t o, int e) { return ((uint64_t)o << 32) | (uint64_t)(0xFFFFFFFFu - (uint32_t)e); }

// The elements of the listed steps that reach T (ABOVE: that exceed it), to the list of candidates, a vector a thread.
template <bool BF16, bool ABOVE, int CL, int NT>
__device__ __forceinline__ void rows_take_hits(RowsShared<CL, NT>* sh, const uint4* vec, const RowsPiece& pc, int nhits, float Tf, int tid) {
    using T = VT<BF16>;
    using Sh = RowsShared<CL, NT>;
#pragma unroll 1
    for (int i = tid; i < nhits * VEC_PER_LANE; i += NT) {
        const uint32_t at = sh->hits[i / VEC_PER_LANE];
        const int s = (int)(at / NT) * Sh::TILE + (i % VEC_PER_LANE) * NT + (int)(at % NT);
        if (s >= pc.nvec) continue;
        const uint4 x = vec[s];
        const uint32_t w[4] = {x.x, x.y, x.z, x.w};
        const int e = pc.e_vec0 + s * T::EPV;
        uint32_t in = 0u;
#pragma unroll
        for (int j = 0; j < T::EPV; ++j) {
            const uint32_t xb = !BF16 ? w[j] : (j & 1) ? (w[j >> 1] & 0xFFFF0000u) : (w[j >> 1] << 16);
            in |= (ABOVE ? __uint_as_float(xb) > Tf : __uint_as_float(xb) >= Tf) ? 1u << j : 0u;
        }
        if (!ABOVE && in != 0u && (s == 0 || s == pc.nvec - 1)) {  // (places that are nobody's, which only a T of -inf lets in)
#pragma unroll
            for (int j = 0; j < T::EPV; ++j)
                if (e + j < pc.e0 || e + j >= pc.e1) in &= ~(1u << j);
        }
        if (in != 0u) {
            int pos = atomicAdd(&sh->ncand, __popc(in));
#pragma unroll 1
            for (; in != 0u; in &= in - 1u, ++pos) {
                const int j = __ffs(in) - 1;
                if (pos < Sh::CAP)
                    sh->cand[pos] = rows_key(ord_from_float(load_elem_f32((const char*)(vec + s) + j * T::ESZ, BF16)), e + j);
            }
        }
    }
}

// A piece in which more elements reach T than its list holds: leaves the list (in this CTA's memory) with the best K of the
// piece, in no order, and returns their number (K or more, or all elements of a shorter piece).  First what lies above the bound
// and then elements equal to it in the order of their ids (bulk ties, a vocabulary masked to -inf or to a low value); if what lies
// above it overflows too (a poor bound: sorted rows), a bound that keeps between K and CAP elements is bisected for, and where
// one value alone spans that gap its elements are taken in the order of their ids.  All threads of the row; out of line.
// cmax: the steps' maxima; vmax: an image that no element exceeds; fresh: nothing has been listed yet.
//
// Masked rows are ordinary work, so what lies above the bound is found as in other rows, by the steps' maxima.  (All elements by every
// thread and, in fp32, a bisection whenever the value of the masked has one of the six bits that T is cut by, took 288 us at V = 151,936,
// fp32, batch 4, where the streaming kernel takes 14.7.)
template <bool BF16, int CL, int NT>
__device__ __noinline__ int rows_select_exact(RowsShared<CL, NT>* sh, const uint4* vec, const uint16_t* cmax, const RowsPiece pc, uint32_t T,
                                              uint32_t vmax, uint32_t tmax, int K, bool fresh, uint64_t* list, int tid) {
    constexpr int CAP = RowsShared<CL, NT>::CAP;
    constexpr int SH = BF16 ? 16 : 0;  // (bf16: images that differ differ in their upper halves)
    const int warp = tid >> 5, lane = tid & 31;
    // T with the bits that it was cut by: the least of the group maxima that reach it, K or more
    {
        uint32_t least = 0xFFFFFFFFu;
#pragma unroll
        for (int h = 0; h < kVpGroups / 32; ++h) {
            uint32_t m = CL > 1 ? 0u : sh->gmax[lane + 32 * h];
#pragma unroll
            for (int i = 0; i < (CL > 1 ? CL : 0); ++i) m = max(m, sh->gall[i][lane + 32 * h]);
            if (m >= T) least = min(least, m);
        }
        T = __reduce_min_sync(0xFFFFFFFFu, least);
    }
    int n;
    {
        // the steps of threads that hold more than T, and their elements
        if (!fresh) {
            rows_bar<NT>();
            if (tid == 0) sh->ncand = sh->nhits = 0;
            rows_bar<NT>();
        }
        const float Tf = __uint_as_float(bits_from_ord(T));
        const uint32_t tb = __float_as_uint(Tf);
        // (fp32: a step's maximum is rounded up, so that one whose rounded maximum is T's has to be looked at, unless T itself is that)
        const uint32_t up = BF16 ? T : ord_from_bits((tb >> 31 ? tb >> 16 : (tb + 0xFFFFu) >> 16) << 16);
        const bool look = !BF16 && (tb & 0xFFFFu) != 0u;
        if (tmax > T) {
            uint32_t steps = 0u;
            const int ntiles = (pc.nvec + RowsShared<CL, NT>::TILE - 1) / RowsShared<CL, NT>::TILE;
#pragma unroll 1
            for (int t = 0; t < ntiles; ++t) {
                const uint32_t m = ord_from_bits((uint32_t)cmax[t * NT + tid] << 16);
                bool hit = m > up;
                if (look && m == up) {
#pragma unroll
                    for (int i = 0; i < VEC_PER_LANE; ++i) {
                        const int s = t * RowsShared<CL, NT>::TILE + i * NT + tid;
                        if (s < pc.nvec) {
                            const uint4 x = vec[s];
                            hit |= __uint_as_float(x.x) > Tf || __uint_as_float(x.y) > Tf || __uint_as_float(x.z) > Tf || __uint_as_float(x.w) > Tf;
                        }
                    }
                }
                steps |= hit ? 1u << t : 0u;
            }
            int pos = atomicAdd(&sh->nhits, __popc(steps));
#pragma unroll 1
            for (; steps != 0u; steps &= steps - 1u, ++pos)
                if (pos < kRowsHits) sh->hits[pos] = (uint16_t)((__ffs(steps) - 1) * NT + tid);
        }
        __syncwarp();
        rows_bar<NT>();
        const int nhits = sh->nhits;
        if (nhits <= kRowsHits) rows_take_hits<BF16, true>(sh, vec, pc, nhits, Tf, tid);
        __syncwarp();
        rows_bar<NT>();
        n = nhits <= kRowsHits ? sh->ncand : CAP + 1;
    }
    // the elements whose image reaches `least`, to the list; their number
    auto collect = [&](uint32_t least) {
        rows_bar<NT>();
        if (tid == 0) sh->ncand = 0;
        rows_bar<NT>();
        if (tmax >= least)
            rows_each<BF16, NT>(vec, pc, least, tid, [&](uint32_t o, int e, bool in) {
                if (!in) return;
                const int pos = atomicAdd(&sh->ncand, 1);
                if (pos < CAP) list[pos] = rows_key(o, e);
            });
        __syncwarp();
        rows_bar<NT>();
        return sh->ncand;
    };
    uint32_t lo = T >> SH, hi = 0u;  // more than CAP elements reach lo, fewer than K reach hi (0: not looked for yet)
    if (n > CAP) {
        n = collect((lo + 1u) << SH);
        if (n <= CAP && n >= K) return n;
    }
    if (n > CAP) {
        if (tid == 0) sh->count[0] = sh->count[1] = 0;
        rows_bar<NT>();
        ++lo;
        hi = (vmax >> SH) + 1u;
        int turn = 0;
        bool found = false;
#pragma unroll 1
        while (hi - lo > 1u) {
            const uint32_t mid = lo + (hi - lo) / 2u, least = mid << SH;
            int c = 0;
            if (__any_sync(0xFFFFFFFFu, tmax >= least))
                rows_each<BF16, NT>(vec, pc, least, tid, [&](uint32_t, int, bool in) { c += in ? 1 : 0; });
            c = __reduce_add_sync(0xFFFFFFFFu, c);
            if (lane == 0 && c) atomicAdd(&sh->count[turn], c);
            rows_bar<NT>();
            c = sh->count[turn];
            turn ^= 1;
            if (tid == 0) sh->count[turn] = 0;  // (read before the last barrier)
            rows_bar<NT>();
            if (c > CAP) {
                lo = mid;
            } else if (c < K) {
                hi = mid;
            } else {
                lo = mid;
                found = true;
                break;
            }
        }
        if (found) return collect(lo << SH);
        n = collect(hi << SH);
        if (n > CAP) n = CAP;  // (only if more than CAP elements are NaN: a row that is reported as bad)
    }
    if (n >= K) return n;
    // the first K - n elements equal to the value of lo, by id
    const uint32_t tie = lo, tie_ord = SH == 0 ? lo : lo >> 15 ? lo << 16 : (lo << 16) | 0xFFFFu;
#pragma unroll 1
    for (int s0 = 0; s0 < pc.nvec && n < K; s0 += NT) {  // (uniform)
        const int s = s0 + tid;
        uint32_t eq = 0u;
        uint4 x = make_uint4(0u, 0u, 0u, 0u);
        if (s < pc.nvec) x = vec[s];
        const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int j = 0; j < VT<BF16>::EPV; ++j) {
            const uint32_t xb = !BF16 ? w[j] : (j & 1) ? (w[j >> 1] & 0xFFFF0000u) : (w[j >> 1] << 16);
            const int e = pc.e_vec0 + s * VT<BF16>::EPV + j;
            if (s < pc.nvec && (ord_from_bits(xb) >> SH) == tie && e >= pc.e0 && e < pc.e1) eq |= 1u << j;
        }
        int before = __popc(eq);
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xFFFFFFFFu, before, d);
            if (lane >= d) before += o;
        }
        if (lane == 31) sh->scan[warp] = before;
        rows_bar<NT>();
        int total = 0;
        before -= __popc(eq);
#pragma unroll
        for (int i = 0; i < (NT / 32); ++i) {
            if (i < warp) before += sh->scan[i];
            total += sh->scan[i];
        }
#pragma unroll 1
        for (; eq != 0u && n + before < K; eq &= eq - 1u, ++before) {
            const int j = __ffs(eq) - 1;
            list[n + before] = rows_key(tie_ord, pc.e_vec0 + s * VT<BF16>::EPV + j);
        }
        n = n + total < K ? n + total : K;
        rows_bar<NT>();
    }
    return n;
}

template <bool BF16, int CL, int NT>
__global__ void __launch_bounds__(NT + 32, NT == 256 ? 4 : 2) vocab_rows_kernel(const RowsParams p) {
    using T = VT<BF16>;
    using Sh = RowsShared<CL, NT>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    uint4* const vec = (uint4*)smem_raw;
    Sh* const sh = (Sh*)(vec + p.vecs);
    uint16_t* const cmax = (uint16_t*)(sh + 1);  // [steps][threads]: the largest of a thread's four vectors (fp32: rounded up to bf16)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = CL > 1 ? cluster_ctarank() : 0u;
    const int row = (int)blockIdx.x / CL;
    pdl_launch_dependents();

    // the piece: whole 16-byte vectors of the row, an equal share a CTA; the first CTA also has what is ahead of them, the
    // last what is behind them
    const char* const rowp = p.logits + (size_t)row * p.V * T::ESZ;
    RowsPiece pc;
    const char* body;
    int nbody;
    {
        const uintptr_t a0 = (uintptr_t)rowp, a1 = a0 + (size_t)p.V * T::ESZ;
        uintptr_t b0 = (a0 + 15) & ~(uintptr_t)15, b1 = a1 & ~(uintptr_t)15;
        if (b1 < b0) b1 = b0;
        const int all = (int)((b1 - b0) / 16), first = (int)((b0 - a0) / T::ESZ);
        const int v0 = (int)((long long)all * rank / CL), v1 = (int)((long long)all * (rank + 1) / CL);
        body = (const char*)b0 + (size_t)v0 * 16;
        nbody = v1 - v0;
        pc.e_vec0 = first + (v0 - 1) * T::EPV;
        pc.e0 = rank == 0 ? 0 : first + v0 * T::EPV;
        pc.e1 = rank == CL - 1 ? p.V : min(p.V, first + v1 * T::EPV);
        pc.nvec = nbody + 2;
    }
    const int ntiles = (pc.nvec + Sh::TILE - 1) / Sh::TILE;
    const uint32_t full0 = smem_u32(sh->full), x1 = smem_u32(&sh->x1), x2 = smem_u32(&sh->x2), x3 = smem_u32(&sh->x3);

    if (tid == NT) {
#pragma unroll 1
        for (int t = 0; t < ntiles; ++t) mbar_init(full0 + 8 * t, 1);
        if (CL > 1) {
            mbar_init(x1, 1);
            mbar_init(x2, 1);
            mbar_init(x3, CL);
        }
        mbar_fence_init();
        if (CL > 1) {
            mbar_arrive_expect_tx(x1, CL * kVpGroups * 4 + (rank == 0 ? CL * Sh::WARPS * 8 : 0));
            if (rank == 0) mbar_arrive_expect_tx(x2, CL * (32 + 1) * 8);
        }
        sh->abort_flag = 0;
        sh->ncand = 0;
        sh->nhits = 0;
    }
    if (tid < kVpGroups) sh->gmax[tid] = 0u;
    __syncthreads();
    // this CTA's barriers are set up (the fence above orders their initialisation; a releasing arrival costs a microsecond)
    if (CL > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    pdl_wait();  // (as in the streaming kernel: nothing is read or written before the kernel ahead has completed)

    if (warp == Sh::WARPS) {
        // ------------------------------ copies, then the cosines of the SABA state -----------------
        if (lane == 0) {
            const uint64_t policy = l2_policy_evict_first();
#pragma unroll 1
            for (int t = 0; t < ntiles; ++t) {
                // vectors [t, t + 1) * Sh::TILE, as far as they are the body's [1, nbody + 1)
                const int s0 = t == 0 ? 1 : t * Sh::TILE;
                const int s1 = (t + 1) * Sh::TILE < nbody + 1 ? (t + 1) * Sh::TILE : nbody + 1;
                const uint32_t bytes = s1 > s0 ? (uint32_t)(s1 - s0) * 16u : 0u;
                mbar_arrive_expect_tx(full0 + 8 * t, bytes);
#ifdef GRAFT_TEST_WITHHOLD_TILE
                if (blockIdx.x == GRAFT_TEST_WITHHOLD_CTA && t == GRAFT_TEST_WITHHOLD_TILE) continue;  // (as in the streaming kernel: test builds only)
#endif
                if (bytes) tma_load_1d_hint(smem_u32(vec + s0), body + (size_t)(s0 - 1) * 16, bytes, full0 + 8 * t, policy);
            }
        }
        __syncwarp();
        if (CL > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (p.cos_out != nullptr && rank == CL - 1) {
            const int npairs = (p.rows / p.L) * (p.L - 1);
            if (row < npairs) {
                const int sb = row / (p.L - 1), d = row - sb * (p.L - 1);
                const double r = warp_adjacent_cosine(p.hidden, p.hidden_bf16, p.hidden_dim, ((size_t)sb * p.L + d) * p.hidden_dim, lane);
                if (lane == 0) p.cos_out[(size_t)sb * p.L + d] = r;
            }
        }
        __syncwarp();
        if (CL > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        if (CL > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        return;
    }

    // ------------------------------ the stream ---------------------------------------------------
    // the vectors that no copy brings: the elements ahead of the body and behind it (each read by the thread that writes it)
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        const int s = h == 0 ? 0 : nbody + 1;
        if (tid == s % NT) {
            uint32_t w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) w[k] = T::NEG_INF_WORD;
#pragma unroll
            for (int j = 0; j < T::EPV; ++j) {
                const int e = pc.e_vec0 + s * T::EPV + j;
                if (e >= pc.e0 && e < pc.e1) {
                    const uint32_t xb = __float_as_uint(load_elem_f32(rowp + (size_t)e * T::ESZ, BF16));
                    if (!BF16)
                        w[j] = xb;
                    else if (j & 1)
                        w[j >> 1] = (w[j >> 1] & 0xFFFFu) | xb;
                    else
                        w[j >> 1] = (w[j >> 1] & 0xFFFF0000u) | (xb >> 16);
                }
            }
            vec[s] = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
    Acc a;
    acc_init<BF16>(a);
#pragma unroll 1
    for (int t = 0; t < ntiles; ++t) {
        mbar_wait_bounded_hint(full0 + 8 * t, 0, &sh->abort_flag, 2000u);
        const int s = t * Sh::TILE + tid;
        uint16_t* const slot = cmax + t * NT + tid;
        if ((t + 1) * Sh::TILE <= pc.nvec) {  // (uniform)
            uint4 v[VEC_PER_LANE];
#pragma unroll
            for (int i = 0; i < VEC_PER_LANE; ++i) v[i] = vec[s + i * NT];
            rows_step<BF16>(v, a, slot);
        } else if (t * Sh::TILE + 2 * NT < pc.nvec) {
            uint4 v[VEC_PER_LANE];
#pragma unroll
            for (int i = 0; i < VEC_PER_LANE; ++i) {
                v[i] = make_uint4(T::NEG_INF_WORD, T::NEG_INF_WORD, T::NEG_INF_WORD, T::NEG_INF_WORD);
                if (s + i * NT < pc.nvec) v[i] = vec[s + i * NT];
            }
            rows_step<BF16>(v, a, slot);
        } else {
            // a last step of two vectors a thread or fewer: vector by vector, as far as the warp has any (V = 19,000, batch 256:
            // 48.8 -> 45.5 us; of three or four: 1 to 3 % slower than a whole step)
            float most = -INFINITY;
#pragma unroll 1
            for (int i = 0; s - lane + i * NT < pc.nvec && i < VEC_PER_LANE; ++i) {
                uint4 v[1] = {make_uint4(T::NEG_INF_WORD, T::NEG_INF_WORD, T::NEG_INF_WORD, T::NEG_INF_WORD)};
                if (s + i * NT < pc.nvec) v[0] = vec[s + i * NT];
                most = fmaxf(most, rows_step<BF16>(v, a, nullptr));
            }
            const uint32_t mb = __float_as_uint(most);
            *slot = (uint16_t)((mb >> 31) ? (mb >> 16) : ((mb + 0xFFFFu) >> 16));
        }
    }
    const uint32_t tmax = ord_from_float(BF16 ? pair_max_bf16(a.rmax) : __uint_as_float(a.rmax));
    atomicMax(&sh->gmax[tid & (kVpGroups - 1)], tmax);
    {
        // the warp's sum, at the largest reference of its lanes (references are whole numbers: exact; a thread without one has
        // added up zeros, or a NaN, which marks the row)
        const float c = __uint_as_float(bits_from_ord(__reduce_max_sync(0xFFFFFFFFu, ord_from_float(a.ref))));
        float s = acc_sum<BF16>(a) * (a.ref == -INFINITY ? 1.f : ex2_whole(a.ref - c));
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, d);
        if (lane == 0) sh->lse[CL > 1 ? rank : 0][warp] = make_float2(c, s);
    }
    rows_bar<NT>();
    if (CL > 1) {
        // every CTA gets every CTA's group maxima, the first one also the sums
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // (the others' barriers are set up: long since)
        if (warp < CL) {
            const uint32_t bar = mapa_u32(x1, warp);
            st_async_v2(mapa_u32(smem_u32(&sh->gall[rank][2 * lane]), warp), sh->gmax[2 * lane], sh->gmax[2 * lane + 1], bar);
            if (warp == 0 && lane < Sh::WARPS) {
                const float2 cs = sh->lse[rank][lane];
                st_async_v2(mapa_u32(smem_u32(&sh->lse[rank][lane]), 0), __float_as_uint(cs.x), __float_as_uint(cs.y), bar);
            }
        }
        mbar_wait_cluster(x1, 0, &sh->abort_flag);
    }
    if (tid < kVpGroups) {
        uint32_t m = CL > 1 ? 0u : sh->gmax[tid];
#pragma unroll
        for (int i = 0; i < (CL > 1 ? CL : 0); ++i) m = max(m, sh->gall[i][tid]);
        sh->gc[tid] = (m & ~(uint32_t)(kVpGroups - 1)) | (uint32_t)tid;
    }
    rows_bar<NT>();
    // ------------------------------ T: the K-th largest of the row's 64 group maxima (its low bits cut off) --------------
    // a group by four threads, each against sixteen others; no two are equal, so one of them has rank K - 1
    if (tid < 4 * kVpGroups) {
        const int g = tid >> 2;
        constexpr uint32_t low = kVpGroups - 1;
        const uint32_t mine = sh->gc[g];
        const uint4* const others = (const uint4*)sh->gc + (tid & 3) * 4;
        int r = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint4 o = others[i];
            r += (o.x > mine ? 1 : 0) + (o.y > mine ? 1 : 0) + (o.z > mine ? 1 : 0) + (o.w > mine ? 1 : 0);
        }
        r += __shfl_xor_sync(0xFFFFFFFFu, r, 1);
        r += __shfl_xor_sync(0xFFFFFFFFu, r, 2);
        if ((tid & 3) == 0) {
            if (r == p.K - 1) sh->T = mine & ~low;
            if (r == 0) sh->gmost = mine | low;
            if (r == kVpGroups - 1) sh->gleast = mine & ~low;
        }
    }
    rows_bar<NT>();
    // ------------------------------ candidates -----------------------------------------------------
    const uint32_t Tv = sh->T;
    // Where the least of the groups holds T too, the rest of the row is one value (masked tokens) or nearly so: such rows go to
    // rows_select_exact at once.
    const bool tied = sh->gleast == Tv;
    // A list of the steps of threads that reach T, about K + 12 in the row, ...
    if (!tied) {
        uint32_t steps = 0u;
        if (tmax >= Tv) {
#pragma unroll 4
            for (int t = 0; t < ntiles; ++t)
                steps |= ord_from_bits((uint32_t)cmax[t * NT + tid] << 16) >= Tv ? 1u << t : 0u;
            int pos = atomicAdd(&sh->nhits, __popc(steps));
#pragma unroll 1
            for (; steps != 0u; steps &= steps - 1u, ++pos)
                if (pos < kRowsHits) sh->hits[pos] = (uint16_t)((__ffs(steps) - 1) * NT + tid);
        }
        rows_bar<NT>();
    }
    const int nhits = tied ? 0 : sh->nhits;
    // (the same order but for NaN, which makes a row bad anyway; cut off below -inf the image is not a number's)
    const float Tf = Tv <= 0x007FFFFFu ? -INFINITY : __uint_as_float(bits_from_ord(Tv));
    // ... and their elements, a vector a thread.
    rows_take_hits<BF16, false>(sh, vec, pc, nhits <= kRowsHits ? nhits : 0, Tf, tid);
    if (warp == Sh::WARPS - 1 && rank == 0) {
        // meanwhile, one warp: the log-sum-exp
        constexpr int N = CL * Sh::WARPS, H = (N + 31) / 32;
        const float2* const all = &sh->lse[0][0];
        float2 cs[H];
        uint32_t co = 0u;
#pragma unroll
        for (int i = 0; i < H; ++i) {
            cs[i] = lane + 32 * i < N ? all[lane + 32 * i] : make_float2(-INFINITY, 0.f);
            co = max(co, ord_from_float(cs[i].x));
        }
        const float cm = __uint_as_float(bits_from_ord(__reduce_max_sync(0xFFFFFFFFu, co)));
        double S = 0.0;
#pragma unroll
        for (int i = 0; i < H; ++i) S += (double)cs[i].y * (cs[i].x == -INFINITY ? 1.0 : (double)ex2_whole(cs[i].x - cm));
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) S += __shfl_xor_sync(0xFFFFFFFFu, S, d);
        uint32_t vm = 0u;
#pragma unroll
        for (int i = 0; i < CL; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) vm = max(vm, CL > 1 ? sh->gall[i][lane + 32 * h] : sh->gmax[lane + 32 * h]);
        vm = __reduce_max_sync(0xFFFFFFFFu, vm);
        if (lane == 0) {
            sh->C = (double)cm;
            sh->S = S;
            sh->vmax = vm;
            sh->lse_d = vp_lse((double)cm, S, __uint_as_float(bits_from_ord(vm)));
        }
    }
    if (!tied) rows_bar<NT>();
    int n = tied ? 0 : sh->ncand;
    if (tied || n > Sh::CAP || nhits > kRowsHits) {  // (uniform)
        n = rows_select_exact<BF16, CL, NT>(sh, vec, cmax, pc, Tv, sh->gmost, tmax, p.K, tied, sh->cand, tid);
        rows_bar<NT>();
    }
    if (CL > 1) {
        // The first CTA gets the list: 32 entries in any case (most lists have a handful), their number, and what is more than
        // 32 by plain stores ahead of a releasing arrival, for which it waits only where some list is that long.
        const uint32_t to = mapa_u32(smem_u32(&sh->in[rank][0]), 0);
        if (n > 32) {  // (uniform)
#pragma unroll 1
            for (int i = 32 + tid; i < n; i += NT) st_cluster_u64(to + 8 * i, sh->cand[i]);
            rows_bar<NT>();
        }
        if (warp == 0) {
            const uint32_t bar = mapa_u32(x2, 0);
            const uint64_t key = lane < n ? sh->cand[lane] : 0ull;
            st_async_v2(to + 8 * lane, (uint32_t)key, (uint32_t)(key >> 32), bar);
            if (lane == 0) {
                st_async_v2(mapa_u32(smem_u32(&sh->cnt[rank]), 0), (uint32_t)n, sh->abort_flag ? 1u : 0u, bar);
#ifdef GRAFT_TEST_WITHHOLD_LISTS
                if (rank != 1)  // (test builds only: the rest of a long list is never said to be there)
#endif
                    mbar_arrive_cluster(mapa_u32(x3, 0));
            }
        }
        __syncwarp();
        if (rank == 0) mbar_wait_cluster(x2, 0, &sh->abort_flag);
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    }
    // ------------------------------ ranks, outputs (the first CTA) ---------------------------------
    if (rank == 0) {
        int total = n;
        bool internal = false;
        uint64_t* const all = sh->cand;
        if (CL > 1) {
            // the lists one behind the other; a warp moves a list (CL = 2 and 4: some do nothing)
            int before = 0, mine = 0;
            bool rest = false;
            total = 0;
#pragma unroll
            for (int i = 0; i < CL; ++i) {
                const uint2 x = sh->cnt[i];
                int c = (int)x.x;
                if (c < 0 || c > Sh::CAP) c = 0;  // (after a wait that ran out the word may be anything)
                internal |= x.y != 0u;
                rest |= c > 32;
                if (i < warp) before += c;
                if (i == warp) mine = c;
                total += c;
            }
            if (rest) mbar_wait_cluster(x3, 0, &sh->abort_flag);
            __syncwarp();
#pragma unroll 1
            for (int i = lane; i < mine; i += 32) all[before + i] = sh->in[warp][i];
            rows_bar<NT>();
        }
        // four threads a candidate, each against every fourth other: keys are distinct, so ranks are a permutation
#pragma unroll 1
        for (int i0 = 0; i0 < total; i0 += NT / 4) {
            const int i = i0 + (tid >> 2);
            const uint64_t key = i < total ? all[i] : ~0ull;
            int r = 0;
#pragma unroll 4
            for (int j = tid & 3; j < total; j += 4) r += all[j] > key ? 1 : 0;
            r += __shfl_xor_sync(0xFFFFFFFFu, r, 1);
            r += __shfl_xor_sync(0xFFFFFFFFu, r, 2);
            if (i < total && (tid & 3) == 0 && r < p.K) sh->outk[r] = key;
        }
        rows_bar<NT>();
        const int nk = total < p.K ? total : p.K;
        internal |= sh->abort_flag != 0;  // (behind the barrier: no warp of this CTA waits for anything any more)
        if (warp == 0) {
            if (p.partial_out != nullptr) {
                graft_vocab_partial* po = p.partial_out + row;
                if (lane < kMaxK) po->keys[lane] = lane < nk ? sh->outk[lane] : 0ull;
                if (lane == 0) {
                    po->c = sh->C;
                    po->s = sh->S;
                    po->vmax_ord = sh->vmax;
                    po->nkeys = (uint32_t)nk | (internal ? 0x80000000u : 0u);
                }
            } else {
                const int status = (vp_bad_row(sh->S, sh->vmax, nk, p.K) ? GRAFT_ST_BAD_LOGITS : 0) | (internal ? GRAFT_ST_INTERNAL : 0);
                vp_write_row(sh->lse_d, status, nk, p.K, lane < nk ? sh->outk[lane] : 0ull, lane, p.topk_id + (size_t)row * p.K,
                             p.topk_lp + (size_t)row * p.K, p.lse + row, p.row_status + row);
            }
        }
    }
    if (tid == 0 && sh->abort_flag) {
        atomicOr(p.errflag, 1);
        // a wait gave up: none of this CTA's copies may be in flight when it retires
#pragma unroll 1
        for (int t = 0; t < ntiles; ++t)
            for (uint32_t tries = 0; !mbar_try_wait(full0 + 8 * t, 0) && tries < GRAFT_SPIN_LIMIT; ++tries) {
            }
    }
    __syncwarp();
    // no CTA retires while another may write into its shared memory or read its words
    if (CL > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

}  // namespace

}  // namespace graft

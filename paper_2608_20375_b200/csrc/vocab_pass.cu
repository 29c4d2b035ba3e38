// Vocab pass: for every (sequence, future position) row of the drafter logits, one streaming read that
// yields log-sum-exp over the vocabulary and the K top-ranked tokens with their log-probabilities
// (Preliminaries, "DFlash one-pass marginals": q_{t,d} and c^{(r)}_{t,d}; Eq. 3's log q).
//
// Rows that fit into shared memory, and few rows of any length, are held there (vocab_rows.cuh; rows_plan below has the rule);
// the rest go through the streaming kernel of this file.
//
// Shape of the streaming kernel (sm_100a):
//   * persistent grid, one CTA per SM at most; a CTA gets whole rows where that comes out even enough, else the
//     rows*V element stream is cut into equal contiguous shares, so a CTA sees at most two partial rows plus whole
//     rows in between ("segments"; vp_make_plan has the rule);
//   * warp roles: one producer warp feeds a four-stage shared-memory ring with 32 KiB TMA bulk copies
//     (cp.async.bulk + mbarrier complete_tx); sixteen streaming warps read the ring with 16-byte shared loads;
//     two epilogue groups of four warps finish segments in turn while the
//     streaming warps are already in later ones; one warp computes the adjacent-position cosines of the SABA state (Eq. 15) beside the stream;
//   * per 32-element chunk a streaming lane takes a packed max (stored for the second stage, 2 bytes per
//     chunk), keeps a lazily rescaled reference exponent and adds 2^(z log2e - ref) with ex2.approx;
//   * top-K needs no per-element work in the stream: after the segment, the K-th largest of 64 group maxima
//     is a lower bound T for the K-th largest element; only chunks whose stored max reaches T
//     (about K of them) are re-read, their elements >= T become 64-bit keys (value desc, id asc) and the
//     exact top-K is found by rank counting.  Rows that defeat the bound: when more chunks reach T than the
//     hit list holds, T is raised to the K-th largest chunk maximum (or, where the group maxima tie, the
//     elements above T and the first ones equal to T are taken); hundreds of keys are selected by a search
//     over the key's bits instead of ranked; an overflow of the key buffer falls back to an exact selection
//     over the segment whose filter starts at T;
//   * rows shared by several CTAs are merged by the last CTA to arrive (a counter, no waiting);
//   * vocabulary-parallel use: the row's pieces are left for a merge over shards instead (vocab_merge_kernel).
// Every wait on an mbarrier is bounded; when one runs out the kernel raises an error flag and drains.
// Loops outside the stream are not unrolled unless that measured faster: the epilogue's code comes from L2 round after
// round, beside the tree kernel's (156 -> 112 KB of code, half a per cent of a round at batch 64 and 256).
#include <stdlib.h>
#include <string.h>

#include <mutex>

#include "common.cuh"
#include "internal.h"
#include "cosine.cuh"
#include "vocab_common.cuh"
#include "vocab_rows.cuh"

namespace graft {

namespace {


constexpr int NW = kVpConsumerWarps;          // streaming warps
constexpr int NT = kVpConsumers;              // streaming threads
constexpr int PROD_WARP = NW + kVpEpiWarps;  // warp index of the producer warp
constexpr int TILE = kVpTileBytes;
constexpr int WBLK = TILE / NW;               // bytes of a tile owned by one warp (2048)
static_assert(WBLK == 2048, "one warp owns 2 KiB of every tile");
static_assert(VEC_PER_LANE == WBLK / 16 / 32, "four 16-byte vectors per lane per tile");
static_assert(WBLK == 32 * 4 * 16, "the exact fall-back selection reads one warp block per batch");
constexpr uint32_t kOrdNegInf = 0x007FFFFFu;  // ord_from_bits of -inf: every finite value maps above it
constexpr uint32_t kVpIdleHintNs = 10000;  // suspend hint of the waits of the producer and epilogue warps
constexpr int COS_WARP = PROD_WARP + 1;  // warp that computes the SABA cosines beside the stream
static_assert(kVpThreads == NT + kVpEpiWarps * 32 + 64,
              "thread count = streaming warps + epilogue warps + producer warp + cosine warp");

// The eight epilogue warps work as two groups, each on a segment of its own (segments in turn).  An epilogue is a chain
// of latencies (8k cycles alone, 10k beside the stream; 20 % more with two warps instead of four).
constexpr int GROUPS = 2;
constexpr int ET = kVpEpiWarps * 32 / GROUPS;  // threads of a group
constexpr int BUFS = 2 * GROUPS;               // hand-over buffers between streaming and epilogue warps

struct VpParams {
    const char* logits;
    int rows, V, K;
    long long nq;  // quanta per row
    long long Q;   // quanta in total
    int stages;
    int n_cmax;    // chunk-max slots per buffer (two buffers): 256 threads x max_tiles
    int max_tiles; // slots per streaming thread
    VpRecord* records;
    int* row_counter;
    int32_t* topk_id;
    float* topk_lp;
    float* lse;
    int32_t* row_status;
    int32_t* errflag;
    graft_vocab_partial* partial_out;  // vocabulary-parallel use: the row's pieces go here instead of the outputs
    // adjacent-position cosines of the SABA state (Eq. 15), computed by a warp of their own beside the stream;
    // cos_out == nullptr: not asked for
    const void* hidden;
    int hidden_bf16, hidden_dim, L;
    double* cos_out;  // [rows / L, L]
    int use_hint;
};

struct Seg {
    int row, e0, e1;
    const char* body;
    uint32_t body_bytes;
    int e_body0, e_tail0;
    int ntiles;
};

__device__ __forceinline__ long long cta_start(long long g, long long Q, long long G) { return g * Q / G; }
__device__ __forceinline__ int cta_of(long long x, long long Q, long long G) {
    return (int)(((x + 1) * G + Q - 1) / Q - 1);
}

// The piece [qr0, qr1) (in quanta) of row `row`.  No division: segment boundaries are on the streaming warps' path.
template <bool BF16>
__device__ __forceinline__ Seg make_seg(const VpParams& p, int row, int qr0, int qr1) {
    using T = VT<BF16>;
    Seg s;
    s.row = row;
    s.e0 = qr0 * kVpQuantum;
    s.e1 = qr1 == (int)p.nq ? p.V : qr1 * kVpQuantum;  // the last quantum of a row also takes the remainder
    const char* a0 = p.logits + ((size_t)s.row * p.V + s.e0) * T::ESZ;
    const char* a1 = p.logits + ((size_t)s.row * p.V + s.e1) * T::ESZ;
    uintptr_t b0 = ((uintptr_t)a0 + 15) & ~(uintptr_t)15;
    uintptr_t b1 = (uintptr_t)a1 & ~(uintptr_t)15;
    if (b1 < b0) b1 = b0;
    if (b0 > (uintptr_t)a1) {  // the segment holds no 16-byte aligned address at all
        b0 = b1 = (uintptr_t)a1;
    }
    s.body = (const char*)b0;
    s.body_bytes = (uint32_t)(b1 - b0);
    s.e_body0 = s.e0 + (int)((b0 - (uintptr_t)a0) / T::ESZ);
    s.e_tail0 = s.e_body0 + (int)(s.body_bytes / T::ESZ);
    s.ntiles = (int)((s.body_bytes + TILE - 1) / TILE);
    return s;
}

// A CTA's share of the stream as a list of segments.  The share's last segment (usually a partial row that is
// shared with the next CTA) is visited FIRST, so that the cross-CTA merge of shared rows happens early instead
// of at the kernel's tail; the remaining segments follow in stream order.  Two divisions when the walk begins, none
// per segment.
struct SegIter {
    int r_first, r_last;  // rows of the share's first and last quantum
    int qr_first;         // where the share begins within r_first
    int qr_last0, qr_last1;  // the last segment's piece of r_last
    int row;              // next row of the walk over [r_first, r_last)
    int state;            // 0: emit the last segment, 1: walk, 2: nothing at all
    bool whole_last;      // the last segment is the only one (it starts where the share starts)
};
template <bool BF16>
__device__ __forceinline__ SegIter seg_iter_begin(const VpParams& p, long long q0, long long q1) {
    SegIter it;
    it.state = q0 < q1 ? 0 : 2;
    it.r_first = (int)(q0 / p.nq);
    it.qr_first = (int)(q0 - (long long)it.r_first * p.nq);
    it.r_last = (int)((q1 - 1) / p.nq);
    // the last segment starts at the last row boundary inside the share (or where the share starts)
    it.whole_last = it.r_last == it.r_first;
    it.qr_last0 = it.whole_last ? it.qr_first : 0;
    it.qr_last1 = (int)(q1 - (long long)it.r_last * p.nq);
    it.row = it.r_first;
    return it;
}
template <bool BF16>
__device__ __forceinline__ bool seg_iter_next(const VpParams& p, SegIter& it, Seg& sg) {
    if (it.state == 0) {
        sg = make_seg<BF16>(p, it.r_last, it.qr_last0, it.qr_last1);
        it.state = 1;
        return true;
    }
    if (it.state == 2 || it.row >= it.r_last) return false;
    sg = make_seg<BF16>(p, it.row, it.row == it.r_first ? it.qr_first : 0, (int)p.nq);
    ++it.row;
    return true;
}
// After seg_iter_next returned a segment: is it the one this CTA visits last?
__device__ __forceinline__ bool seg_iter_at_end(const SegIter& it) { return it.row >= it.r_last; }

// One chunk of a streaming lane: four 16-byte vectors of a tile (32 bf16 or 16 fp32 logits).  The chunk maximum goes
// to *cmax_slot for the second stage (2 bytes: the bf16 value, or the fp32 maximum rounded up to bf16).
template <bool BF16, bool GUARD>
__device__ __forceinline__ void process_chunk(const uint4* __restrict__ wb, int lane, int nvalid_vec, Acc& a,
                                              typename VT<BF16>::cm_t* cmax_slot) {
    using T = VT<BF16>;
    uint4 v[VEC_PER_LANE];
    uint32_t vm[VEC_PER_LANE];
#pragma unroll
    for (int i = 0; i < VEC_PER_LANE; ++i) {
        // A lane's chunk is 64 contiguous bytes (vectors 4 lane .. 4 lane + 3 of the warp's block), so that the second
        // stage re-reads a hit chunk as one 64-byte piece of one line instead of four sectors of four lines (random
        // DRAM accesses beside the stream cost it bandwidth).  The lanes take their four vectors in rotated order,
        // (i + lane / 2) mod 4, which spreads the eight lanes of a shared-memory phase over all bank groups.
        const int vi = 4 * lane + ((i + (lane >> 1)) & 3);
        if (!GUARD || vi < nvalid_vec)
            v[i] = wb[vi];
        else
            v[i] = make_uint4(T::NEG_INF_WORD, T::NEG_INF_WORD, T::NEG_INF_WORD, T::NEG_INF_WORD);
    }
    uint32_t cmk;
    if (BF16) {
#pragma unroll
        for (int i = 0; i < VEC_PER_LANE; ++i) vm[i] = hmax2_bf16(hmax2_bf16(v[i].x, v[i].y), hmax2_bf16(v[i].z, v[i].w));
        cmk = hmax2_bf16(hmax2_bf16(vm[0], vm[1]), hmax2_bf16(vm[2], vm[3]));
        a.rmax = hmax2_bf16(a.rmax, cmk);
        {
            // the larger half of the pair, as 16 bits: the halves swapped (one byte permute), one more packed maximum
            uint32_t sw;
            asm("prmt.b32 %0, %1, %1, 0x1032;" : "=r"(sw) : "r"(cmk));
            *cmax_slot = (typename T::cm_t)(hmax2_bf16(cmk, sw) & 0xFFFFu);
        }
        if (hmax2_bf16(cmk, a.thr) != a.thr) acc_raise<BF16>(a, pair_max_bf16(cmk));  // some half above the threshold
    } else {
        float m = -INFINITY;
#pragma unroll
        for (int i = 0; i < VEC_PER_LANE; ++i) {
            const float mi = fmaxf(fmaxf(__uint_as_float(v[i].x), __uint_as_float(v[i].y)),
                                   fmaxf(__uint_as_float(v[i].z), __uint_as_float(v[i].w)));
            vm[i] = __float_as_uint(mi);
            m = fmaxf(m, mi);
        }
        cmk = __float_as_uint(m);
        a.rmax = __float_as_uint(fmaxf(__uint_as_float(a.rmax), m));
        {
            // round toward +inf onto the bf16 grid: positive values round their magnitude up, negative ones truncate
            const uint32_t mb = cmk;
            *cmax_slot = (typename T::cm_t)((mb >> 31) ? (mb >> 16) : ((mb + 0xFFFFu) >> 16));
        }
        if (m > __uint_as_float(a.thr)) acc_raise<BF16>(a, m);
    }
    acc_add<BF16>(v, a);
}

// (c, s) pairs stand for s * 2^c; merge two of them
__device__ __forceinline__ void merge_cs(float& c, float& s, float c2, float s2) {
    const float cn = fmaxf(c, c2);
    const float f1 = (c == -INFINITY) ? 0.f : ex2_approx(c - cn);
    const float f2 = (c2 == -INFINITY) ? 0.f : ex2_approx(c2 - cn);
    s = s * f1 + s2 * f2;
    c = cn;
}


// ---- shared-memory control block ---------------------------------------------------------------
struct __align__(16) EpiShared {  // private to one epilogue group
    uint64_t cand[kVpCandCap];
    uint64_t outk[kMaxK];
    uint32_t hits[kVpHitCap];
    uint16_t hthreads[NT];  // streaming threads whose maximum reaches T
    int nhits, ncand, nht, ovf;
    int arrived;    // records of a shared row that were there before this CTA's
    int tie_groups;  // groups of threads whose maximum is T (to 16 bits): many of them means bulk ties at T
    int fill_ninf;  // the threshold fell on -inf: the candidates are the finite elements plus the first -inf ones
    int fill_tie;   // too many chunks reach the threshold T (bulk ties at T): the candidates are the elements above T
                    // plus the first elements equal to T
    uint32_t Tv;
};
struct __align__(16) VpShared {
    EpiShared epi[GROUPS];
    uint32_t tmax[BUFS][NT];  // per-thread maxima of a finished segment, one buffer per segment in flight
    uint32_t gmax[BUFS][kVpGroups];  // the same maxima folded into 64 groups (lane, warp parity); zero when idle
    float wc[BUFS][NW], ws[BUFS][NW];
    volatile int abort_flag;
};

__device__ __forceinline__ void epi_bar(int group) { named_bar_sync(2 + group, ET); }

// ---- epilogue-warp helpers (32 threads, warp-synchronous) ----------------------------------------------
// Append `key` for the lanes with pred set; returns the new count.  Entries beyond the capacity are dropped
// and *overflow is raised.
__device__ __forceinline__ int warp_append(uint64_t* buf, int n, int cap, bool pred, uint64_t key, int lane,
                                           int* overflow) {
    const uint32_t m = __ballot_sync(0xFFFFFFFFu, pred);
    if (pred) {
        const int pos = n + __popc(m & ((1u << lane) - 1u));
        if (pos < cap)
            buf[pos] = key;
        else
            *overflow = 1;
    }
    n += __popc(m);
    if (n > cap) {
        *overflow = 1;
        n = cap;
    }
    return n;
}

// Exact top-K of cand[0..n) by rank counting; result sorted descending in outk[0..min(n,K)).  Keys are
// distinct (ids are), so ranks are a permutation.  One warp's n^2 compares are most of the exact selection's time: two keys a
// lane, unrolled, unlike the loops around it (one key, not unrolled: sorted rows 140 us a launch at batch 64 against 104, ramps
// with ties 308 against 204).  Out of line: inlined, the longer code costs every ordinary launch half a per cent.
__device__ __noinline__ void warp_select_topk(EpiShared* sh, int n, int K, int lane) {
    __syncwarp();
#pragma unroll 1
    for (int i = lane; i < n; i += 64) {
        const bool two = i + 32 < n;
        const uint64_t k0 = sh->cand[i], k1 = two ? sh->cand[i + 32] : ~0ull;
        int r0 = 0, r1 = 0;
#pragma unroll 8
        for (int j = 0; j < n; ++j) {
            const uint64_t c = sh->cand[j];
            r0 += c > k0 ? 1 : 0;
            r1 += c > k1 ? 1 : 0;
        }
        if (r0 < K) sh->outk[r0] = k0;
        if (two && r1 < K) sh->outk[r1] = k1;
    }
    __syncwarp();
}

// The K-th largest chunk maximum of a segment (every streaming thread leaves one 16-bit maximum per tile), as a 16-bit
// order-preserving pattern; 0 when the segment has fewer than K chunks.  All threads of an epilogue group; two
// histogram passes of eight bits each over the idle hit list.  Out of line: rows that need it are rare.
__device__ __noinline__ uint32_t epi_kth_chunk_max(EpiShared* es, const uint16_t* cmx, int max_tiles, int ntiles, int K,
                                                   int etid, int grp) {
    uint32_t* hist = es->hits;  // [0, 256) counts, [256] the bin found, [257] the count above it
    uint32_t prefix = 0u;
    int want = K;
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
#pragma unroll 1
        for (int i = etid; i < 258; i += ET) hist[i] = 0u;
        epi_bar(grp);
#pragma unroll 1
        for (int t = etid; t < NT; t += ET) {
            const uint16_t* row = cmx + (size_t)t * max_tiles;
#pragma unroll 1
            for (int tile = 0; tile < ntiles; ++tile) {
                const uint32_t v = ord_from_bits((uint32_t)row[tile] << 16) >> 16;
                if (pass == 0)
                    atomicAdd(&hist[v >> 8], 1u);
                else if ((v >> 8) == prefix)
                    atomicAdd(&hist[v & 255u], 1u);
            }
        }
        epi_bar(grp);
        if (etid < 32) {  // the bin in which the count from the top reaches `want`: eight bins a lane
            uint32_t own = 0u;
#pragma unroll
            for (int i = 0; i < 8; ++i) own += hist[8 * etid + i];
            uint32_t above = own;  // inclusive sum over the lanes from this one up
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t o = __shfl_down_sync(0xFFFFFFFFu, above, d);
                if (etid + d < 32) above += o;
            }
            if (above >= (uint32_t)want && above - own < (uint32_t)want) {  // (one lane at most)
                uint32_t acc = above - own;
#pragma unroll 1
                for (int i = 7; i >= 0; --i) {
                    const uint32_t c = hist[8 * etid + i];
                    if (acc + c >= (uint32_t)want) {
                        hist[256] = (uint32_t)(8 * etid + i) | 0x100u;
                        hist[257] = acc;
                        break;
                    }
                    acc += c;
                }
            }
        }
        epi_bar(grp);
        const uint32_t bin = hist[256];
        if (bin == 0u) {  // fewer than K chunks (uniform)
            prefix = 0u;
            pass = 2;
        } else {
            prefix = (prefix << 8) | (bin & 255u);
            want -= (int)hist[257];
        }
        epi_bar(grp);  // (read before the next pass clears it)
    }
    return prefix;
}

// Exact top-K of cand[0..n) for hundreds of keys, K < n: ranking them against each other costs n^2 compares; here the
// K-th largest key is found by a search over its bits, two at a time with three counts each -- over the value word
// first; over the id word, among the keys of that value, only if more keys share the K-th largest value than are
// wanted -- and the K keys that reach it (keys are distinct: exactly K) are ranked into outk.  Whatever the keys'
// order or values.  All threads of an epilogue group; the counts of its warps meet in the idle hit list.  Out of
// line: rows that need it are rare.
__device__ __noinline__ void epi_select_many(EpiShared* es, int n, int K, int etid, int grp) {
    uint32_t* cnt = es->hits;                       // [2 * 16 * 3] counts of the steps, [96], [97] above / at the value, [98] kept
    uint64_t* kept = (uint64_t*)(es->hits + 128);   // [K] the keys that reach the K-th largest
    const uint32_t* word = (const uint32_t*)es->cand;  // key i: id word at 2 i, value word at 2 i + 1
#pragma unroll 1
    for (int i = etid; i < 99; i += ET) cnt[i] = 0u;
    epi_bar(grp);
    uint32_t vk = 0u, ik = 0u;  // the K-th largest key's value word and id word
    int want = K;
#pragma unroll 1
    for (int phase = 0; phase < 2; ++phase) {
        uint32_t kth = 0u;
#pragma unroll 1
        for (int step = 0; step < 16; ++step) {
            const int bit = 30 - 2 * step;
            const uint32_t t1 = kth | (1u << bit), t2 = kth | (2u << bit), t3 = kth | (3u << bit);
            int c1 = 0, c2 = 0, c3 = 0;
#pragma unroll 2
            for (int i = etid; i < n; i += ET) {
                const uint32_t hi = word[2 * i + 1];
                const uint32_t x = phase == 0 ? hi : (hi == vk ? word[2 * i] : 0u);  // (an id word is never 0)
                c1 += (x >= t1) ? 1 : 0;
                c2 += (x >= t2) ? 1 : 0;
                c3 += (x >= t3) ? 1 : 0;
            }
            c1 = __reduce_add_sync(0xFFFFFFFFu, c1);
            c2 = __reduce_add_sync(0xFFFFFFFFu, c2);
            c3 = __reduce_add_sync(0xFFFFFFFFu, c3);
            uint32_t* slot = cnt + (phase * 16 + step) * 3;
            if ((etid & 31) == 0) {
                atomicAdd(&slot[0], (uint32_t)c1);
                atomicAdd(&slot[1], (uint32_t)c2);
                atomicAdd(&slot[2], (uint32_t)c3);
            }
            epi_bar(grp);
            const int n1 = (int)slot[0], n2 = (int)slot[1], n3 = (int)slot[2];
            kth = n3 >= want ? t3 : (n2 >= want ? t2 : (n1 >= want ? t1 : kth));
        }
        if (phase == 1) {
            ik = kth;
            break;
        }
        vk = kth;
        int above = 0, at = 0;
#pragma unroll 1
        for (int i = etid; i < n; i += ET) {
            const uint32_t hi = word[2 * i + 1];
            above += (hi > vk) ? 1 : 0;
            at += (hi == vk) ? 1 : 0;
        }
        above = __reduce_add_sync(0xFFFFFFFFu, above);
        at = __reduce_add_sync(0xFFFFFFFFu, at);
        if ((etid & 31) == 0) {
            atomicAdd(&cnt[96], (uint32_t)above);
            atomicAdd(&cnt[97], (uint32_t)at);
        }
        epi_bar(grp);
        want = K - (int)cnt[96];
        if ((int)cnt[97] == want) break;  // (uniform) every key of that value is wanted: ik = 0 lets them all through
    }
    const uint64_t kth_key = ((uint64_t)vk << 32) | ik;
#pragma unroll 1
    for (int i = etid; i < n; i += ET) {
        const uint64_t k = es->cand[i];
        if (k >= kth_key) {
            const uint32_t pos = atomicAdd(&cnt[98], 1u);
            if (pos < (uint32_t)kMaxK) kept[pos] = k;
        }
    }
    epi_bar(grp);
    const int m = (int)cnt[98] < K ? (int)cnt[98] : K;
    if (etid < m) {
        const uint64_t k = kept[etid];
        int rank = 0;
#pragma unroll 1
        for (int j2 = 0; j2 < m; ++j2) rank += (kept[j2] > k) ? 1 : 0;
        es->outk[rank] = k;
    }
}

// ord() of the largest element of a 16-byte vector
template <bool BF16>
__device__ __forceinline__ uint32_t vec_max_ord(const uint4& x) {
    if (BF16) return ord_from_float(pair_max_bf16(hmax2_bf16(hmax2_bf16(x.x, x.y), hmax2_bf16(x.z, x.w))));
    return ord_from_float(fmaxf(fmaxf(__uint_as_float(x.x), __uint_as_float(x.y)),
                                fmaxf(__uint_as_float(x.z), __uint_as_float(x.w))));
}

// Exact selection over a whole segment straight from global memory.  Used only when the fast path's buffers
// overflowed, which means that most of the segment ties with its K-th largest element (rows that are flat, masked
// to -inf, or all but one element equal).  The running K-th best key is the filter: an element enters the buffer
// only if its key (value, then smaller id) beats it, and once the first K of a flat row are in, nothing else does.
// The segment's 16-byte aligned body is read in batches of one streaming warp's 2 KiB of a tile; a batch whose
// chunk maxima (left by the streaming warps) rule out a key above the filter is not read at all; the few elements
// before and after the body go one by one.
// When the buffer fills up, the best K are kept and the filter rises.
template <bool BF16>
__device__ int warp_fallback_select(EpiShared* sh, const VpParams& p, const Seg& sg,
                                    const typename VT<BF16>::cm_t* cmx, int lane, uint64_t thr) {
    using T = VT<BF16>;
    const int K = p.K;
    const char* rowp = p.logits + (size_t)sg.row * p.V * T::ESZ;
    // thr: keys must beat this one (on entry: what the threshold T of the fast path rules out, or 0)
    int n = 0, ovf = 0;
    // ranking n keys against each other costs n^2 / 32 steps per lane: the buffer is cut back to its best K well
    // before it is full (96 more keys at a time)
    constexpr int kFallbackFill = 128 - 32;
    auto shrink = [&]() {  // keep the best K of the buffer
        if (n > K) {
            warp_select_topk(sh, n, K, lane);
            if (lane < K) sh->cand[lane] = sh->outk[lane];
            thr = sh->outk[K - 1];
            n = K;
            __syncwarp();
        }
    };
    auto one_by_one = [&](int e_begin, int e_end) {
#pragma unroll 1
        for (int e0 = e_begin; e0 < e_end; e0 += 32) {
            const int e = e0 + lane;
            uint64_t key = 0;
            if (e < e_end) key = make_key(__float_as_uint(load_elem_f32(rowp + (size_t)e * T::ESZ, BF16)), (uint32_t)e);
            n = warp_append(sh->cand, n, kVpCandCap, e < e_end && key > thr, key, lane, &ovf);
            if (n > kFallbackFill) shrink();
        }
    };
    one_by_one(sg.e0, sg.e_body0);
    constexpr int U = 4;
    const int nvec = (int)(sg.body_bytes / 16);
    const uint4* body = (const uint4*)sg.body;
#pragma unroll 1
    for (int v0 = 0; v0 < nvec; v0 += 32 * U) {
        // The batch is one streaming warp's 2 KiB of a tile, and this lane's four consecutive vectors are the chunk whose
        // maximum (rounded up to bf16) that warp's lane left in cmx.  A chunk cannot hold a key above the filter if
        // its maximum is below the filter's value, or not above it while all its ids come after the filter's id.
        if (thr != 0ull) {
            const int tile = v0 / (TILE / 16), wb = (v0 % (TILE / 16)) / (32 * U);
            const uint32_t mx = ord_from_bits((uint32_t)cmx[(size_t)(wb * 32 + lane) * p.max_tiles + tile] << 16);
            const uint32_t v_thr = (uint32_t)(thr >> 32);
            const uint32_t first_id = (uint32_t)(sg.e_body0 + (v0 + 4 * lane) * T::EPV);
            const bool need = !(mx < v_thr || (mx <= v_thr && first_id > key_id(thr)));
            if (!__any_sync(0xFFFFFFFFu, need)) continue;  // (uniform)
        }
#pragma unroll 1
        for (int u = 0; u < U; ++u) {  // (one vector at a time: this path must not cost the kernel registers)
            const int v = v0 + u * 32 + lane;
            uint4 x = make_uint4(T::NEG_INF_WORD, T::NEG_INF_WORD, T::NEG_INF_WORD, T::NEG_INF_WORD);
            if (v < nvec) x = body[v];
            const uint32_t wv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int q = 0; q < T::EPV; ++q) {
                uint32_t xb;
                if (BF16)
                    xb = (q & 1) ? (wv[q >> 1] & 0xFFFF0000u) : (wv[q >> 1] << 16);
                else
                    xb = wv[q];
                const uint64_t key = v < nvec ? make_key(xb, (uint32_t)(sg.e_body0 + v * T::EPV + q)) : 0ull;
                n = warp_append(sh->cand, n, kVpCandCap, key > thr, key, lane, &ovf);
                if (n > kFallbackFill) shrink();  // (uniform)
            }
        }
    }
    one_by_one(sg.e_tail0, sg.e1);
    warp_select_topk(sh, n, K, lane);
    return n < K ? n : K;
}

template <bool BF16>
__global__ void __launch_bounds__(kVpThreads, 1) vocab_pass_kernel(const VpParams p) {
    using T = VT<BF16>;
    using cm_t = typename T::cm_t;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    pdl_launch_dependents();  // the edge-score kernel's CTAs may move in as this grid's CTAs leave; they wait for it
    unsigned char* ring = smem_raw;
    uint64_t* bars = (uint64_t*)(ring + (size_t)p.stages * TILE);  // full[8], empty[8], ready[BUFS], done[BUFS]
    VpShared* sh = (VpShared*)(bars + 16 + 2 * BUFS);
    cm_t* cmax = (cm_t*)(sh + 1);  // [BUFS][n_cmax]

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const long long G = gridDim.x;
    const long long q0 = cta_start(blockIdx.x, p.Q, G), q1 = cta_start(blockIdx.x + 1, p.Q, G);
    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + 8);
    const uint32_t ready0 = smem_u32(bars + 16), done0 = smem_u32(bars + 16 + BUFS);

    if (tid == 0) {
#pragma unroll 1
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, NW);
        }
#pragma unroll 1
        for (int s = 0; s < BUFS; ++s) {
            mbar_init(ready0 + 8 * s, NW);
            mbar_init(done0 + 8 * s, 1);
        }
        mbar_fence_init();
        sh->abort_flag = 0;
    }
    if (tid < BUFS * kVpGroups) (&sh->gmax[0][0])[tid] = 0u;
    __syncthreads();
    // Launched with programmatic stream serialization inside a round: the CTA is set up while the kernel ahead of it in
    // the stream (the previous round's walk or tree kernel) drains; nothing is read or written before that kernel has
    // completed (the logits may come from it, and the scratch this kernel writes is read by the previous round's
    // kernels).  Launched the ordinary way this returns at once.
    pdl_wait();

    if (warp == PROD_WARP) {
        // ------------------------------ producer warp --------------------------------------------
        if (lane == 0) {
            uint64_t policy = 0;
            if (p.use_hint) policy = l2_policy_evict_first();
            uint32_t t = 0, st = 0, ph = 1;  // ph: parity of the "empty" phase to wait for (first lap: none)
            const uint32_t nst = (uint32_t)p.stages;
            SegIter it = seg_iter_begin<BF16>(p, q0, q1);
            Seg sg;
            while (seg_iter_next<BF16>(p, it, sg)) {
                // the segment this CTA visits last is read the ordinary way instead of evict-first: the second
                // stage of its epilogue, which nothing overlaps any more, then finds its chunks in L2
                const bool hint = p.use_hint && !seg_iter_at_end(it);
#pragma unroll 1
                for (int tile = 0; tile < sg.ntiles; ++tile, ++t) {
                    if (t >= nst) mbar_wait_bounded_hint(empty0 + 8 * st, ph, &sh->abort_flag, kVpIdleHintNs);
#ifdef GRAFT_TEST_WITHHOLD_TILE
                    // Test builds only (the shipped library is never compiled with this): CTA 0 does not issue the
                    // copy of one of its tiles, so that the streaming warps' bounded wait for it runs out and the
                    // time-out path (error flag, status bit, drain) can be exercised without faulting anything.
                    if (blockIdx.x == 0 && t == GRAFT_TEST_WITHHOLD_TILE) {
                        if (++st == nst) {
                            st = 0;
                            ph ^= 1;
                        }
                        continue;
                    }
#endif
                    uint32_t off = (uint32_t)tile * TILE;
                    uint32_t bytes = sg.body_bytes - off < (uint32_t)TILE ? sg.body_bytes - off : (uint32_t)TILE;
                    mbar_arrive_expect_tx(full0 + 8 * st, bytes);
                    if (hint)
                        tma_load_1d_hint(smem_u32(ring + (size_t)st * TILE), sg.body + off, bytes, full0 + 8 * st, policy);
                    else
                        tma_load_1d(smem_u32(ring + (size_t)st * TILE), sg.body + off, bytes, full0 + 8 * st);
                    if (++st == nst) {
                        st = 0;
                        ph ^= 1;
                    }
                }
            }
            if (sh->abort_flag) {
                // a consumer gave up: make sure none of our copies is still in flight before the CTA retires
#pragma unroll 1
                for (uint32_t back = 0; back < nst && back < t; ++back) {
                    const uint32_t tt = t - 1 - back;
                    uint32_t tries = 0;
                    while (!mbar_try_wait(full0 + 8 * (tt % nst), (tt / nst) & 1) && ++tries < GRAFT_SPIN_LIMIT) {
                    }
                }
            }
        }
    } else if (warp < NW) {
        // ------------------------------ streaming warps ------------------------------------------
        uint32_t st = 0, ph = 0;  // ring position and parity of the "full" phase to wait for
        const uint32_t nst = (uint32_t)p.stages;
        uint32_t k = 0;           // segment counter: hand-over buffers are indexed by k % BUFS
        SegIter it = seg_iter_begin<BF16>(p, q0, q1);
        Seg sg;
#pragma unroll 1
        for (; seg_iter_next<BF16>(p, it, sg); ++k) {
            const uint32_t pb = k % BUFS;
            Acc a;
            acc_init<BF16>(a);
            // buffer pb is free once the epilogue of segment k - BUFS is done
            if (k >= BUFS) mbar_wait_bounded(done0 + 8 * pb, ((k / BUFS) - 1u) & 1u, &sh->abort_flag);
            {
                const int nfull = (int)(sg.body_bytes / TILE);
                cm_t* slot = cmax + (size_t)pb * p.n_cmax + (size_t)tid * p.max_tiles;  // this thread's slots, by tile
#pragma unroll 1
                for (int tile = 0; tile < sg.ntiles; ++tile, ++slot) {
                    mbar_wait_bounded_hint(full0 + 8 * st, ph, &sh->abort_flag, 2000u);
                    const uint4* wb = (const uint4*)(ring + (size_t)st * TILE + (size_t)warp * WBLK);
                    if (tile < nfull) {
                        process_chunk<BF16, false>(wb, lane, 0, a, slot);
                    } else {
                        int nv = ((int)(sg.body_bytes - (uint32_t)tile * TILE) - warp * WBLK) / 16;
                        nv = nv < 0 ? 0 : (nv > WBLK / 16 ? WBLK / 16 : nv);
                        process_chunk<BF16, true>(wb, lane, nv, a, slot);
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(empty0 + 8 * st);
                    if (++st == nst) {
                        st = 0;
                        ph ^= 1;
                    }
                }
            }
            // hand the segment over to the epilogue warp
            // (a thread that saw no data keeps 0 = nothing seen)
            const uint32_t tmo = sg.ntiles > 0 ? ord_from_float(BF16 ? pair_max_bf16(a.rmax) : __uint_as_float(a.rmax)) : 0u;
            sh->tmax[pb][tid] = tmo;
            atomicMax(&sh->gmax[pb][(warp & 1) * 32 + lane], tmo);
            {
                // the warp's piece of the log-sum-exp: the largest reference of its lanes (one integer reduction over
                // the order-preserving images), every lane's sum rescaled to it once, then a butterfly of plain adds
                // (a fixed order: the result does not depend on timing).  A lane without a reference has added up zeros, or a
                // NaN, which marks the row.
                const uint32_t co = __reduce_max_sync(0xFFFFFFFFu, ord_from_float(a.ref));
                const float c = __uint_as_float(bits_from_ord(co));
                float s = acc_sum<BF16>(a) * (a.ref == -INFINITY ? 1.f : ex2_approx(a.ref - c));
#pragma unroll
                for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, d);
                if (lane == 0) {
                    sh->wc[pb][warp] = c;
                    sh->ws[pb][warp] = s;
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(ready0 + 8 * pb);
        }
    } else if (warp == COS_WARP) {
        // ------------------------------ cosine warp ----------------------------------------------
        // Adjacent-position cosines of the SABA state (Eq. 15): a few pairs of hidden-state rows per CTA, read
        // beside the logits stream (under 3 % of its bytes) so that nothing downstream waits for them.
        if (p.cos_out != nullptr) {
            const int npairs = (p.rows / p.L) * (p.L - 1);
#pragma unroll 1
            for (int q = (int)blockIdx.x; q < npairs; q += (int)gridDim.x) {
                const int sb = q / (p.L - 1), d = q - sb * (p.L - 1);
                const double r = warp_adjacent_cosine(p.hidden, p.hidden_bf16, p.hidden_dim,
                                                      ((size_t)sb * p.L + d) * p.hidden_dim, lane);
                if (lane == 0) p.cos_out[(size_t)sb * p.L + d] = r;
            }
        }
    } else {
        // ------------------------------ epilogue groups ----------------------------------------
        // Group g finishes the segments with k % GROUPS == g, so a group has GROUPS segment times for one epilogue.
        // Warp 0 of a group owns the hand-over barriers and the sequential parts; the data-parallel parts (which
        // chunks reach T, re-reading them, ranking the candidates) are shared by the group's threads.
        const int grp = (warp - NW) / (ET / 32), ew = (warp - NW) % (ET / 32);
        const int etid = (tid - NT) % ET;
        EpiShared* const es = &sh->epi[grp];
        uint32_t k = 0;
        SegIter it = seg_iter_begin<BF16>(p, q0, q1);
        const int my_first_row = it.r_first;
        Seg sg;
#pragma unroll 1
        for (; seg_iter_next<BF16>(p, it, sg); ++k) {
            if ((int)(k % GROUPS) != grp) continue;
            const uint32_t pb = k % BUFS;
            const char* rowp = p.logits + (size_t)sg.row * p.V * T::ESZ;
            const cm_t* cmx = cmax + (size_t)pb * p.n_cmax;
            if (ew == 0) mbar_wait_bounded_hint(ready0 + 8 * pb, (k / BUFS) & 1u, &sh->abort_flag, kVpIdleHintNs);
            float c = -INFINITY, s = 0.f;
            uint32_t vmo = 0;
            if (ew == 0) {
                int overflow = 0, ncand = 0;
                // (a) log-sum-exp pieces of the streaming warps
                c = lane < NW ? sh->wc[pb][lane] : -INFINITY;
                s = lane < NW ? sh->ws[pb][lane] : 0.f;
                // (b) ragged head / tail that the 16-byte bulk copies cannot carry: plain loads, every element a
                //     candidate (at most 7 + 7 elements unless the whole segment is shorter than 16 bytes)
                {
                    const int nhead = sg.e_body0 - sg.e0, ntail = sg.e1 - sg.e_tail0;
#pragma unroll 1
                    for (int i0 = 0; i0 < nhead + ntail; i0 += 32) {
                        const int i = i0 + lane;
                        const bool in = i < nhead + ntail;
                        uint64_t key = 0;
                        if (in) {
                            const int e = i < nhead ? sg.e0 + i : sg.e_tail0 + (i - nhead);
                            const float x = load_elem_f32(rowp + (size_t)e * T::ESZ, BF16);
                            const uint32_t o = ord_from_float(x);
                            vmo = o > vmo ? o : vmo;
                            // x log2(e) = c1 + r with c1 the rounded product and r its exact remainder (one FMA):
                            // 2^r = 1 + r ln 2 keeps what the rounding of c1 drops (up to 2e-6 of the term at
                            // |x| = 30, which is the whole error of the row when its largest logit sits here)
                            float c1 = __fmul_rn(x, kLog2e);
                            float s1 = fmaf(fmaf(x, kLog2e, -c1), 0.69314718f, 1.0f);
                            if (c1 == -INFINITY) {  // (-inf, or a finite value whose term is 0 and whose remainder is infinite)
                                s1 = 0.f;
                            } else if (!(x < INFINITY)) {
                                s1 = NAN;  // +inf or NaN poisons the sum and marks the row
                                c1 = 0.f;
                            }
                            merge_cs(c, s, c1, s1);
                            key = make_key(__float_as_uint(x), (uint32_t)e);
                        }
                        ncand = warp_append(es->cand, ncand, kVpCandCap, in, key, lane, &overflow);
                    }
                }
                // (c) T = the K-th largest group maximum, truncated to its top 16 bits: a lower bound of
                //     the K-th largest element of the segment's body (0 when fewer than K threads saw data)
                uint32_t Tv = 0;
                int tie_groups = 0;
                {
                    // over 64 group maxima rather than the 512 thread maxima: any partition of the elements into
                    // at least K groups gives a lower bound, and this one costs an eighth of the compares for about
                    // a third more candidates (groups = (lane, warp parity), so that a segment that only reaches
                    // two streaming warps still fills all of them)
                    uint32_t mine[kVpGroups / 32];
#pragma unroll
                    for (int i = 0; i < kVpGroups / 32; ++i) {
                        mine[i] = sh->gmax[pb][i * 32 + lane];
                        sh->gmax[pb][i * 32 + lane] = 0u;  // idle again (published by the `done` arrival below)
                        vmo = mine[i] > vmo ? mine[i] : vmo;
                    }
#pragma unroll 1
                    for (int bit = 30; bit >= 16; bit -= 2) {  // two bits per step: three independent counts
                        const uint32_t t1 = Tv | (1u << bit), t2 = Tv | (2u << bit), t3 = Tv | (3u << bit);
                        int c1 = 0, c2 = 0, c3 = 0;
#pragma unroll
                        for (int i = 0; i < kVpGroups / 32; ++i) {
                            c1 += (mine[i] >= t1) ? 1 : 0;
                            c2 += (mine[i] >= t2) ? 1 : 0;
                            c3 += (mine[i] >= t3) ? 1 : 0;
                        }
                        c1 = __reduce_add_sync(0xFFFFFFFFu, c1);
                        c2 = __reduce_add_sync(0xFFFFFFFFu, c2);
                        c3 = __reduce_add_sync(0xFFFFFFFFu, c3);
                        Tv = c3 >= p.K ? t3 : (c2 >= p.K ? t2 : (c1 >= p.K ? t1 : Tv));
                    }
#pragma unroll
                    for (int i = 0; i < kVpGroups / 32; ++i) tie_groups += ((mine[i] ^ Tv) >> 16) == 0u ? 1 : 0;
                    tie_groups = __reduce_add_sync(0xFFFFFFFFu, tie_groups);
                }
                // fold (c, s, max) across the warp
#pragma unroll
                for (int d = 16; d > 0; d >>= 1) {
                    const float c2 = __shfl_xor_sync(0xFFFFFFFFu, c, d);
                    const float s2 = __shfl_xor_sync(0xFFFFFFFFu, s, d);
                    merge_cs(c, s, c2, s2);
                }
                vmo = __reduce_max_sync(0xFFFFFFFFu, vmo);
                overflow = __any_sync(0xFFFFFFFFu, overflow);
                // A threshold at -inf (a vocabulary masked down to fewer finite tokens than the filter needs) would let
                // every element through.  The K best are then the finite elements and, after them, the -inf elements
                // of smallest id: the filter rises to the lowest finite value and the first K -inf elements of the
                // segment are added below.
                const bool ninf = Tv <= kOrdNegInf;
                if (ninf) Tv = kOrdNegInf + 1u;
                if (lane == 0) {
                    es->fill_ninf = ninf ? 1 : 0;
                    es->fill_tie = 0;
                    es->Tv = Tv;
                    es->nhits = 0;
                    es->nht = 0;
                    es->ncand = ncand;
                    es->ovf = overflow;
                    es->tie_groups = tie_groups;
                }
            }
            epi_bar(grp);
            uint32_t Tv = es->Tv;
            // (d) chunks whose stored maximum reaches T: only threads whose own maximum reaches T can have one.
            //     List positions come from shared-memory atomics (the order does not matter: the final selection
            //     ranks exact keys).  A hit is recorded as the byte offset of the chunk's first vector.
#pragma unroll 1
            for (int t = etid; t < NT; t += ET) {
                const uint32_t x = sh->tmax[pb][t];
                if (x >= Tv && x != 0u) es->hthreads[atomicAdd(&es->nht, 1)] = (uint16_t)t;
            }
            epi_bar(grp);
            // Te: what a chunk's maximum (and, below, an element) must reach.  T itself at first.  If more chunks reach T
            // than the list holds, either thousands of elements tie with T (a flat rest under a few winners: most of the
            // 64 group maxima are T itself) or T is a poor bound (the groups of threads are a partition that a pattern in
            // step with the lanes defeats: a row of ramps as long as a warp's block leaves half the groups' maxima far down
            // every ramp).  Ties: the scan is repeated for what lies above T, and the first elements equal to T in id
            // order are taken by a walk over the chunks further down.  A poor bound: T is raised to the K-th largest chunk
            // maximum, the best bound the chunk maxima give, and the scan is repeated.  Whichever comes first, the other
            // follows if the list overflows again: four scans at most, then the exact selection.
            uint32_t Te = Tv;
            bool refined = false, tied = false;
#pragma unroll 1
            for (int pass = 0;; ++pass) {  // (uniform)
                // (listed thread, tile) pairs, four per thread at a time with their loads in flight together; the pair's
                // thread comes from a multiplication (idx / ntiles for idx < 2^16 and ntiles < 2^16, exactly)
                const int npairs = es->nht * sg.ntiles;
                const uint32_t magic = sg.ntiles > 1 ? 0xFFFFFFFFu / (uint32_t)sg.ntiles + 1u : 0u;  // ceil(2^32 / ntiles)
                constexpr int PU = 4;
                bool stop = false;
#pragma unroll 1
                for (int base = 0; base < npairs && !stop; base += ET * PU) {
                    uint32_t raw[PU], off[PU];
#pragma unroll
                    for (int u = 0; u < PU; ++u) {
                        const int idx = base + u * ET + etid;
                        raw[u] = 0u;
                        off[u] = 0u;
                        if (idx < npairs) {
                            const int h = sg.ntiles > 1 ? (int)__umulhi((uint32_t)idx, magic) : idx, tile = idx - h * sg.ntiles;
                            const uint32_t t = es->hthreads[h];
                            raw[u] = cmx[(size_t)t * p.max_tiles + tile];
                            off[u] = (uint32_t)tile * TILE + (t >> 5) * WBLK + (t & 31) * 64;
                        }
                    }
#pragma unroll
                    for (int u = 0; u < PU; ++u) {
                        if (ord_from_bits(raw[u] << 16) >= Te && base + u * ET + etid < npairs && !stop) {
                            const int pos = atomicAdd(&es->nhits, 1);
                            if (pos >= kVpHitCap)
                                stop = true;  // too many: the exact selection over the segment takes over
                            else
                                es->hits[pos] = off[u];
                        }
                    }
                }
                epi_bar(grp);
                // (a list several times as long as a good bound leaves it -- about K chunks -- also says that T is poor:
                // its chunks would overflow the key buffer)
                const bool over = es->nhits > kVpHitCap;
                if (es->fill_ninf || (refined && tied)) break;  // (uniform)
                if (!over && !(pass == 0 && es->nhits > 5 * p.K && es->tie_groups < 16)) break;  // (uniform)
                epi_bar(grp);  // (everybody has read the count)
                if (!refined && (tied || !BF16 || es->tie_groups < 16)) {
                    uint32_t kth = epi_kth_chunk_max(es, cmx, p.max_tiles, sg.ntiles, p.K, etid, grp);
                    // (fp32 logits: the stored maxima are rounded up to bf16, the pattern below is a bound)
                    if (!BF16 && kth > 0u) kth -= 1u;
                    refined = true;
                    if ((kth << 16) > Tv || !over) {  // (uniform; the search used the hit list: scan again in any case)
                        if ((kth << 16) > Tv) Tv = kth << 16;
                        Te = Tv;
                        tied = false;
                        if (etid == 0) {
                            es->nhits = 0;
                            es->fill_tie = 0;
                            es->Tv = Tv;
                        }
                        epi_bar(grp);
                        continue;
                    }
                    if (tied) break;  // (no better bound and what lies above T overflows the list: the exact selection)
                }
                if (!BF16 || tied) break;
                tied = true;
                if (etid == 0) {
                    es->nhits = 0;
                    es->fill_tie = 1;
                }
                Te = Tv + 0x10000u;  // (the next bf16 value up, whatever the sign: T holds the value's upper 16 bits)
                epi_bar(grp);
            }
            // (e) the 16-byte vectors of the hit chunks, re-read from global memory; elements >= T become keys.
            //     A thread issues its loads of a round before it uses any: under a saturated memory system one
            //     round trip costs microseconds.
            {
                // (with too many hits nothing is re-read: a segment that is mostly ties would send every element
                // through one shared counter)
                const bool hit_ovf = es->nhits > kVpHitCap;
                const int nhits = hit_ovf ? 0 : es->nhits;
                if (etid == 0 && hit_ovf) es->ovf = 1;
                constexpr int RU = 256 / ET;
                const int nvec = nhits * VEC_PER_LANE;
                bool full = false;
#pragma unroll 1
                for (int base = 0; base < nvec && !full; base += ET * RU) {
                    uint4 vv[RU];
                    uint32_t offs[RU];
#pragma unroll
                    for (int u = 0; u < RU; ++u) {
                        const int i = base + u * ET + etid;
                        vv[u] = make_uint4(T::NEG_INF_WORD, T::NEG_INF_WORD, T::NEG_INF_WORD, T::NEG_INF_WORD);
                        offs[u] = 0xFFFFFFFFu;
                        if (i < nvec) {
                            const uint32_t off = es->hits[i / VEC_PER_LANE] + (uint32_t)(i % VEC_PER_LANE) * 16u;
                            if (off < sg.body_bytes) {
                                offs[u] = off;
                                vv[u] = *(const uint4*)(sg.body + off);
                            }
                        }
                    }
#pragma unroll
                    for (int u = 0; u < RU; ++u) {
                        if (offs[u] == 0xFFFFFFFFu) continue;
                        // (three of a hit chunk's four vectors hold nothing that reaches T: one test for the vector)
                        if (vec_max_ord<BF16>(vv[u]) < Te) continue;
                        const uint32_t wv[4] = {vv[u].x, vv[u].y, vv[u].z, vv[u].w};
#pragma unroll
                        for (int j = 0; j < T::EPV; ++j) {
                            uint32_t xb;
                            if (BF16)
                                xb = (j & 1) ? (wv[j >> 1] & 0xFFFF0000u) : (wv[j >> 1] << 16);
                            else
                                xb = wv[j];
                            if (ord_from_bits(xb) >= Te && !full) {
                                const int pos = atomicAdd(&es->ncand, 1);
                                if (pos < kVpCandCap)
                                    es->cand[pos] = make_key(xb, (uint32_t)(sg.e_body0 + offs[u] / T::ESZ + j));
                                else
                                    full = true;  // (the count stays above the capacity: the exact selection takes over)
                            }
                        }
                    }
                }
            }
            epi_bar(grp);
            if (es->fill_ninf || es->fill_tie) {  // (uniform)
                if (ew == 0) {
                    // The first K elements equal to -inf (or, for bulk ties, to T) of the segment's body in id order (the
                    // few elements before and after the body are candidates already): a walk over the chunks in id
                    // order -- tile, streaming warp, lane -- that reads only chunks whose stored maximum reaches T (any
                    // chunk when the value looked for is -inf), 32 elements at a time.  Every chunk read for ties holds
                    // one at least unless a larger element put it on the list, so the walk is short wherever the ties
                    // are; the walk for -inf gives up after 256 chunks and the exact selection takes over.
                    const bool tie = es->fill_tie != 0;
                    const uint32_t T16 = Tv >> 16;
                    // (K chunks or more with an element above T: no tied element is wanted.  Otherwise fewer than 2 K
                    // visits find K tied elements or the end of the segment.)
                    int need = tie && es->nhits >= p.K ? 0 : p.K, visits = 0;
                    const int max_visits = tie ? 2 * p.K : 256;
                    bool gave_up = false;
#pragma unroll 1
                    for (int blk = 0; blk < sg.ntiles * NW && need > 0; ++blk) {
                        const int tile = blk / NW, w = blk % NW;
                        const uint32_t cm = ord_from_bits((uint32_t)cmx[(size_t)(w * 32 + lane) * p.max_tiles + tile] << 16) >> 16;
                        uint32_t todo = __ballot_sync(0xFFFFFFFFu, !tie || cm >= T16);
                        while (todo != 0u && need > 0) {  // (uniform)
                            if (++visits > max_visits) {
                                gave_up = true;
                                need = 0;
                                break;
                            }
                            const uint32_t off = (uint32_t)tile * TILE + (uint32_t)w * WBLK + (uint32_t)(__ffs(todo) - 1) * 64u +
                                                 (uint32_t)lane * T::ESZ;
                            todo &= todo - 1u;
                            uint32_t xb = 0u;
                            bool is = false;
                            if (lane < 64 / T::ESZ && off < sg.body_bytes) {
                                xb = __float_as_uint(load_elem_f32(sg.body + off, BF16));
                                is = tie ? (ord_from_bits(xb) >> 16) == T16 : xb == 0xFF800000u;  // (-0 and +0 are one value)
                            }
                            const uint32_t mk = __ballot_sync(0xFFFFFFFFu, is);
                            if (is && __popc(mk & ((1u << lane) - 1u)) < need) {
                                const int pos = atomicAdd(&es->ncand, 1);
                                if (pos < kVpCandCap) es->cand[pos] = make_key(xb, (uint32_t)sg.e_body0 + off / T::ESZ);
                            }
                            need -= __popc(mk);
                        }
                    }
                    if (gave_up && lane == 0) es->ovf = 1;
                }
                epi_bar(grp);
            }
            // (f) exact top-K of the candidates by rank counting (keys are distinct, so ranks are a permutation)
            // (ranking n candidates costs n^2 compares shared by 128 threads: beyond 256 -- rows whose large elements sit
            // side by side, such as sorted rows, fill every chunk that reaches T with candidates -- one warp finds the
            // K-th largest key by its bits instead)
            const bool overflow = es->ovf != 0 || es->ncand > kVpRankCap;
            const int ncand = es->ncand < kVpCandCap ? es->ncand : kVpCandCap;
            int nk = ncand < p.K ? ncand : p.K;
            if (!overflow) {
                // two neighbouring lanes per candidate, each over every other key, two running counts each
#pragma unroll 1
                for (int i0 = 0; i0 < ncand; i0 += ET / 2) {
                    const int i = i0 + (etid >> 1);
                    const uint64_t key = i < ncand ? es->cand[i] : ~0ull;
                    int r0 = 0, r1 = 0;
                    for (int j = etid & 1; j < ncand; j += 4) {
                        r0 += (es->cand[j] > key) ? 1 : 0;
                        r1 += (j + 2 < ncand && es->cand[j + 2] > key) ? 1 : 0;
                    }
                    int rank = r0 + r1;
                    rank += __shfl_xor_sync(0xFFFFFFFFu, rank, 1);
                    if (i < ncand && (etid & 1) == 0 && rank < p.K) es->outk[rank] = key;
                }
            } else if (es->ovf == 0 && es->ncand <= kVpCandCap) {  // (uniform; every candidate is in the buffer)
                epi_select_many(es, ncand, p.K, etid, grp);
            } else if (ew == 0) {
                // (T is a lower bound of the K-th largest element: the filter starts there, not at nothing -- a row sorted
                // in ascending order would otherwise send every element through the buffer; with the threshold moved up
                // from -inf, elements equal to -inf may be among the K best and nothing is ruled out)
                nk = warp_fallback_select<BF16>(es, p, sg, cmx, lane, es->fill_ninf ? 0ull : ((uint64_t)Tv << 32) - 1ull);
            }
            epi_bar(grp);
            // the double-buffered arrays of parity pb may be reused from here on
            if (ew == 0) {
                __syncwarp();
                if (lane == 0) mbar_arrive(done0 + 8 * pb);
            }
            // (g) finish the row, or leave a record for the CTA that arrives last
            // (a whole row is nobody else's: the divisions that find a shared row's CTAs are for partial rows only)
            const bool whole_row = sg.e0 == 0 && sg.e1 == p.V;
            double Cd = (double)c, Sd = (double)s;
            uint32_t Vm = vmo;
            bool finish = whole_row;
            int rec_internal = 0;  // a bounded wait ran out in one of the CTAs that left a record for this row
            if (!whole_row) {
                const long long x0 = (long long)sg.row * p.nq;
                const int c_first = cta_of(x0, p.Q, G), nseg = cta_of(x0 + p.nq - 1, p.Q, G) - c_first + 1;
                if (ew == 0) {
                    VpRecord* rec = p.records + (size_t)blockIdx.x * 2 + (sg.row == my_first_row ? 0 : 1);
                    if (lane < kMaxK) rec->keys[lane] = lane < nk ? es->outk[lane] : 0ull;
                    if (lane == 0) {
                        rec->c = c;
                        rec->s = s;
                        rec->vmax = __uint_as_float(vmo);
                        rec->nkeys = (uint32_t)nk | (sh->abort_flag ? 0x80000000u : 0u);
                    }
                    __syncwarp();
#ifdef GRAFT_TEST_LATE_RECORDS
                    // Test builds only: every CTA but the first waits some milliseconds here, so that a row of which CTA 0 has
                    // a piece is merged by another.
                    for (int i = 0; blockIdx.x != 0 && i < GRAFT_TEST_LATE_RECORDS; ++i) __nanosleep(1000000u);
#endif
                    if (lane == 0) es->arrived = atom_add_acq_rel(p.row_counter + sg.row, 1);  // (the lanes' stores included)
                }
                epi_bar(grp);
                if (es->arrived == nseg - 1) {  // (uniform)
                    finish = true;
                    // Merge the records of the row's CTAs, the group's threads together.  Every CTA after the first
                    // starts inside the row, so the row is its first and its record the first of its two; every record's
                    // keys are in descending order (empty ones, 0, last): a key's rank is its place in its own record plus
                    // the places that a binary search finds for it in the others.  (One warp that ranked all keys against
                    // each other took 10 us for nine records.)
                    const VpRecord* rec0 = p.records + (size_t)c_first * 2 + ((int)(cta_start(c_first, p.Q, G) / p.nq) == sg.row ? 0 : 1);
                    auto record = [&](int i) { return i == 0 ? rec0 : p.records + (size_t)(c_first + i) * 2; };
                    // the log-sum-exp pieces (warp 0), on their way while the keys are ranked
                    float rc = -INFINITY, rs = 0.f;
                    uint32_t rv = 0u;
                    int have_all = 0;
                    if (ew == 0 && lane < nseg) {
                        const VpRecord* r = record(lane);
                        rc = __ldcg(&r->c);
                        rs = __ldcg(&r->s);
                        rv = __float_as_uint(__ldcg(&r->vmax));
                        const uint32_t kn = __ldcg(&r->nkeys);
                        have_all = (int)(kn & 0x7FFFFFFFu);
                        rec_internal = (int)(kn >> 31);
                    }
                    constexpr int kRound = kVpCandCap / kMaxK - 1;  // records a round, behind the best of the rounds before
                    int have = 0;                                   // lists of kMaxK keys carried over: 0 or 1
#pragma unroll 1
                    for (int r0 = 0; r0 < nseg; r0 += kRound) {
                        const int cnt = nseg - r0 < kRound ? nseg - r0 : kRound, n = (have + cnt) * kMaxK;
#pragma unroll 1
                        for (int i = etid; i < cnt * kMaxK; i += ET)
                            es->cand[have * kMaxK + i] = __ldcg((const unsigned long long*)&record(r0 + i / kMaxK)->keys[i % kMaxK]);
                        if (etid < kMaxK) es->outk[etid] = 0ull;
                        epi_bar(grp);
#pragma unroll 1
                        for (int i = etid; i < n; i += ET) {
                            const uint64_t key = es->cand[i];
                            int rank = i % kMaxK;
#pragma unroll 1
                            for (int l = 0; l < n; l += kMaxK) {
                                if (l == i - i % kMaxK) continue;
                                int pos = 0;  // keys of list l above this one
#pragma unroll
                                for (int step = kMaxK / 2; step >= 1; step >>= 1)
                                    if (es->cand[l + pos + step - 1] > key) pos += step;
                                rank += pos + (es->cand[l + pos] > key ? 1 : 0);
                            }
                            if (key != 0ull && rank < p.K) es->outk[rank] = key;
                        }
                        epi_bar(grp);
                        if (r0 + kRound < nseg) {  // (uniform)
                            if (etid < kMaxK) es->cand[etid] = es->outk[etid];
                            have = 1;
                            epi_bar(grp);
                        }
                    }
                    if (ew == 0) {
                        // log-sum-exp pieces, folded in double
                        double Cm = (double)rc, S = 0.0;
                        uint32_t vm = rv;
#pragma unroll 1
                        for (int i = lane + 32; i < nseg; i += 32) {
                            const VpRecord* r = record(i);
                            const uint32_t kn = __ldcg(&r->nkeys), v2 = __float_as_uint(__ldcg(&r->vmax));
                            have_all += (int)(kn & 0x7FFFFFFFu);
                            rec_internal |= (int)(kn >> 31);
                            Cm = fmax(Cm, (double)__ldcg(&r->c));
                            vm = vm > v2 ? vm : v2;
                        }
#pragma unroll
                        for (int d = 16; d > 0; d >>= 1) Cm = fmax(Cm, __shfl_xor_sync(0xFFFFFFFFu, Cm, d));
                        vm = __reduce_max_sync(0xFFFFFFFFu, vm);
                        have_all = __reduce_add_sync(0xFFFFFFFFu, have_all);
#pragma unroll 1
                        for (int i = lane; i < nseg; i += 32) {
                            const float c2 = i < 32 ? rc : __ldcg(&record(i)->c), s2 = i < 32 ? rs : __ldcg(&record(i)->s);
                            if (c2 != -INFINITY)
                                S += (double)s2 * exp2((double)c2 - Cm);
                            else if (s2 != s2)
                                S += (double)s2;
                        }
#pragma unroll
                        for (int d = 16; d > 0; d >>= 1) S += __shfl_xor_sync(0xFFFFFFFFu, S, d);
                        rec_internal = __any_sync(0xFFFFFFFFu, rec_internal);
                        nk = have_all < p.K ? have_all : p.K;
                        Cd = Cm;
                        Sd = S;
                        Vm = vm;
                        if (lane == 0) p.row_counter[sg.row] = 0;
                    }
                }
            }
            if (ew != 0) continue;
            if (finish && p.partial_out != nullptr) {
                graft_vocab_partial* po = p.partial_out + sg.row;
                if (lane < kMaxK) po->keys[lane] = lane < nk ? es->outk[lane] : 0ull;
                if (lane == 0) {
                    po->c = Cd;
                    po->s = Sd;
                    po->vmax_ord = Vm;
                    po->nkeys = (uint32_t)nk | ((rec_internal || sh->abort_flag) ? 0x80000000u : 0u);
                }
            } else if (finish) {
                vp_finalize(Cd, Sd, Vm, nk, p.K, es->outk, lane, p.topk_id + (size_t)sg.row * p.K,
                            p.topk_lp + (size_t)sg.row * p.K, p.lse + sg.row, p.row_status + sg.row,
                            rec_internal || sh->abort_flag != 0);
            }
            __syncwarp();
        }
    }
    __syncthreads();
    if (tid == 0 && sh->abort_flag) atomicOr(p.errflag, 1);
}

// ---- vocabulary-parallel merge: two warps a row ------------------------------------------------------------------------
// A latency chain (1024 rows of 8 shards are 2.3 MB): every load is issued at once, then one warp merges the shards' descending
// lists two by two, a lane a key, in registers (what is not among the 32 best drops out on the way), and the other folds the
// pieces of the log-sum-exp.  One launch after the other: those rows 5.6 -> 4.4 us, 1600 rows of 2 shards 4.2 -> 3.3, 64 of 4 2.1
// as before (a CTA a row whose 256 threads looked for their keys' places in all lists by binary search: reads of shared memory
// whose places collide; one warp a row for both: 4.8, 4.4 and 2.8; one row a CTA 5.5, two 4.5).
constexpr int kMergeRows = 4;  // of a CTA; a warp more a row for its log-sum-exp
constexpr int kMergeMaxShards = 64;
struct MergeParams {
    const graft_vocab_partial* parts;  // [n_shards, rows]
    int n_shards, rows, K;
    int32_t v_offset[kMergeMaxShards];
    int32_t* topk_id;
    float* topk_lp;
    float* lse;
    int32_t* row_status;
};
// The 32 largest of two lists of 32, each a lane a key in descending order: the larger of every key and its opposite in the other
// list, in bitonic order, then five exchanges.
__device__ __forceinline__ uint64_t merge_lists(uint64_t a, uint64_t b, int lane) {
    const uint64_t o = __shfl_sync(0xFFFFFFFFu, b, 31 - lane);
    uint64_t m = a > o ? a : o;
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        const uint64_t x = __shfl_xor_sync(0xFFFFFFFFu, m, d);
        m = ((lane & d) == 0) == (x > m) ? x : m;
    }
    return m;
}
__global__ void __launch_bounds__(64 * kMergeRows) vocab_merge_kernel(const __grid_constant__ MergeParams p) {
    __shared__ double s_lse[kMergeRows];
    __shared__ int s_status[kMergeRows], s_nk[kMergeRows];
    const int lane = threadIdx.x & 31, warp = (int)(threadIdx.x >> 5), w = warp % kMergeRows, n = p.n_shards;
    const int row = (int)blockIdx.x * kMergeRows + w;
    const bool on = row < p.rows;
    pdl_launch_dependents();
    pdl_wait();
    const auto part = [&](int shard) { return p.parts + (size_t)shard * p.rows + row; };
    if (warp >= kMergeRows) {
        if (on) {  // the shards' pieces of the sum (two a lane: up to 64 shards)
            double c2[2] = {-INFINITY, -INFINITY}, s2[2] = {0.0, 0.0};
            uint32_t vm = 0u;
            int have = 0, internal = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = lane + 32 * h;
                if (i < n) {
                    const graft_vocab_partial* r = part(i);
                    c2[h] = r->c;
                    s2[h] = r->s;
                    const uint32_t v = r->vmax_ord, kn = r->nkeys;  // bit 31: a bounded wait ran out while the shard was scanned
                    vm = vm > v ? vm : v;
                    have += (int)(kn & 0x7FFFFFFFu);
                    internal |= (int)(kn >> 31);
                }
            }
            double Cm = fmax(c2[0], c2[1]), S = 0.0;
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) Cm = fmax(Cm, __shfl_xor_sync(0xFFFFFFFFu, Cm, d));
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (c2[h] != -INFINITY)
                    S += s2[h] * exp2(c2[h] - Cm);
                else if (s2[h] != s2[h])
                    S += s2[h];
            }
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) S += __shfl_xor_sync(0xFFFFFFFFu, S, d);
            vm = __reduce_max_sync(0xFFFFFFFFu, vm);
            have = __reduce_add_sync(0xFFFFFFFFu, have);
            internal = __any_sync(0xFFFFFFFFu, internal);
            if (lane == 0) {
                const int nk = have < p.K ? have : p.K;
                s_lse[w] = vp_lse(Cm, S, __uint_as_float(bits_from_ord(vm)));
                s_status[w] = (vp_bad_row(S, vm, nk, p.K) ? GRAFT_ST_BAD_LOGITS : 0) | (internal ? GRAFT_ST_INTERNAL : 0);
                s_nk[w] = nk;
            }
        }
        __syncthreads();
        return;
    }
    uint64_t best = 0ull;
    if (on) {
#pragma unroll 1
        for (int s0 = 0; s0 < n; s0 += 8) {
            const int left = n - s0;  // (uniform)
            uint64_t k[8];
            uint32_t nk[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                k[q] = q < left ? part(s0 + q)->keys[lane] : 0ull;
                nk[q] = q < left ? part(s0 + q)->nkeys & 0x7FFFFFFFu : 0u;
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {  // with global token ids; an empty place (0) stands behind every key
                if (lane >= (int)nk[q] || lane >= p.K) k[q] = 0ull;
                if (k[q] != 0ull) k[q] = make_key(bits_from_ord((uint32_t)(k[q] >> 32)), key_id(k[q]) + (uint32_t)p.v_offset[s0 + q]);
            }
            if (left > 1) k[0] = merge_lists(k[0], k[1], lane);
            if (left > 2) {
                k[2] = merge_lists(k[2], k[3], lane);
                if (left > 4) {
                    k[4] = merge_lists(k[4], k[5], lane);
                    k[6] = merge_lists(k[6], k[7], lane);
                    k[4] = merge_lists(k[4], k[6], lane);
                }
                k[0] = merge_lists(k[0], k[2], lane);
                if (left > 4) k[0] = merge_lists(k[0], k[4], lane);
            }
            best = s0 == 0 ? k[0] : merge_lists(best, k[0], lane);
        }
    }
    __syncthreads();
    if (on)
        vp_write_row(s_lse[w], s_status[w], s_nk[w], p.K, best, lane, p.topk_id + (size_t)row * p.K, p.topk_lp + (size_t)row * p.K,
                     p.lse + row, p.row_status + row);
}

}  // namespace

// ---- host side ----------------------------------------------------------------------------------
static void (*vp_kernel(bool bf16))(const VpParams) { return bf16 ? vocab_pass_kernel<true> : vocab_pass_kernel<false>; }
static size_t vp_smem_bytes(int stages, int n_cmax) {
    return (size_t)stages * TILE + (16 + 2 * BUFS) * sizeof(uint64_t) + sizeof(VpShared) + (size_t)BUFS * n_cmax * 2 + 16;
}

// ---- rows in shared memory (vocab_rows.cuh) ----
typedef void (*RowsKernel)(const RowsParams);
static RowsKernel rows_kernel(bool bf16, int cl, int nt) {
    if (cl == 4) return bf16 ? vocab_rows_kernel<true, 4, 256> : vocab_rows_kernel<false, 4, 256>;
    if (nt == 512) return bf16 ? vocab_rows_kernel<true, 1, 512> : vocab_rows_kernel<false, 1, 512>;
    return bf16 ? vocab_rows_kernel<true, 1, 256> : vocab_rows_kernel<false, 1, 256>;
}
static int rows_vecs(long long row_bytes, int cl) { return (int)((row_bytes / 16 + cl - 1) / cl) + 3; }
static size_t rows_smem_bytes(long long row_bytes, int cl, int nt) {
    const size_t sh = cl == 4 ? sizeof(RowsShared<4, 256>) : nt == 512 ? sizeof(RowsShared<1, 512>) : sizeof(RowsShared<1, 256>);
    const int vecs = rows_vecs(row_bytes, cl);
    return (size_t)vecs * 16 + sh + (size_t)((vecs + rows_tile_vecs(nt) - 1) / rows_tile_vecs(nt)) * nt * 2;
}
// CTAs of a size that an SM holds side by side (threads and registers allow four of 256 threads, two of 512)
static int rows_per_sm(long long row_bytes, int cl, int nt) {
    if (rows_vecs(row_bytes, cl) > kRowsMaxBytes / 16) return 0;  // (barriers for so many tiles)
    const int n = (int)(227 * 1024 / (rows_smem_bytes(row_bytes, cl, nt) + 1024)), most = nt == 512 ? 2 : 4;
    return n < most ? n : most;
}
// The cluster that holds a row, or 0: the streaming kernel.  Measured on 148 SMs, L = 16, K = 32, one launch after the other,
// streaming kernel -> rows in shared memory.
static void rows_plan(long long rows, long long row_bytes, int num_sms, bool round, VpPlan* pl) {
    pl->cluster = 0;
    const int per_sm = rows_per_sm(row_bytes, 4, 256);
    const bool alone = rows * 4 <= num_sms;  // four CTAs a row and an SM for each
    if (rows_per_sm(row_bytes, 1, 256) >= 2 && !(alone && row_bytes >= 80 * 1024)) {
        // a row a CTA where two or more share an SM, any number of rows.  bf16, V = 32,000 (three an SM): batch 1 8.3 -> 5.8 us,
        // batch 16 11.2 -> 9.5, batch 64 25.2 -> 20.7, batch 256 74.7 -> 62.5; V = 16,000 (four): batch 64 20.9 -> 13.5, batch
        // 256 63.5 -> 41.2; V = 50,021 (two): batch 64 34.3 -> 30.8, batch 256 114 -> 102.5.  With one CTA an SM nothing loads
        // while a row is finished: fp32, V = 32,000, batch 64 29.5 -> 45
        pl->cluster = 1;
        pl->threads = 256;
    } else if (!alone && rows <= num_sms && rows_per_sm(row_bytes, 1, 512) >= 1) {
        // longer rows, an SM for each (bf16, V = 75,000: batch 4 10.4 -> 7.2, batch 8 10.8 -> 7.8; with 256 threads 7.7, 8.3)
        pl->cluster = 1;
        pl->threads = 512;
    } else if (rows * 4 <= (long long)num_sms * per_sm * (round && per_sm == 1 ? 2 : 1)) {
        // rows too long for one CTA, or rows of 80 KB and more where four times as many SMs would stand idle, as far as all
        // pieces are resident at once.  V = 151,936: bf16 batch 1 12.7 -> 8.0, batch 4 13.4 -> 8.9, batch 8 (two turns) 15.1 ->
        // 18.5; fp32 batch 1 13.7 -> 7.2.  V = 50,021, bf16, batch 1 10.0 -> 5.8 (6.6 in one CTA), V = 32,000 the same in one
        // CTA as in four.  (512 threads: 9.0 at batch 1, V = 151,936; eight CTAs a row 7.9, but 10.0 at batch 4.)
        // Two turns in rounds on rows of which an SM holds one piece (over 390 KB), which the streaming kernel would cut and merge:
        // fp32, batch 3 and 4, rounds V = 101,000 45.2 -> 39.9 and 46.7 -> 41.0 us, V = 151,936 45.2 -> 41.6 and 47.5 -> 44.8 (with a
        // fixed budget 42.3 -> 37.7 and 44.3 -> 41.4); calls of their own 12.5 -> 12.2, 13.1 -> 12.9, 13.4 -> 14.2 and 14.3 -> 15.6.
        // With two pieces an SM two turns are slower in rounds too (V = 97,600, batch 5: 41.6 -> 45.2).
        pl->cluster = 4;
        pl->threads = 256;
    }
}
static cudaError_t rows_launch(bool bf16, const VpPlan& pl, long long row_bytes, const RowsParams& p, bool pdl, cudaStream_t st) {
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(p.rows * pl.cluster);
    lc.blockDim = dim3(pl.threads + 32);
    lc.dynamicSmemBytes = rows_smem_bytes(row_bytes, pl.cluster, pl.threads);
    lc.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = pl.cluster;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = pl.cluster > 1 ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&lc, rows_kernel(bf16, pl.cluster, pl.threads), p);
    return e != cudaSuccess ? e : cudaGetLastError();
}
static cudaError_t rows_configure(bool bf16) {
    cudaError_t e = cudaSuccess;
    const int variants[3][2] = {{1, 256}, {1, 512}, {4, 256}};
    for (int i = 0; i < 3 && e == cudaSuccess; ++i)
        e = allow_smem((const void*)rows_kernel(bf16, variants[i][0], variants[i][1]), 225 * 1024);
    return e;
}

VpPlan vp_make_plan(const graft_config& cfg, int num_sms, int batch, VpUse use) {
    const bool equal_shares = use == VpUse::neutral_round;
    VpPlan pl;
    const bool bf16 = cfg.logits_dtype == GRAFT_BF16;
    const long long esz = bf16 ? 2 : 4, rows = (long long)batch * cfg.L, row_bytes = (long long)cfg.V * esz;
    const long long nq = cfg.V / kVpQuantum > 0 ? cfg.V / kVpQuantum : 1;
    pl.cluster = 0;
    if (!equal_shares) rows_plan(rows, row_bytes, num_sms, use == VpUse::round, &pl);
    long long G, share_q, per = 0;  // CTAs (one per SM at most), a CTA's share at most, whole rows of a CTA at most
    // A row that no other CTA has a piece of needs no merge, which is what a small input waits for (a record and a merge
    // take 5 to 6 us): whole rows wherever the CTAs' shares come out even enough.  Measured
    // on 148 SMs, one launch after the other, bf16, L = 16.
    if (equal_shares) {
        // Rounds without edge scores.  Their path scores are sums of log-probabilities alone, and of logits with few digits
        // hundreds of such sums are equal but for the rounding of the rows' log-sum-exp: its last bit, which hangs on how a
        // row's sum is cut into pieces, decides which prefix stands first.  These rounds keep the partition that all rounds
        // once had (equal shares of at least 64 KB of the whole stream), so that a batch gives the trees that it always gave;
        // whole rows would make a round 7 % shorter (batch 37, L = 11, V = 50,021).  It is no more than that: in a batch of
        // another size, in another place of it or on another number of SMs a row is cut elsewhere, and such prefixes may
        // come out in another order.
        G = nq * rows / (64 * 1024 / (kVpQuantum * esz));
        if (G > num_sms) G = num_sms;
        if (G < 1) G = 1;
        pl.whole = 0;
        share_q = (nq * rows + G - 1) / G;
    } else if (rows < num_sms) {
        // n pieces of each row of 76 KB or more, n = 1 unless the stream gets shorter by more than the merge costs (190 KB), as
        // rows of 380 KB do (measured on bf16 rows of 300 KB: 16 rows n = 1 18.5 us, n = 2 18.6, n = 4 17.1, n = 9 20.9; 64 rows
        // n = 1 18.9, n = 2 19.7)
        long long n = row_bytes / (76 * 1024);
        if (n > num_sms / rows) n = num_sms / rows;
        if (n > nq) n = nq;
        if (n < 1 || row_bytes - row_bytes / n < 190 * 1024) n = 1;
        G = rows * n;
        pl.whole = n == 1;
        share_q = (nq + n - 1) / n;
        per = 1;
    } else {
        // whole rows, unless that gives some CTA over 90 KB more than the average (V = 151,936: batch 16 28.5 -> 27.0 us with
        // whole rows, batch 24 the same, batch 20 30.3 -> 33.3, batch 256 204 -> 207); rows up to 132 KB always (rows
        // of 100 KB: batch 16 23.7 -> 19.9 us, batch 28 27.2 -> 26.9)
        per = (rows + num_sms - 1) / num_sms;
        pl.whole = row_bytes <= 132 * 1024 || per * row_bytes - rows * row_bytes / num_sms <= 90 * 1024;
        G = pl.whole ? (rows + per - 1) / per : num_sms;
        share_q = pl.whole ? per * nq : (nq * rows + G - 1) / G;
    }
    if (!equal_shares && pl.whole == 0 && G > nq * rows) G = nq * rows;
    pl.grid = (int)G;
    long long seg_elems = share_q * kVpQuantum + kVpQuantum;  // a row's last quantum also takes the remainder
    if (pl.whole || seg_elems > cfg.V) seg_elems = cfg.V;
    pl.max_seg_tiles = (int)((seg_elems * esz + TILE - 1) / TILE) + 1;
    const size_t budget = 224 * 1024;  // one CTA per SM
    int stages = 6;
    while (stages > 2 && vp_smem_bytes(stages, pl.max_seg_tiles * NT) > budget) --stages;
    pl.stages = stages;
    pl.smem_bytes = vp_smem_bytes(stages, pl.max_seg_tiles * NT);
    return pl;
}

cudaError_t vp_launch(graft_ctx* ctx, int batch, const void* d_logits, int32_t* d_topk_id, float* d_topk_lp,
                      float* d_lse, int32_t* d_row_status, const void* d_hidden, double* d_cos,
                      graft_vocab_partial* d_partial, VpUse use, cudaStream_t st) {
    const graft_config& cfg = ctx->cfg;
    const bool bf16 = cfg.logits_dtype == GRAFT_BF16;
    VpPlan pl = vp_make_plan(cfg, ctx->num_sms, batch, use);
    if (pl.cluster > 0) {
        RowsParams r;
        r.logits = (const char*)d_logits;
        r.rows = batch * cfg.L;
        r.V = cfg.V;
        r.K = cfg.K;
        r.topk_id = d_topk_id;
        r.topk_lp = d_topk_lp;
        r.lse = d_lse;
        r.row_status = d_row_status;
        r.errflag = ctx->w_errflag;
        r.partial_out = d_partial;
        r.hidden = d_hidden;
        r.hidden_bf16 = cfg.hidden_dtype == GRAFT_BF16 ? 1 : 0;
        r.hidden_dim = cfg.hidden_dim;
        r.L = cfg.L;
        r.cos_out = (d_hidden != nullptr && cfg.L > 1) ? d_cos : nullptr;
        r.vecs = rows_vecs((long long)cfg.V * (bf16 ? 2 : 4), pl.cluster);
        ctx->launches += 1;
        return rows_launch(bf16, pl, (long long)cfg.V * (bf16 ? 2 : 4), r, true, st);
    }
    VpParams p;
    p.logits = (const char*)d_logits;
    p.rows = batch * cfg.L;
    p.V = cfg.V;
    p.K = cfg.K;
    p.nq = pl.whole || cfg.V < kVpQuantum ? 1 : cfg.V / kVpQuantum;
    p.Q = p.nq * p.rows;
    p.stages = pl.stages;
    p.n_cmax = pl.max_seg_tiles * NT;
    p.max_tiles = pl.max_seg_tiles;
    p.records = ctx->vp_records;
    p.row_counter = ctx->vp_row_counter;
    p.topk_id = d_topk_id;
    p.topk_lp = d_topk_lp;
    p.lse = d_lse;
    p.row_status = d_row_status;
    p.errflag = ctx->w_errflag;
    p.partial_out = d_partial;
    p.hidden = d_hidden;
    p.hidden_bf16 = cfg.hidden_dtype == GRAFT_BF16 ? 1 : 0;
    p.hidden_dim = cfg.hidden_dim;
    p.L = cfg.L;
    p.cos_out = (d_hidden != nullptr && cfg.L > 1) ? d_cos : nullptr;
    p.use_hint = 1;
    const cudaError_t e = launch_pdl(vp_kernel(bf16), dim3(pl.grid), dim3(kVpThreads), pl.smem_bytes, st, p);
    ctx->launches += 1;
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t vp_merge_launch(graft_ctx* ctx, int batch, int n_shards, const graft_vocab_partial* d_parts,
                            const int32_t* h_v_offset, int32_t* d_topk_id, float* d_topk_lp, float* d_lse,
                            int32_t* d_row_status, cudaStream_t st) {
    MergeParams p;
    p.parts = d_parts;
    p.n_shards = n_shards;
    p.rows = batch * ctx->cfg.L;
    p.K = ctx->cfg.K;
    for (int i = 0; i < kMergeMaxShards; ++i) p.v_offset[i] = i < n_shards ? h_v_offset[i] : 0;
    p.topk_id = d_topk_id;
    p.topk_lp = d_topk_lp;
    p.lse = d_lse;
    p.row_status = d_row_status;
    const cudaError_t e = launch_pdl(vocab_merge_kernel, dim3((p.rows + kMergeRows - 1) / kMergeRows), dim3(64 * kMergeRows), 0, st, p);
    ctx->launches += 1;
    return e != cudaSuccess ? e : cudaGetLastError();
}
int vp_merge_max_shards() { return kMergeMaxShards; }

cudaError_t vp_configure(const graft_config& cfg, int num_sms, size_t* max_smem) {
    // the largest dynamic shared-memory request any batch can produce (segment = a whole row)
    VpPlan pl = vp_make_plan(cfg, num_sms, cfg.max_batch > 4096 ? cfg.max_batch : 4096, VpUse::call);
    *max_smem = pl.smem_bytes;
    if (pl.smem_bytes > 225 * 1024) return cudaErrorInvalidValue;
    cudaError_t e = cudaSuccess;
    e = rows_configure(cfg.logits_dtype == GRAFT_BF16);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(vp_kernel(cfg.logits_dtype == GRAFT_BF16), cudaFuncAttributeMaxDynamicSharedMemorySize, 225 * 1024);
    return e;
}

}  // namespace graft

// ---- allocation-free variant of the vocab pass ------------------------------------------------------------
// Some callers cannot let this library allocate: a serving process that handed all device memory to its own
// pool at start-up (a cudaMalloc there fails, or stalls every stream while the driver synchronises), or code
// that must stay off the driver's allocation lock on its latency path.  For them the scratch of the vocab
// pass -- the per-CTA records of rows shared between CTAs, the per-row arrival counters and the error word --
// lives in the file-scope device array below instead of a context's cudaMalloc'ed workspace.  Every GPU that
// loads this library holds the array (about 0.4 MB) until the process exits.
namespace graft {
namespace {

constexpr int kStaticMaxGrid = 512;     // CTAs (one per SM is launched): room for any device
constexpr int kStaticMaxRows = 16384;   // batch * L

struct VpStaticScratch {
    VpRecord records[kStaticMaxGrid * 2];
    int row_counter[kStaticMaxRows];
    int errflag[64];
};

static __device__ __align__(256) unsigned char g_vp_static_scratch[sizeof(VpStaticScratch)];

struct VpStaticDevice {
    bool ready = false;
    VpStaticScratch* scratch = nullptr;  // device address of g_vp_static_scratch on this device
    int num_sms = 0;
};
VpStaticDevice g_vp_static_dev[64];
std::mutex g_vp_static_mutex;

}  // namespace
}  // namespace graft

extern "C" graft_status graft_vocab_pass_static(int32_t batch, int32_t L, int32_t V, int32_t K,
                                                graft_dtype logits_dtype, const void* d_logits, int32_t* d_topk_id,
                                                float* d_topk_lp, float* d_lse, int32_t* d_row_status, void* stream) {
    using namespace graft;
    if (!d_logits || !d_topk_id || !d_topk_lp || !d_lse || !d_row_status) return GRAFT_ERR_INVALID_ARG;
    if (logits_dtype != GRAFT_F32 && logits_dtype != GRAFT_BF16) return GRAFT_ERR_INVALID_ARG;
    if (batch < 1 || L < 1 || V < 1 || K < 1) return GRAFT_ERR_INVALID_ARG;
    if ((uintptr_t)d_logits % (logits_dtype == GRAFT_BF16 ? 2 : 4)) return GRAFT_ERR_INVALID_ARG;
    if (K > kMaxK || K > V || L > kMaxL || (long long)V > 2147483647LL - 64) return GRAFT_ERR_UNSUPPORTED;
    if ((long long)batch * L > kStaticMaxRows) return GRAFT_ERR_UNSUPPORTED;  // beyond the static scratch
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return GRAFT_ERR_CUDA;
    }
    graft_config cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.V = V;
    cfg.L = L;
    cfg.K = K;
    cfg.max_batch = batch;
    cfg.logits_dtype = logits_dtype;
    VpStaticDevice* sd = &g_vp_static_dev[dev];
    {
        // set-up, once per device, with that device current: the array's name is only a host-side stand-in
        // here, so its device address has to be asked for
        std::lock_guard<std::mutex> lock(g_vp_static_mutex);
        if (!sd->ready) {
            void* ptr = nullptr;
            if (cudaGetSymbolAddress(&ptr, g_vp_static_scratch) != cudaSuccess || !ptr) {
                cudaGetLastError();
                return GRAFT_ERR_CUDA;
            }
            int sms = 0;
            if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
                cudaGetLastError();
                return GRAFT_ERR_CUDA;
            }
            for (int i = 0; i < 2; ++i)
                if (cudaFuncSetAttribute(vp_kernel(i != 0), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         225 * 1024) != cudaSuccess) {
                    cudaGetLastError();
                    return GRAFT_ERR_CUDA;
                }
            if (rows_configure(true) != cudaSuccess || rows_configure(false) != cudaSuccess) {
                cudaGetLastError();
                return GRAFT_ERR_CUDA;
            }
            sd->scratch = (VpStaticScratch*)ptr;
            sd->num_sms = sms;
            sd->ready = true;
        }
    }
    const VpPlan pl = vp_make_plan(cfg, sd->num_sms, batch, VpUse::call);
    if (pl.cluster > 0) {
        cudaStream_t st = (cudaStream_t)stream;
        if (cudaMemsetAsync(sd->scratch->errflag, 0, sizeof(sd->scratch->errflag), st) != cudaSuccess) {
            cudaGetLastError();
            return GRAFT_ERR_CUDA;
        }
        RowsParams r;
        memset(&r, 0, sizeof r);
        r.logits = (const char*)d_logits;
        r.rows = batch * L;
        r.V = V;
        r.K = K;
        r.topk_id = d_topk_id;
        r.topk_lp = d_topk_lp;
        r.lse = d_lse;
        r.row_status = d_row_status;
        r.errflag = sd->scratch->errflag;
        r.L = L;
        const long long row_bytes = (long long)V * (logits_dtype == GRAFT_BF16 ? 2 : 4);
        r.vecs = rows_vecs(row_bytes, pl.cluster);
        return rows_launch(logits_dtype == GRAFT_BF16, pl, row_bytes, r, false, st) == cudaSuccess ? GRAFT_OK : GRAFT_ERR_CUDA;
    }
    if (pl.grid > kStaticMaxGrid || pl.smem_bytes > 225 * 1024) return GRAFT_ERR_UNSUPPORTED;
    cudaStream_t st = (cudaStream_t)stream;
    // the array keeps whatever the previous call left: the arrival counters and the error word must start at 0
    if (cudaMemsetAsync(sd->scratch->row_counter, 0, sizeof(int) * (size_t)batch * L, st) != cudaSuccess ||
        cudaMemsetAsync(sd->scratch->errflag, 0, sizeof(sd->scratch->errflag), st) != cudaSuccess) {
        cudaGetLastError();
        return GRAFT_ERR_CUDA;
    }
    VpParams p;
    p.logits = (const char*)d_logits;
    p.rows = batch * L;
    p.V = V;
    p.K = K;
    p.nq = pl.whole || V < kVpQuantum ? 1 : V / kVpQuantum;
    p.Q = p.nq * p.rows;
    p.stages = pl.stages;
    p.n_cmax = pl.max_seg_tiles * NT;
    p.max_tiles = pl.max_seg_tiles;
    p.records = sd->scratch->records;
    p.row_counter = sd->scratch->row_counter;
    p.topk_id = d_topk_id;
    p.topk_lp = d_topk_lp;
    p.lse = d_lse;
    p.row_status = d_row_status;
    p.errflag = sd->scratch->errflag;
    p.partial_out = nullptr;
    p.hidden = nullptr;
    p.hidden_bf16 = 0;
    p.hidden_dim = 0;
    p.L = L;
    p.cos_out = nullptr;
    p.use_hint = 1;
    vp_kernel(logits_dtype == GRAFT_BF16)<<<pl.grid, kVpThreads, pl.smem_bytes, st>>>(p);
    return cudaGetLastError() == cudaSuccess ? GRAFT_OK : GRAFT_ERR_CUDA;
}

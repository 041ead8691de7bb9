// Device code of Cussen's compression-reconstruction PC-MM shared by the
// single-instance kernels (k_cussen.cu) and the persistent batched kernel
// (k_batched.cu): workspace layout, the plan of one strip, the table build of
// one warp item and the gather of one warp item.
#pragma once
#include <cuda_runtime.h>

#include <math.h>

#include "common.cuh"

namespace pcmm {
namespace cussen {

constexpr int NLEV = PCMM_N_ITER;   // compression iterations N

// Which field operations the gather's mixed addition and the table build's
// chain additions inline (build-time switches, see jacz_madd_t).  Measured
// on GB300 (w = 4, 1024 x 1024 x 256): gather 25.3 ms all out of line, 25.0 with
// the squarings and a b - c d inlined (3), 23.9 all inlined (31) at four blocks
// per SM, 24.6 at three and 25.1 at five: a call moves its operands on the pipe
// that multiplies.
#ifndef PCMM_GATHER_INLINE
#define PCMM_GATHER_INLINE 31
#endif
#ifndef PCMM_TABLE_INLINE
#define PCMM_TABLE_INLINE 0
#endif
// The same for the digit build's chains: table of 1024 x 1024 x 256 at w = 8 (without
// signed pairs) 12.6, 12.7, 12.6 and 12.3 ms at 0, 1, 2 and 3.
#ifndef PCMM_DIGIT_INLINE
#define PCMM_DIGIT_INLINE 3
#endif
// And for the build with signed pairs: 10.8, 10.7, 10.5 and 10.7 ms.
#ifndef PCMM_SIGNED_INLINE
#define PCMM_SIGNED_INLINE 2
#endif
// Of two columns' digits (w = 4): 5.4, -, 5.3 and 5.4 ms.
#ifndef PCMM_CROSS_INLINE
#define PCMM_CROSS_INLINE 2
#endif
constexpr uint16_t NO_RANK = 0xFFFFu;
constexpr int PLAN_THREADS = 256;

struct Layout {
    int m, n, l, w, k;
    int nstrips, n1max, l2max, emax, lp, njb, ptr_stride;
    size_t off_rank, off_nent, off_codes, off_len, off_vN, off_ptr, off_rank1, plan_bytes;
    size_t item_u4, items_per_strip, table_points_per_strip, per_strip_bytes;
};

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Largest d with d (d + 1) / 2 <= 2^w - 1: the distinct positive differences
// of distinct values below 2^w sum to at most 2^w - 1, so every level after
// the first holds at most d entries.
inline int level2_bound(int w) {
    int lim = (1 << w) - 1, d = 0;
    while ((d + 1) * (d + 2) / 2 <= lim) d++;
    return d < 1 ? 1 : d;
}

// Workspace layout of one PC-MM (host and device agree on it).  Entries of A
// have up to PCMM_MAX_W16 bits; a strip code has w k <= PCMM_MAX_WK bits.
// Per column the plan holds the level lengths, the level-N values (uint16,
// l2max per column) and the tracking pointers of levels 1..N-1 (uint16:
// n1max for level 1, then l2max per further level).
inline bool make_layout(Layout& L, int m, int n, int l, int w, int k) {
    if (m < 1 || n < 1 || l < 1 || w < 1 || w > PCMM_MAX_W16 || k < 1 || w * k > PCMM_MAX_WK) return false;
    L.m = m; L.n = n; L.l = l; L.w = w; L.k = k;
    L.nstrips = (n + k - 1) / k;
    L.n1max = (1 << w) - 1 < m ? (1 << w) - 1 : m;
    L.l2max = level2_bound(w) < L.n1max ? level2_bound(w) : L.n1max;
    L.emax = (1 << (w * k)) - 1 < m ? (1 << (w * k)) - 1 : m;
    L.ptr_stride = L.n1max + (NLEV > 2 ? NLEV - 2 : 0) * L.l2max;
    L.njb = (l + 31) / 32;
    L.lp = L.njb * 32;
    size_t off = 256;  // status word and padding
    L.off_rank = off;  off = align256(off + (size_t)L.nstrips * m * 2);
    L.off_nent = off;  off = align256(off + (size_t)L.nstrips * 4);
    L.off_codes = off; off = align256(off + (size_t)L.nstrips * L.emax * 2);
    L.off_len = off;   off = align256(off + (size_t)n * NLEV * 2);
    L.off_vN = off;    off = align256(off + (size_t)n * L.l2max * 2);
    L.off_ptr = off;   off = align256(off + (size_t)n * L.ptr_stride * 2);
    L.off_rank1 = off; off = align256(off + (k > 1 ? (size_t)n * 256 : 0));
    L.plan_bytes = off;
    // Per warp item (lane-planar): Jacobian column table and level ping-pong;
    // affine level-2 entries, affine column tables and tuple partial sums
    // (k > 1); prefix products for the normalisations.
    const size_t jac_ents = (size_t)L.n1max + 2 * (size_t)L.l2max;
    const size_t aff_ents = (size_t)L.l2max + (k > 1 ? (size_t)k * L.n1max + (size_t)L.emax : 0);
    const size_t pref_ents = (size_t)(L.emax > L.n1max ? L.emax : L.n1max);
    L.item_u4 = jac_ents * 6 * 32 + aff_ents * 4 * 32 + pref_ents * 2 * 32;
    L.items_per_strip = 2 * (size_t)L.njb;
    L.table_points_per_strip = (size_t)L.emax * 2 * L.lp;
    L.per_strip_bytes = L.items_per_strip * L.item_u4 * 16 + align256(L.table_points_per_strip * 64);
    return true;
}

struct PlanPtrs {
    uint32_t* status;
    uint16_t* rank;
    int32_t* nent;
    uint16_t* codes;
    uint16_t* col_len;
    uint16_t* col_vN;      // [col][l2max]
    uint16_t* col_ptr;     // [col][ptr_stride]
    uint8_t* col_rank1;    // [col][256] (k > 1, so w <= 8)
    int n1max, l2max, ptr_stride, emax;
};

inline PlanPtrs plan_ptrs(const Layout& L, void* ws) {
    uint8_t* b = (uint8_t*)ws;
    PlanPtrs P;
    P.status = (uint32_t*)b;
    P.rank = (uint16_t*)(b + L.off_rank);
    P.nent = (int32_t*)(b + L.off_nent);
    P.codes = (uint16_t*)(b + L.off_codes);
    P.col_len = (uint16_t*)(b + L.off_len);
    P.col_vN = (uint16_t*)(b + L.off_vN);
    P.col_ptr = (uint16_t*)(b + L.off_ptr);
    P.col_rank1 = b + L.off_rank1;
    P.n1max = L.n1max;
    P.l2max = L.l2max;
    P.ptr_stride = L.ptr_stride;
    P.emax = L.emax;
    return P;
}

// Tracking pointers of level lev (1 .. NLEV-1) of column col: entry e of
// level lev sits at position ptr[e] of level lev + 1.
__device__ __forceinline__ uint16_t* col_level_ptr(const PlanPtrs& P, int col, int lev) {
    return P.col_ptr + (size_t)col * P.ptr_stride + (lev == 1 ? 0 : P.n1max + (size_t)(lev - 2) * P.l2max);
}

__device__ __forceinline__ int warp_excl_scan(int v, int& total) {
    const unsigned lane = threadIdx.x & 31u;
    int incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        int o = __shfl_up_sync(0xffffffffu, incl, d);
        if ((int)lane >= d) incl += o;
    }
    total = __shfl_sync(0xffffffffu, incl, 31);
    return incl - v;
}

// Sorted list of the values marked in a 256-bit presence map; also a
// value -> position map.  Each lane owns 8 consecutive values.
__device__ __forceinline__ int extract_sorted(const uint32_t* bm, uint16_t* out, uint8_t* pos_of) {
    const unsigned lane = threadIdx.x & 31u;
    const uint32_t bits8 = (bm[lane >> 2] >> ((lane & 3u) * 8u)) & 0xffu;
    int total;
    int pos = warp_excl_scan(__popc(bits8), total);
    for (int b = 0; b < 8; b++) {
        if ((bits8 >> b) & 1u) {
            const int v = (int)lane * 8 + b;
            out[pos] = (uint16_t)v;
            pos_of[v] = (uint8_t)pos;
            pos++;
        }
    }
    __syncwarp();
    return total;
}

// ---- block-level helpers of the plan (blockDim.x == PLAN_THREADS) ----

// Exclusive prefix sum of one value per thread over the block; every thread
// receives the total.  All threads must call.
__device__ __forceinline__ int block_excl_scan(int v, int& total) {
    __shared__ int wsum[PLAN_THREADS / 32];
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    int wt;
    const int x = warp_excl_scan(v, wt);
    __syncthreads();
    if (lane == 0) wsum[warp] = wt;
    __syncthreads();
    int base = 0, tot = 0;
    for (int q = 0; q < PLAN_THREADS / 32; q++) {
        const int t = wsum[q];
        if (q < (int)warp) base += t;
        tot += t;
    }
    total = tot;
    return base + x;
}

// Exclusive prefix maximum (identity -1) of one value per thread.
__device__ __forceinline__ int block_excl_max(int v) {
    __shared__ int wmax[PLAN_THREADS / 32];
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, incl, d);
        if ((int)lane >= d) incl = o > incl ? o : incl;
    }
    int ex = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 0) ex = -1;
    __syncthreads();
    if (lane == 31) wmax[warp] = incl;
    __syncthreads();
    for (int q = 0; q < (int)warp; q++) ex = wmax[q] > ex ? wmax[q] : ex;
    return ex;
}

// Words [w0, w0 + wpt) of an nw-word presence map belong to this thread.
__device__ __forceinline__ int map_words_per_thread(int nw) { return (nw + PLAN_THREADS - 1) / PLAN_THREADS; }

// pf[x] = number of set bits in words 0..x-1 of bm; returns the total.
__device__ __forceinline__ int map_prefix(const uint32_t* bm, uint32_t* pf, int nw) {
    const int wpt = map_words_per_thread(nw);
    const int w0 = (int)threadIdx.x * wpt;
    int cnt = 0;
    for (int q = 0; q < wpt; q++)
        if (w0 + q < nw) cnt += __popc(bm[w0 + q]);
    int total;
    int base = block_excl_scan(cnt, total);
    for (int q = 0; q < wpt; q++)
        if (w0 + q < nw) {
            pf[w0 + q] = (uint32_t)base;
            base += __popc(bm[w0 + q]);
        }
    __syncthreads();
    return total;
}

// Position of the present value v in the sorted list of present values.
__device__ __forceinline__ int map_rank(const uint32_t* bm, const uint32_t* pf, uint32_t v) {
    return (int)(pf[v >> 5] + __popc(bm[v >> 5] & ((1u << (v & 31u)) - 1u)));
}

__device__ __forceinline__ void map_clear(uint32_t* bm, int nw) {
    for (int x = threadIdx.x; x < nw; x += PLAN_THREADS) bm[x] = 0u;
}

// Levels 2..N of one column whose values have up to 16 bits (w > 8, hence
// k = 1), computed by the whole block.  Level 1 (the sorted distinct
// non-zero values) is given as the presence map bm1 of nw words with its
// prefix counts pf1.  Level q + 1 is the sorted distinct set of the
// differences of consecutive level-q values (the first minus zero); the
// tracking pointer of a level-q entry is the position of its difference in
// level q + 1.  bm/pf: nw-word work maps; lvA/lvB: lists of l2max entries.
__device__ __forceinline__ void plan_column_wide(const uint32_t* bm1, const uint32_t* pf1, int nw, int len1,
                                                 int col, const PlanPtrs& P, uint32_t* bm, uint32_t* pf,
                                                 uint16_t* lvA, uint16_t* lvB) {
    const int wpt = map_words_per_thread(nw);
    const int w0 = (int)threadIdx.x * wpt;
    if (threadIdx.x == 0) P.col_len[(size_t)col * NLEV] = (uint16_t)len1;
    // Level 1 -> 2.  The predecessor of the first value in this thread's
    // words is the largest value in the words before them.
    int last = -1;
    for (int q = 0; q < wpt; q++)
        if (w0 + q < nw && bm1[w0 + q]) last = (w0 + q) * 32 + 31 - __clz(bm1[w0 + q]);
    const int prev0 = block_excl_max(last);
    map_clear(bm, nw);
    __syncthreads();
    for (int pass = 0; pass < 2; pass++) {
        int prev = prev0 < 0 ? 0 : prev0;
        uint16_t* ptr1 = col_level_ptr(P, col, 1);
        for (int q = 0; q < wpt; q++) {
            if (w0 + q >= nw) break;
            uint32_t x = bm1[w0 + q];
            while (x) {
                const uint32_t v = (uint32_t)(w0 + q) * 32u + (uint32_t)(__ffs(x) - 1);
                const uint32_t d = v - (uint32_t)prev;
                if (pass == 0) atomicOr(&bm[d >> 5], 1u << (d & 31u));
                else ptr1[map_rank(bm1, pf1, v)] = (uint16_t)map_rank(bm, pf, d);
                prev = (int)v;
                x &= x - 1u;
            }
        }
        __syncthreads();
        if (pass == 0) map_prefix(bm, pf, nw);
    }
    uint16_t* cur = lvA;
    uint16_t* nxt = lvB;
    int len = 0;
    for (int lev = 1; lev < NLEV; lev++) {
        if (lev > 1) {
            // Differences of the level-lev list into the work map.
            map_clear(bm, nw);
            __syncthreads();
            for (int e = threadIdx.x; e < len; e += PLAN_THREADS) {
                const uint32_t d = (uint32_t)cur[e] - (e ? (uint32_t)cur[e - 1] : 0u);
                atomicOr(&bm[d >> 5], 1u << (d & 31u));
            }
            __syncthreads();
            map_prefix(bm, pf, nw);
            uint16_t* ptr = col_level_ptr(P, col, lev);
            for (int e = threadIdx.x; e < len; e += PLAN_THREADS) {
                const uint32_t d = (uint32_t)cur[e] - (e ? (uint32_t)cur[e - 1] : 0u);
                ptr[e] = (uint16_t)map_rank(bm, pf, d);
            }
        }
        // Level lev + 1: the sorted present values of the work map.
        int nlen;
        {
            int cnt = 0;
            for (int q = 0; q < wpt; q++)
                if (w0 + q < nw) cnt += __popc(bm[w0 + q]);
            block_excl_scan(cnt, nlen);
        }
        for (int q = 0; q < wpt; q++) {
            if (w0 + q >= nw) break;
            uint32_t x = bm[w0 + q];
            while (x) {
                const uint32_t d = (uint32_t)(w0 + q) * 32u + (uint32_t)(__ffs(x) - 1);
                const int r = map_rank(bm, pf, d);
                if (r < P.l2max) nxt[r] = (uint16_t)d;
                x &= x - 1u;
            }
        }
        if (threadIdx.x == 0) P.col_len[(size_t)col * NLEV + lev] = (uint16_t)nlen;
        __syncthreads();
        uint16_t* tmp = cur; cur = nxt; nxt = tmp;
        len = nlen < P.l2max ? nlen : P.l2max;
    }
    for (int e = threadIdx.x; e < len; e += PLAN_THREADS) P.col_vN[(size_t)col * P.l2max + e] = cur[e];
    __syncthreads();
}

// Block-level plan of strip s (all PLAN_THREADS threads of the block call):
// the presence map of the strip's codes (a code is the k-tuple of a row's
// entries, w bits each), each row's rank among the distinct non-zero codes,
// the list of distinct codes (k > 1) and the compression levels of every
// column of the strip.  TA is the element type of A (uint8 or uint16).
template <class TA>
__device__ __forceinline__ void plan_strip(const TA* __restrict__ A, int m, int n, int w, int k,
                                           const PlanPtrs& P, int s) {
    constexpr int MAP_WORDS = 1 << (PCMM_MAX_WK - 5);
    __shared__ uint32_t spres[MAP_WORDS];
    __shared__ uint32_t spref[MAP_WORDS];
    __shared__ uint32_t work[2 * MAP_WORDS];
    __shared__ uint16_t lv[2][512];
    const int c0 = s * k;
    const int kw = (c0 + k <= n) ? k : n - c0;
    const uint32_t amask = (1u << w) - 1u;
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const int emax = P.emax;

    // ---- strip codes, distinct codes and per-row ranks ----
    const int cbits = w * k;
    const int nwc = cbits > 5 ? 1 << (cbits - 5) : 1;
    map_clear(spres, nwc);
    __syncthreads();
    bool bad = false;
    for (int i = threadIdx.x; i < m; i += PLAN_THREADS) {
        uint32_t code = 0;
        for (int t = 0; t < kw; t++) {
            const uint32_t v = (uint32_t)A[(size_t)i * n + c0 + t];
            bad |= v > amask;
            code |= (v & amask) << (w * t);
        }
        if (code) atomicOr(&spres[code >> 5], 1u << (code & 31u));
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(P.status, DEV_ERR_A_RANGE);
    const int total = map_prefix(spres, spref, nwc);
    if (threadIdx.x == 0) P.nent[s] = total;
    for (int i = threadIdx.x; i < m; i += PLAN_THREADS) {
        uint32_t code = 0;
        for (int t = 0; t < kw; t++) code |= ((uint32_t)A[(size_t)i * n + c0 + t] & amask) << (w * t);
        P.rank[(size_t)s * m + i] = code ? (uint16_t)map_rank(spres, spref, code) : NO_RANK;
    }
    if (k > 1) {
        for (int wd = threadIdx.x; wd < nwc; wd += PLAN_THREADS) {
            uint32_t bits = spres[wd];
            uint32_t r = spref[wd];
            while (bits) {
                const int b = __ffs(bits) - 1;
                if ((int)r < emax) P.codes[(size_t)s * emax + r] = (uint16_t)(wd * 32 + b);
                r++;
                bits &= bits - 1u;
            }
        }
    }

    if (w > 8) {
        // ---- wide values: k = 1, the strip map is the column's level 1 ----
        plan_column_wide(spres, spref, 1 << (w - 5), total, c0, P, work, work + MAP_WORDS, lv[0], lv[1]);
        return;
    }

    // ---- narrow values: per-column levels, one warp per column ----
    uint32_t* wbm = work + warp * 8;                                                   // 8 words
    uint16_t* wlev = (uint16_t*)(work + 64) + (size_t)warp * 512;                      // 2 x 256
    uint8_t* pos = (uint8_t*)(work + 64 + 256 * (PLAN_THREADS / 32)) + (size_t)warp * 256;
    for (int t = (int)warp; t < kw; t += PLAN_THREADS / 32) {
        const int col = c0 + t;
        uint32_t* bm = wbm;
        if (lane < 8) bm[lane] = 0u;
        __syncwarp();
        for (int i = (int)lane; i < m; i += 32) {
            const uint32_t v = (uint32_t)A[(size_t)i * n + col] & amask;
            if (v) atomicOr(&bm[v >> 5], 1u << (v & 31u));
        }
        __syncwarp();
        uint16_t* cur = wlev;
        uint16_t* nxt = wlev + 256;
        int len = extract_sorted(bm, cur, pos);
        if (k > 1) {
            // value -> level-1 position, for the k-tuple assembly
            for (int v = (int)lane; v < 256; v += 32) {
                const bool present = v > 0 && ((bm[v >> 5] >> (v & 31)) & 1u);
                P.col_rank1[(size_t)col * 256 + v] = present ? pos[v] : (uint8_t)0xff;
            }
        }
        if (lane == 0) P.col_len[(size_t)col * NLEV] = (uint16_t)len;
        __syncwarp();
        for (int lev = 1; lev < NLEV; lev++) {
            // Differences of consecutive sorted values; level lev + 1 is their
            // sorted distinct set.
            if (lane < 8) bm[lane] = 0u;
            __syncwarp();
            for (int e = (int)lane; e < len; e += 32) {
                const int d = (int)cur[e] - (e ? (int)cur[e - 1] : 0);
                atomicOr(&bm[d >> 5], 1u << (d & 31));
            }
            __syncwarp();
            const int nlen = extract_sorted(bm, nxt, pos);
            uint16_t* ptr = col_level_ptr(P, col, lev);
            for (int e = (int)lane; e < len; e += 32) {
                const int d = (int)cur[e] - (e ? (int)cur[e - 1] : 0);
                ptr[e] = pos[d];
            }
            if (lane == 0) P.col_len[(size_t)col * NLEV + lev] = (uint16_t)nlen;
            __syncwarp();
            uint16_t* tmp = cur; cur = nxt; nxt = tmp;
            len = nlen < P.l2max ? nlen : P.l2max;
        }
        for (int e = (int)lane; e < len; e += 32) P.col_vN[(size_t)col * P.l2max + e] = cur[e];
        __syncwarp();
    }
}

// The warps of a strip's table and of an output row take the 2 l ciphertext
// chains in blocks of 32: component c's chain j is lane c span + j. Each
// component starts a block of its own (span = lp), so that loads are aligned,
// unless packing them (span = l) saves a block: l = 1 .. 16 beyond a multiple
// of 32. Lanes without a chain of their own do their neighbour's, and write no
// output. 333 x 517 x 97 at w = 5 takes 7 blocks instead of 8: 4.48 -> 3.91 ms.
__host__ __device__ inline int lane_span(int l) {
    const int lp = (l + 31) / 32 * 32;
    return (l + 15) / 16 < lp / 16 ? l : lp;
}
__host__ __device__ inline int lane_blocks(int l) { return (lane_span(l) + 15) / 16; }

// Lane's component and chain (clamped) in block qb; whether it is its own.
__device__ __forceinline__ bool lane_chain(int qb, int span, int l, int& c, int& j) {
    const int q = qb * 32 + (int)(threadIdx.x & 31u);
    c = q >= span;
    j = q - (c ? span : 0);
    if (j < l) return true;
    j = l - 1;
    return false;
}

struct TableArgs {
    const uint4* ctB;      // affine ciphertext matrix n x l
    int m, n, l, w, k, lp, span, nq, n1max, l2max, emax;   // span, nq: lane_span, lane_blocks
    int s0, nstrips_chunk;
    uint4* scratch;        // lane-planar per-item scratch
    size_t item_u4;
    uint4* table;          // affine, quad-planar, table_points points
    size_t table_points;
    bool bshare;           // the 4 warps of each block share one strip's plan: share inversions
    // Digit build (table_block): digits per column, digits of all columns,
    // digits of the low half and the bits of both halves.
    int dpc, nd, ns, hl, hh;
    int pairs;             // signed pairs: 0 none, 1 of one column's digits, 2 of two columns
};

// What strip_excess compares, and whether a pass of few codes goes by chains
// (either; small: in launches of few blocks too).
struct FewArgs {
    bool either, small;
    int fixed, entry;
};

__device__ __forceinline__ void lp_store_aff(uint4* base, int e, unsigned lane, const aff& Q) {
    uint4* b = base + (size_t)e * 4 * 32 + lane;
    b[0] = fe_lo(Q.x);
    b[32] = fe_hi(Q.x);
    b[64] = fe_lo(Q.y);
    b[96] = fe_hi(Q.y);
}

__device__ __forceinline__ void lp_load_aff(aff& Q, const uint4* base, int e, unsigned lane) {
    const uint4* b = base + (size_t)e * 4 * 32 + lane;
    fe_from_quads(Q.x, b[0], b[32]);
    fe_from_quads(Q.y, b[64], b[96]);
}


// One forward step of the simultaneous inversion, for loops that produce
// lane-planar Jacobian entries: acc *= Z_e (a zero Z, i.e. infinity, counts
// as 1), prefix product stored as entry e of pref; ones tracks whether every
// Z so far is 1.
__device__ __forceinline__ void lp_pref_step(fe& acc, bool& ones, const fe& Z, uint4* pref, int e,
                                             unsigned lane) {
    fe z = Z;
    ones &= fe_is_one(z);
    if (fe_is_zero(z)) fe_one(z);
    acc = fmul(acc, z);
    lp_store_fe(pref, e, lane, acc);
}

// Backward half of the normalisation of E lane-planar Jacobian entries to
// affine (infinity -> (0, 0)), each handed to store(e, point):
// pref holds the per-lane prefix products of the Z's and acc their total
// (lp_pref_step).  One warp-wide inversion; when every Z in the warp is 1 the
// entries are copied without any.  The loads of entry e - 2 are prefetched
// into L2 while entry e is converted (lanes 0-23: the 24 lines of the
// Jacobian entry, lanes 24-31: the 8 lines of its prefix product).  All 32
// lanes call with the same E.
template <class Store>
__device__ __forceinline__ void lp_normalize_back(const uint4* src, int E, const uint4* pref, unsigned lane,
                                                  fe acc, bool ones, Store store, bool shared) {
    if (E <= 0) return;
    if (group_all(ones, shared)) {
        for (int e = 0; e < E; e++) {
            jac Pe;
            lp_load_jac(Pe, src, e, lane);
            aff out;
            out.x = Pe.X;
            out.y = Pe.Y;
            store(e, out);
        }
        return;
    }
    fe inv;
    group_inverse(inv, acc, shared);
    for (int e = E - 1; e >= 0; e--) {
        if (e >= 2) {
            const char* line = lane < 24u ? (const char*)(src + (size_t)(e - 2) * 192) + lane * 128u
                                          : (e >= 3 ? (const char*)(pref + (size_t)(e - 3) * 64) + (lane - 24u) * 128u
                                                    : nullptr);
            if (line) asm volatile("prefetch.global.L2 [%0];" ::"l"(line));
        }
        fe zinv;
        if (e > 0) {
            fe pr;
            lp_load_fe(pr, pref, e - 1, lane);
            zinv = fmul(inv, pr);
        } else {
            zinv = inv;
        }
        jac Pe;
        lp_load_jac(Pe, src, e, lane);
        fe z = Pe.Z;
        const bool is_inf = fe_is_zero(z);
        if (is_inf) fe_one(z);
        inv = fmul(inv, z);
        aff out;
        if (is_inf) {
            fe_zero(out.x);
            fe_zero(out.y);
        } else {
            jac_to_aff_with_zinv(out, Pe, zinv);
        }
        store(e, out);
    }
}

// Normalises E lane-planar Jacobian entries already in scratch (both passes).
template <class Store>
__device__ __forceinline__ void lp_normalize(const uint4* src, int E, uint4* pref, unsigned lane,
                                             Store store, bool shared) {
    if (E <= 0) return;
    bool ones = true;
    fe acc;
    fe_one(acc);
    for (int e = 0; e < E; e++) {
        fe z;
        lp_load_z(z, src, e, lane);
        lp_pref_step(acc, ones, z, pref, e, lane);
    }
    lp_normalize_back(src, E, pref, lane, acc, ones, store, shared);
}

// Normalises the E entries of a chain kept as (X, Y, ZZ, ZZZ)
// (jacz_madd_ratio_t): entry e holds X and Y in quads 0-3 of its 6-quad
// lane-planar slot in src and its ZZZ factor rr3_e in quads 4-5, and its ZZ
// factor rr2_e is entry e of rat, so ZZ_e = rr2_0 ... rr2_e (likewise ZZZ);
// zz, zzz are those of the last entry.  One inversion of zz zzz gives both
// ZZ^-1 and ZZZ^-1 of the last entry; going backwards each step multiplies
// them by the entry's factors: 4M per entry in all.  ones: every factor of
// this lane is 1.  With `shared` all threads of the block must call.
// STD: the points handed to store are canonical standard coordinates (the
// walk then starts from ZZ^-1 / R and ZZZ^-1 / R, and every product with X and
// Y is standard); otherwise they stay in the Montgomery domain.
template <bool STD, class Store>
__device__ __forceinline__ void lp_normalize_zz(const uint4* src, int E, const uint4* rat, unsigned lane,
                                                const fe& zz, const fe& zzz, bool ones, Store store,
                                                bool shared) {
    if (E <= 0) return;
    if (group_all(ones, shared)) {
        for (int e = 0; e < E; e++) {
            const uint4* b = src + (size_t)e * 6 * 32 + lane;
            aff out;
            fe_from_quads(out.x, b[0], b[32]);
            fe_from_quads(out.y, b[64], b[96]);
            if (STD) aff_from_mont(out);
            store(e, out);
        }
        return;
    }
    fe inv;
    group_inverse(inv, fmul(zz, zzz), shared);
    fe zzinv = fmul(inv, zzz);
    fe zzzinv = fmul(inv, zz);
    if (STD) {
        fe_from_mont(zzinv, zzinv);
        fe_from_mont(zzzinv, zzzinv);
    }
    for (int e = E - 1; e >= 0; e--) {
        if (e >= 2) {
            // lanes 0-23: the 24 lines of slot e - 2; 24-31: its ZZ factor.
            const char* line = lane < 24u ? (const char*)(src + (size_t)(e - 2) * 192) + lane * 128u
                                          : (const char*)(rat + (size_t)(e - 2) * 64) + (lane - 24u) * 128u;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(line));
        }
        const uint4* b = src + (size_t)e * 6 * 32 + lane;
        fe X, Y;
        fe_from_quads(X, b[0], b[32]);
        fe_from_quads(Y, b[64], b[96]);
        aff out;
        out.x = fmul(X, zzinv);
        out.y = fmul(Y, zzzinv);
        if (STD) {
            fe_canon(out.x, out.x);
            fe_canon(out.y, out.y);
        }
        store(e, out);
        if (e > 0) {
            fe r2, r3;
            lp_load_fe(r2, rat, e, lane);
            fe_from_quads(r3, b[128], b[160]);
            zzinv = fmul(zzinv, r2);
            zzzinv = fmul(zzzinv, r3);
        }
    }
}

// The chain P_e = P_{e-1} + A[ptr[e]] (e < len, P_{-1} at infinity) over
// affine addends A (lane-planar, 4 quads per entry), in (X, Y, ZZ, ZZZ):
// entry e's X, Y and ZZZ factor go to slot e of `slots` (6 quads), its ZZ
// factor to entry e of rat, as lp_normalize_zz reads them.  acc ends as the
// last entry; ones and ok as for jacz_madd_ratio_t.
static __device__ __noinline__ void lp_affine_chain(const uint4* A, const uint16_t* ptr, int len, uint4* slots,
                                                    uint4* rat, unsigned lane, jacz& acc, bool& ones, bool& ok) {
    aff D;
    jacz_set_inf(acc);
    ones = true;
    ok = true;
    for (int e = 0; e < len; e++) {
        lp_load_aff(D, A, ptr[e], lane);
        fe r2, r3;
        jacz_madd_ratio_t<PCMM_TABLE_INLINE>(acc, D, r2, r3, ok, e == 0);
        uint4* b = slots + (size_t)e * 6 * 32 + lane;
        b[0] = fe_lo(acc.X);
        b[32] = fe_hi(acc.X);
        b[64] = fe_lo(acc.Y);
        b[96] = fe_hi(acc.Y);
        b[128] = fe_lo(r3);
        b[160] = fe_hi(r3);
        lp_store_fe(rat, e, lane, r2);
        ones &= fe_is_one(r2) && fe_is_one(r3);
    }
}

// One warp per (strip, component c, 32 output columns); all lanes follow the
// same plan, so the control flow is warp-uniform.
// Table of one warp item (strip, component, 32 output columns) of a chunk;
// `scratch` is this warp's private scratch (a.item_u4 uint4).
__device__ __forceinline__ void table_item(const TableArgs& a, const PlanPtrs& P, long long item,
                                           uint4* scratch) {
    static_assert(NLEV >= 2, "the table build assumes at least two compression levels");
    const unsigned lane = threadIdx.x & 31u;
    const int s_local = (int)(item / a.nq);
    int c, j;
    lane_chain((int)(item % a.nq), a.span, a.l, c, j);
    const int s = a.s0 + s_local;
    const int c0 = s * a.k;
    const int kw = (c0 + a.k <= a.n) ? a.k : a.n - c0;
    const size_t nl = (size_t)a.n * a.l;
    const uint4* Bc = a.ctB + (size_t)c * 4 * nl;
    const uint32_t amask = (1u << a.w) - 1u;

    // Scratch regions of this warp item (see make_layout).
    uint4* coltab = scratch;                                              // n1max Jacobian
    uint4* levA = coltab + (size_t)a.n1max * 192;                         // l2max Jacobian
    uint4* levB = levA + (size_t)a.l2max * 192;                           // l2max Jacobian
    uint4* l2aff = levB + (size_t)a.l2max * 192;                          // l2max affine
    uint4* colaff = l2aff + (size_t)a.l2max * 128;                        // k * n1max affine (k > 1)
    uint4* part = colaff + (a.k > 1 ? (size_t)a.k * a.n1max * 128 : 0);   // emax affine (k > 1)
    uint4* pref = part + (a.k > 1 ? (size_t)a.emax * 128 : 0);            // max(emax, n1max) field elements

    const int E = P.nent[s];
    const size_t tbase = (size_t)s_local * a.emax;
    // The strip table holds canonical standard coordinates; everything else
    // in this function is in the Montgomery domain.
    auto store_table = [&](int e, const aff& q) {
        store_aff(a.table, a.table_points, ((tbase + e) * 2 + c) * a.lp + j, q);
    };
    auto store_table_mont = [&](int e, const aff& q) {
        aff t = q;
        aff_from_mont(t);
        store_table(e, t);
    };
    bool bad = false, dbad = false;

    for (int t = 0; t < kw; t++) {
        const int col = c0 + t;
        aff Pb;
        load_aff(Pb, Bc, nl, (size_t)col * a.l + j);
        aff_to_mont(Pb);
        int lens[NLEV];
#pragma unroll
        for (int q = 0; q < NLEV; q++) lens[q] = P.col_len[(size_t)col * NLEV + q];
        bad |= lens[0] > a.n1max;
#pragma unroll
        for (int q = 1; q < NLEV; q++) bad |= lens[q] > a.l2max;
#ifdef PCMM_DEBUG_BOUNDS
        // Each tracking pointer of level lev (lens[lev-1] of them) names an
        // entry of level lev + 1 (lens[lev] entries); for k = 1 the strip
        // table is the column's level 1.
        for (int lev = 1; lev < NLEV && !bad; lev++) {
            const uint16_t* pl = col_level_ptr(P, col, lev);
            for (int e = 0; e < lens[lev - 1]; e++) dbad |= pl[e] >= lens[lev];
        }
        if (a.k == 1) dbad |= E != lens[0];
        bad |= dbad;
#endif
        if (bad) break;
        // Level N: multiples of the compressed values (double-and-add).
        uint4* src = levA;
        for (int e = 0; e < lens[NLEV - 1]; e++) {
            jac T;
            jac_mul_small(T, Pb, P.col_vN[(size_t)col * P.l2max + e]);
            lp_store_jac(src, e, lane, T);
        }
        uint4* alt = levB;
        // Levels N-1..2: un-sort by the tracking pointers, then prefix sums of
        // Jacobian points; level 2 also takes the forward pass of its
        // normalisation.  A long level 2 (wide values: hundreds of entries) is
        // instead built like level 1, as a chain of mixed additions over its
        // level 3 normalised to affine (plan data, so uniform over the strip).
        const bool l2chain = NLEV > 2 && lens[1] >= 32;
        auto store_l2 = [&](int e, const aff& q) { lp_store_aff(l2aff, e, lane, q); };
        fe pacc;
        bool pones = true;
        fe_one(pacc);
        auto jacobian_level = [&](int lev) {
            const uint16_t* ptr = col_level_ptr(P, col, lev);
            jac acc, D;
            jac_set_inf(acc);
            for (int e = 0; e < lens[lev - 1]; e++) {
                lp_load_jac(D, src, ptr[e], lane);
                jac_add(acc, D);
                lp_store_jac(alt, e, lane, acc);
                if (lev == 2) lp_pref_step(pacc, pones, acc.Z, pref, e, lane);
            }
        };
        for (int lev = NLEV - 1; lev >= (l2chain ? 3 : 2); lev--) {
            jacobian_level(lev);
            uint4* tmp = src; src = alt; alt = tmp;
        }
        if (!l2chain) {
            // Level 2 (multiples of the level-1 differences) to affine, so that
            // the level-1 prefix sums are mixed additions.
            if (NLEV > 2) lp_normalize_back(src, lens[1], pref, lane, pacc, pones, store_l2, a.bshare);
            else lp_normalize(src, lens[1], pref, lane, store_l2, a.bshare);
        } else {
            // Level 3 (Jacobian, in src) to affine in l2aff, then level 2 as a
            // chain over it into alt; l2aff then receives level 2.
            lp_normalize(src, lens[2], pref, lane, store_l2, a.bshare);
            jacz acc2;
            bool ones2, ok2;
            lp_affine_chain(l2aff, col_level_ptr(P, col, 2), lens[1], alt, pref, lane, acc2, ones2, ok2);
            if (group_all(ok2, a.bshare)) {
                lp_normalize_zz<false>(alt, lens[1], pref, lane, acc2.ZZ, acc2.ZZZ, ones2, store_l2, a.bshare);
            } else {
                jacobian_level(2);
                lp_normalize_back(alt, lens[1], pref, lane, pacc, pones, store_l2, a.bshare);
            }
        }
        // Level 1: the multiples of the column's sorted distinct values,
        // with the forward pass of their normalisation.
        // The chain runs in (X, Y, ZZ, ZZZ) coordinates; each entry keeps X,
        // Y and the factors its ZZ and ZZZ were multiplied by, for the
        // normalisation.  A chain that meets infinity (an input at infinity)
        // is recomputed in Jacobian coordinates and normalised the general way.
        const uint16_t* ptr1 = col_level_ptr(P, col, 1);
        jacz acc;
        bool cones, cok;
        lp_affine_chain(l2aff, ptr1, lens[0], coltab, pref, lane, acc, cones, cok);
        const bool chain_ok = group_all(cok, a.bshare);
        if (!chain_ok) {
            jac accj;
            aff D;
            jac_set_inf(accj);
            for (int e = 0; e < lens[0]; e++) {
                lp_load_aff(D, l2aff, ptr1[e], lane);
                jac_madd(accj, D);
                lp_store_jac(coltab, e, lane, accj);
            }
        }
        uint4* ca = colaff + (size_t)t * a.n1max * 128;
        auto store_col = [&](int e, const aff& q) { lp_store_aff(ca, e, lane, q); };
        if (a.k == 1) {
            // The column table is the strip table (E = lens[0] entries).
            if (chain_ok) lp_normalize_zz<true>(coltab, E, pref, lane, acc.ZZ, acc.ZZZ, cones, store_table, a.bshare);
            else lp_normalize(coltab, E, pref, lane, store_table_mont, a.bshare);
            return;
        }
        if (chain_ok) lp_normalize_zz<false>(coltab, lens[0], pref, lane, acc.ZZ, acc.ZZZ, cones, store_col, a.bshare);
        else lp_normalize(coltab, lens[0], pref, lane, store_col, a.bshare);
    }
    if (bad) {
        if (lane == 0) atomicOr(P.status, dbad ? DEV_ERR_BOUNDS : DEV_ERR_PLAN);
        return;
    }
#ifdef PCMM_DEBUG_BOUNDS
    // Every component of every tuple names an entry of its column table.
    for (int e = 0; e < E && !dbad; e++) {
        const uint32_t code = P.codes[(size_t)s * a.emax + e];
        for (int t = 0; t < kw; t++) {
            const uint32_t x = (code >> (a.w * t)) & amask;
            if (x) dbad |= P.col_rank1[(size_t)(c0 + t) * 256 + x] >= P.col_len[(size_t)(c0 + t) * NLEV];
        }
    }
    if (E > a.emax || dbad) {
        if (lane == 0) atomicOr(P.status, DEV_ERR_BOUNDS);
        return;
    }
#endif
    // k > 1: one entry per distinct k-tuple, the sum of its columns' (affine)
    // entries, computed in affine coordinates one addition round at a time:
    // round r adds the (r+1)-th non-zero component of every tuple that has
    // one.  The additions of a round are independent, so their slopes share
    // one simultaneous inversion (per-lane prefix products of the x
    // differences, then one warp-wide inversion): about 5M + 1S per entry
    // instead of a mixed addition and a normalisation.  Pairs the affine
    // formula cannot take (infinity, equal or opposite points) use the
    // complete Jacobian addition and their own inversion on a rare branch.
    auto comp = [&](uint32_t code, int nth, uint32_t& v) -> int {
        int cnt = 0;
        for (int t = 0; t < kw; t++) {
            const uint32_t x = (code >> (a.w * t)) & amask;
            if (x) {
                if (cnt == nth) { v = x; return t; }
                cnt++;
            }
        }
        return -1;
    };
    auto col_entry = [&](aff& Q, int t, uint32_t v) {
        const int r1 = P.col_rank1[(size_t)(c0 + t) * 256 + v];
        lp_load_aff(Q, colaff + (size_t)t * a.n1max * 128, r1, lane);
    };
    int maxc = 0;
    for (int e = 0; e < E; e++) {
        const uint32_t code = P.codes[(size_t)s * a.emax + e];
        int cnt = 0;
        for (int t = 0; t < kw; t++) cnt += ((code >> (a.w * t)) & amask) != 0u;
        maxc = cnt > maxc ? cnt : maxc;
    }
    for (int r = 1; r < maxc; r++) {
        fe acc;
        fe_one(acc);
        for (int e = 0; e < E; e++) {
            const uint32_t code = P.codes[(size_t)s * a.emax + e];
            uint32_t vq, v0;
            const int tq = comp(code, r, vq);
            fe dx;
            fe_one(dx);
            if (tq >= 0) {
                aff Pp, Qq;
                if (r == 1) col_entry(Pp, comp(code, 0, v0), v0);
                else lp_load_aff(Pp, part, e, lane);
                col_entry(Qq, tq, vq);
                if (!aff_is_inf(Pp) && !aff_is_inf(Qq)) {
                    fe_sub(dx, Qq.x, Pp.x);
                    if (fe_is_zero(dx)) fe_one(dx);
                }
            }
            acc = fmul(acc, dx);
            lp_store_fe(pref, e, lane, acc);
        }
        fe inv;
        group_inverse(inv, acc, a.bshare);
        for (int e = E - 1; e >= 0; e--) {
            const uint32_t code = P.codes[(size_t)s * a.emax + e];
            uint32_t vq, v0;
            const int tq = comp(code, r, vq);
            if (tq < 0) continue;          // its factor was 1
            aff Pp, Qq, R;
            if (r == 1) col_entry(Pp, comp(code, 0, v0), v0);
            else lp_load_aff(Pp, part, e, lane);
            col_entry(Qq, tq, vq);
            fe dinv;
            if (e > 0) {
                fe pr;
                lp_load_fe(pr, pref, e - 1, lane);
                dinv = fmul(inv, pr);
            } else {
                dinv = inv;
            }
            bool special = aff_is_inf(Pp) || aff_is_inf(Qq);
            fe dx;
            if (!special) {
                fe_sub(dx, Qq.x, Pp.x);
                special = fe_is_zero(dx);
            }
            if (!special) {
                inv = fmul(inv, dx);
                fe dy, lam, t0;
                fe_sub(dy, Qq.y, Pp.y);
                lam = fmul(dy, dinv);              // slope
                t0 = fsqr(lam);
                fe_sub(t0, t0, Pp.x);
                fe_sub(R.x, t0, Qq.x);             // x3 = lam^2 - x1 - x2
                fe_sub(t0, Pp.x, R.x);
                t0 = fmul(lam, t0);
                fe_sub(R.y, t0, Pp.y);             // y3 = lam (x1 - x3) - y1
            } else {
                jac J;
                jac_from_aff(J, Pp);
                jac_madd(J, Qq);
                if (jac_is_inf(J)) {
                    fe_zero(R.x);
                    fe_zero(R.y);
                } else {
                    fe zi;
                    fe_inv(zi, J.Z);
                    jac_to_aff_with_zinv(R, J, zi);
                }
            }
            lp_store_aff(part, e, lane, R);
        }
    }
    for (int e = 0; e < E; e++) {
        const uint32_t code = P.codes[(size_t)s * a.emax + e];
        uint32_t v1, v0;
        aff R;
        if (comp(code, 1, v1) < 0) col_entry(R, comp(code, 0, v0), v0);   // a single component
        else lp_load_aff(R, part, e, lane);
        store_table_mont(e, R);
    }
}

// ---------------------------------------------------------------------------
// Table build by digits.
//
// A strip code of w k bits is cut into digits of at most four bits, none
// across two columns, and the digits into a low and a high half. Then
//   1. the multiples of every digit's point: chains of mixed additions, one
//      inversion for all digits of the same place;
//   2. both halves' tables, digit by digit: E[v 2^o + g] = E[v 2^o] + E[g];
//   3. the strip's entries: code = v 2^hl + u gives L[u] + H[v], one affine
//      addition per distinct code.
// Within a round of 2 and in 3 the additions are independent, so their slopes
// share one inversion of the block: 5M + 1S an entry. The chains of prefix
// sums over the sorted values (table_item) are serial, and cost 12M + 2S an
// entry with its normalisation. The values of a column (k = 1) come from its
// compressed levels, prefix sums of integers here.
//
// Points are standard residues from the digits' tables on: with the inverse
// of a product a b / R a slope comes out in the Montgomery domain, its square
// is reduced twice, and its product with x1 - x3 is standard again.

// Pairs whose x's are equal or of which one is at infinity. They take the
// rare, out-of-line way: pair_factor gives the factor that the pair
// contributes to the shared inversion (2 y for a doubling, 1 where there is
// nothing to invert), pair_sum the sum, given the inverse of the factor.
enum : int { PAIR_ADD = 0, PAIR_SECOND = 1, PAIR_FIRST = 2, PAIR_DOUBLE = 3, PAIR_CANCEL = 4 };

__device__ __forceinline__ int pair_kind(const aff& A, const aff& B, const fe& dx) {
    if (aff_is_inf(B)) return PAIR_FIRST;
    if (aff_is_inf(A)) return PAIR_SECOND;
    if (!fe_is_zero(dx)) return PAIR_ADD;
    return fe_equal(A.y, B.y) && !fe_is_zero(A.y) ? PAIR_DOUBLE : PAIR_CANCEL;
}

// The same factor serves A + B and A - B: one of them doubles where the other
// cancels.
static __device__ __noinline__ void pair_factor(fe& dx, const aff& A, const aff& B) {
    const int kind = pair_kind(A, B, dx);
    if (kind == PAIR_ADD) return;
    fe_one(dx);
    if (kind >= PAIR_DOUBLE && !fe_is_zero(A.y)) fe_add(dx, A.y, A.y);
}

// S = A + B for standard residues, finv = (factor)^-1 R^2.
static __device__ __noinline__ void pair_sum(aff& S, const aff& A, const aff& B, const fe& finv) {
    fe d, num;
    fe_sub(d, B.x, A.x);
    const int kind = pair_kind(A, B, d);
    if (kind == PAIR_FIRST) {
        S = A;
        return;
    }
    if (kind == PAIR_SECOND) {
        S = B;
        return;
    }
    if (kind == PAIR_CANCEL) {
        fe_zero(S.x);
        fe_zero(S.y);
        return;
    }
    if (kind == PAIR_DOUBLE) {           // 3 x^2 - 3
        fe one, t;
        fe_zero(one);
        one.v[0] = 1u;
        fe_to_mont(t, fsqr(A.x));
        fe_sub(t, t, one);
        fe_add(num, t, t);
        fe_add(num, num, t);
    } else {
        fe_sub(num, B.y, A.y);
    }
    const fe lam = fmul(num, finv);
    fe t = fsqr(lam);
    fe_from_mont(t, t);
    fe_sub(t, t, A.x);
    fe_sub(S.x, t, B.x);
    fe_sub(t, A.x, S.x);
    t = fmul(lam, t);
    fe_sub(S.y, t, A.y);
}

__device__ __forceinline__ bool words345_zero(const fe& a) { return (a.v[3] | a.v[4] | a.v[5]) == 0u; }

// Canonical form of a sum's coordinate; LATE: behind a test that one value in
// 2^32 passes (p's top word is all ones), 2% off the tables of one column's
// signed pairs (w = 16 22.05 -> 21.6 ms) and 1% onto the others.
template <bool LATE>
__device__ __forceinline__ void canon_of(fe& r, const fe& a) {
    if (!LATE) {
        fe_canon(r, a);
        return;
    }
    r = a;
    if (r.v[7] == 0xffffffffu) fe_canon(r, r);
}

// With both signs the multiplications are called: inlined, two copies of the
// sum outgrow the instruction cache (w = 8 below 11.1 against 10.5 ms).
template <bool BOTH>
__device__ __forceinline__ fe batch_mul(const fe& a, const fe& b) {
    if (BOTH) return fmul(a, b);
    fe r;
    fe_mul(r, a, b);
    return r;
}

// A + B (bit 0 of pair(i, A, B)) and, for BOTH, A - B (bit 1) for i < cnt, each handed to
// put(i, 0 or 1, sum) in canonical form: pair sets the two lane-planar canonical
// entries and returns 0 where there is nothing to add. Both signs share the
// difference of x and its inverse: 7M + 2S instead of 10M + 2S. pref: cnt field
// elements of lane-planar scratch. All 128 threads of the block call; cnt may
// differ from warp to warp. `turn` names the warp that inverts.
template <bool BOTH, bool LATE, class Pair, class Put>
__device__ __forceinline__ void affine_batch(int cnt, Pair pair, Put put, uint4* pref, uint4* sm, unsigned turn) {
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, tid = threadIdx.x;
    const unsigned all = 0xffffffffu;
    // Forward: the prefix products of the differences of x.
    fe run;
    fe_one(run);
#pragma unroll 1
    for (int i = 0; i < cnt; i++) {
        const uint4 *pa, *pb;
        if (!pair(i, pa, pb)) continue;
        fe ax, bx, dx;
        fe_from_quads(ax, pa[0], pa[32]);
        fe_from_quads(bx, pb[0], pb[32]);
        fe_sub_canon(dx, bx, ax);
        // Words 3..5 are zero in 0 and in p: no zero passes this test.
        if (__any_sync(all, words345_zero(dx) || words345_zero(ax) || words345_zero(bx))) {
            aff A, B;
            lp_load_aff(A, pa, 0, 0);
            lp_load_aff(B, pb, 0, 0);
            pair_factor(dx, A, B);
        }
        lp_store_fe(pref, i, lane, run);
        fe_mul(run, run, dx);
    }
    sm[tid] = fe_lo(run);
    sm[128 + tid] = fe_hi(run);
    __syncwarp();
    __syncthreads();
    if (warp == (turn & 3u)) fold_inverse128(sm);
    __syncthreads();
    fe inv;
    fe_from_quads(inv, sm[tid], sm[128 + tid]);
    // Backward: each difference's inverse, the slope and the sum.
#pragma unroll 1
    for (int i = cnt - 1; i >= 0; i--) {
        const uint4 *pa, *pb;
        const unsigned want = pair(i, pa, pb);
        if (!want) continue;
        aff A, B;
        fe pr, dinv, dx;
        lp_load_fe(pr, pref, i, lane);
        lp_load_aff(A, pa, 0, 0);
        lp_load_aff(B, pb, 0, 0);
        fe_sub_canon(dx, B.x, A.x);
        const bool rare = __any_sync(all, words345_zero(dx) || words345_zero(A.x) || words345_zero(B.x));
        if (rare) {
            pair_factor(dx, A, B);
            dinv = fmul(inv, pr);
            inv = fmul(inv, dx);
            for (int sign = 0; sign < (BOTH ? 2 : 1); sign++) {
                aff S;
                if (sign) {
                    fe_zero(S.y);
                    fe_sub_canon(B.y, S.y, B.y);
                }
                if (BOTH && !((want >> sign) & 1u)) continue;
                pair_sum(S, A, B, dinv);
                fe_canon(S.x, S.x);
                fe_canon(S.y, S.y);
                put(i, sign, S);
            }
            continue;
        }
        dinv = batch_mul<BOTH>(inv, pr);
        inv = batch_mul<BOTH>(inv, dx);
        auto finish = [&](int sign) {
            aff S;
            fe lam, t;
            fe_sub_canon(t, B.y, A.y);
            lam = batch_mul<BOTH>(t, dinv);
            if (BOTH) {
                t = fsqr(lam);
                fe_from_mont(t, t);
            } else {
                t = fe_sqr_std(lam);
            }
            fe_sub_canon(t, t, A.x);
            fe_sub_canon(t, t, B.x);
            canon_of<LATE>(S.x, t);
            fe_sub_canon(t, A.x, S.x);
            t = batch_mul<BOTH>(lam, t);
            fe_sub_canon(S.y, t, A.y);
            canon_of<LATE>(S.y, S.y);
            put(i, sign, S);
        };
        if (!BOTH || (want & 1u)) finish(0);
        if (BOTH && (want & 2u)) {
            fe zero;
            fe_zero(zero);
            fe_sub_canon(B.y, zero, B.y);
            finish(1);
        }
    }
}

// The generator (Montgomery domain): it stands in for a point at infinity in
// the digits' chains, whose multiples the lane then stores as infinity.
__device__ __forceinline__ void aff_generator(aff& G) {
    const uint32_t x[8] = {0x18a9143cu, 0x79e730d4u, 0x5fedb601u, 0x75ba95fcu,
                           0x77622510u, 0x79fb732bu, 0xa53755c6u, 0x18905f76u};
    const uint32_t y[8] = {0xce95560au, 0xddf25357u, 0xba19e45cu, 0x8b4ab8e4u,
                           0xdd21f325u, 0xd2e88688u, 0x25885d85u, 0x8571ff18u};
#pragma unroll
    for (int i = 0; i < 8; i++) {
        G.x.v[i] = x[i];
        G.y.v[i] = y[i];
    }
}

// v B in affine coordinates for a lane whose chain met infinity, which takes a
// point of order 16 or less and so an input off the curve.
static __device__ __noinline__ aff small_multiple(const aff& B, uint32_t v) {
    jac J;
    jac_mul_small(J, B, v);
    aff Q;
    if (jac_is_inf(J)) {
        fe_zero(Q.x);
        fe_zero(Q.y);
        return Q;
    }
    fe zi;
    fe_inv(zi, J.Z);
    jac_to_aff_with_zinv(Q, J, zi);
    return Q;
}

// 8 A + v B for a lane whose chain over two columns met infinity.
static __device__ __noinline__ aff small_sum(const aff& A, const aff& B, uint32_t v) {
    jac J, K;
    jac_mul_small(J, A, 8u);
    jac_mul_small(K, B, v);
    jac_add(J, K);
    aff Q;
    if (jac_is_inf(J)) {
        fe_zero(Q.x);
        fe_zero(Q.y);
        return Q;
    }
    fe zi;
    fe_inv(zi, J.Z);
    jac_to_aff_with_zinv(Q, J, zi);
    return Q;
}

// Bits of digit d: four, or what is left of its column.
__host__ __device__ inline int digit_bits(const TableArgs& a, int d) {
    const int r = a.w - 4 * (d % a.dpc);
    return r < 4 ? r : 4;
}

// Signed pairs: two digits d and d + 1 that come first in their half (or are
// the only two), so that one factor of the shared inversion serves two of their
// entries (affine_batch), and the multiples 9..15 of the lower digit's point are
// not needed.
//  - Digits of one column: an entry 16 v + u is 16 v + u for u <= 8 and
//    16 (v + 1) - (16 - u) above. It takes one more multiple of the upper digit's
//    point, 2^bits, which waits in row 0 of the other half (no code 0 is ever
//    read). With one bit in the upper digit there is nothing to share.
//  - Columns of four bits: v P1 + u P0 is (v P1 + 8 P0) + (u - 8) P0, and the
//    upper digit's chain goes on from 8 P0 where the lower one's ends.
// Table times without and with signed pairs (ms): 1024 x 1024 x 256 at w = 8 12.6
// and 10.2, with one value in ten not zero 7.0 and 6.3, at w = 4 6.2 and 5.3; 512
// x 512 x 256 at w = 16 24.0 and 21.6.
__host__ __device__ inline bool signed_pair(const TableArgs& a, int d, int end) {
    if (d + 1 >= end) return false;
    return a.dpc == 1 ? a.w == 4 : d % a.dpc + 1 < a.dpc && digit_bits(a, d + 1) >= 2;
}

// Shared memory of the digit build, in uint4 per block: the shared inversion,
// and for each warp the entry of every code and the list of pairs.
constexpr int DIGIT_SHARED_U4 = 256 + 4 * 48;

// Scratch of the digit build, in uint4 per warp: the values of the level
// lists, the factors of the digits' chains (4 quads an entry; X and Y wait in
// the half's entry), the next places' base points, both halves' tables and
// the prefix products.
struct DigitScratch {
    size_t vals, rat, base, half, pref, total;
};
__host__ __device__ inline DigitScratch digit_scratch(int w, int k, int dpc, int hl, int hh, int n1max, int l2max,
                                                      int emax) {
    DigitScratch D;
    size_t off = 0;
    D.vals = off;
    off += (size_t)((n1max + 2 * l2max) * 2 + 15) / 16 + 1;
    D.rat = off;
    off += (size_t)k * (1 << (w < 4 ? w : 4)) * 128;
    D.base = off;
    off += (size_t)(dpc > 1 ? k : 0) * 128;
    D.half = off;
    off += ((size_t)(1 << hl) + (size_t)(1 << hh)) * 128;
    D.pref = off;
    size_t np = 0;                       // a single digit has no pairs to add
    if (k * dpc > 1) {
        np = (size_t)2 << (hl > hh ? hl : hh);
        if (np < (size_t)emax) np = emax;
    }
    off += (np > (size_t)k ? np : (size_t)k) * 64;
    D.total = off;
    return D;
}

// The values of column col's level 1, in lists of 16-bit words at buf:
// level N's values, and each level below as prefix sums over its tracking
// pointers. One warp.
__device__ __forceinline__ const uint16_t* column_values(const PlanPtrs& P, int col, const int* lens, uint16_t* buf) {
    const unsigned lane = threadIdx.x & 31u;
    const uint16_t* cur = P.col_vN + (size_t)col * P.l2max;
    for (int lev = NLEV - 1; lev >= 1; lev--) {
        const uint16_t* ptr = col_level_ptr(P, col, lev);
        uint16_t* out = lev == 1 ? buf + 2 * P.l2max : buf + (lev & 1) * P.l2max;
        uint32_t carry = 0;
        for (int b = 0; b < lens[lev - 1]; b += 32) {
            const int e = b + (int)lane;
            uint32_t x = e < lens[lev - 1] ? cur[ptr[e]] : 0u;
#pragma unroll
            for (int k = 1; k < 32; k <<= 1) {
                const uint32_t o = __shfl_up_sync(0xffffffffu, x, k);
                if ((int)lane >= k) x += o;
            }
            x += carry;
            if (e < lens[lev - 1]) out[e] = (uint16_t)x;
            carry = __shfl_sync(0xffffffffu, x, 31);
        }
        __syncwarp();
        cur = out;
    }
    return cur;
}

// Table of one warp item by digits; PAIRS: no signed pairs, pairs of one column's
// digits (1; 3 as part of the batched kernel) or of two columns (a.pairs). One copy
// for all would slow each by 2-5%.
// All 128 threads of the block call (valid: the warp has an item); sm:
// DIGIT_SHARED_U4 uint4 of shared memory.
template <int PAIRS>
__device__ __forceinline__ void table_block(const TableArgs& a, const PlanPtrs& P, long long item, bool valid,
                                            uint4* scratch, uint4* sm) {
    constexpr bool SIGNED = PAIRS != 0;
    // Read rather than known from PAIRS: the compiler then made 5.3 ms (w = 4) of
    // what took 5.5.
    const bool cross = PAIRS == 2 && a.dpc == 1;   // of two columns
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, tid = threadIdx.x;
    const int s_local = valid ? (int)(item / a.nq) : 0;
    int c, j;
    lane_chain(valid ? (int)(item % a.nq) : 0, a.span, a.l, c, j);
    const int s = a.s0 + s_local;
    const int c0 = s * a.k;
    const int kw = !valid ? 0 : (c0 + a.k <= a.n) ? a.k : a.n - c0;
    const size_t nl = (size_t)a.n * a.l;
    const uint4* Bc = a.ctB + (size_t)c * 4 * nl;
    const DigitScratch D = digit_scratch(a.w, a.k, a.dpc, a.hl, a.hh, a.n1max, a.l2max, a.emax);
    uint4* rat = scratch + D.rat;
    uint4* base = scratch + D.base;
    uint4* half = scratch + D.half;
    uint4* pref = scratch + D.pref;
    uint4* high = half + ((size_t)128 << a.hl);
    // Signed pairs of each half's first two digits, and of the only two.
    const bool pairs = SIGNED && (a.dpc == 1) == cross;
    const bool two = pairs && a.nd == 2 && signed_pair(a, 0, 2);
    const bool sp[2] = {two || (pairs && signed_pair(a, 0, a.ns)), pairs && signed_pair(a, a.ns, a.nd)};
    const int second[2] = {1, a.ns + 1};
    auto lower = [&](int dg) { return (sp[0] && dg == 0) || (sp[1] && dg == a.ns); };
    auto upper = [&](int dg) { return (sp[0] && dg == second[0]) || (sp[1] && dg == second[1]); };
    int E = valid ? P.nent[s] : 0;
    unsigned turn = blockIdx.x;

    // The strip's distinct codes.
    const uint16_t* codes = P.codes + (size_t)s * a.emax;
    bool bad = E > a.emax, dbad = false;
    for (int t = 0; t < kw; t++) {
        int lens[NLEV];
#pragma unroll
        for (int q = 0; q < NLEV; q++) lens[q] = P.col_len[(size_t)(c0 + t) * NLEV + q];
        bad |= lens[0] > a.n1max;
#pragma unroll
        for (int q = 1; q < NLEV; q++) bad |= lens[q] > a.l2max;
#ifdef PCMM_DEBUG_BOUNDS
        // Each tracking pointer names an entry of the next level, each tuple
        // component an entry of its column.
        for (int lev = 1; lev < NLEV && !bad; lev++) {
            const uint16_t* pl = col_level_ptr(P, c0 + t, lev);
            for (int e = 0; e < lens[lev - 1]; e++) dbad |= pl[e] >= lens[lev];
        }
        for (int e = 0; a.k > 1 && e < E && !bad; e++) {
            const uint32_t x = ((uint32_t)codes[e] >> (a.w * t)) & ((1u << a.w) - 1u);
            if (x) dbad |= P.col_rank1[(size_t)(c0 + t) * 256 + x] >= lens[0];
        }
        bad |= dbad;
#endif
        if (a.k == 1 && !bad) {
            bad |= E > lens[0];
#ifdef PCMM_DEBUG_BOUNDS
            dbad |= E != lens[0];
            bad |= dbad;
#endif
            codes = column_values(P, c0, lens, (uint16_t*)(scratch + D.vals));
        }
    }
    if (bad) {
        if (lane == 0) atomicOr(P.status, dbad ? DEV_ERR_BOUNDS : DEV_ERR_PLAN);
        E = 0;
    }

    // 1. Place by place, the digits' multiples: entry v of a digit at bit o
    // of its half goes to half entry v 2^o (standard coordinates), and 2^4
    // times its point (Montgomery domain) to the column's base. Of the lower
    // digit of a signed pair 1..8 and 16 are made, of the upper one 1..2^bits;
    // across two columns 1..8 and the sums 8 P0 + v P1, in one chain.
    auto half_at = [&](int dg, int& o) -> uint4* {
        o = 0;
        for (int x = dg < a.ns ? 0 : a.ns; x < dg; x++) o += digit_bits(a, x);
        return dg < a.ns ? half : high;
    };
    // Steps of a digit's chain, and the row of its entry e.
    auto chain_len = [&](int dg, bool more) -> int {
        if (lower(dg)) return cross ? 8 : 9;
        return (1 << digit_bits(a, dg)) - (more || upper(dg) ? 0 : 1);
    };
    auto spare = [&](int dg) -> uint4* { return dg < a.ns ? high : half; };
    auto chain_row = [&](int dg, int t, int e, int len, bool more, uint4* hb, int o) -> uint4* {
        if (cross && upper(dg)) return hb + (((size_t)e << o) + (two ? 0 : 8)) * 128;
        if (e == len - 1) {
            if (more) return base + (size_t)t * 128;
            if (upper(dg)) return spare(dg);
        }
        return hb + ((size_t)(e + 1) << o) * 128;
    };
    uint32_t atinf = 0;          // columns (by t) whose point is infinity in this lane
    for (int place = 0; place < a.dpc; place++) {
        const bool more = place + 1 < a.dpc;
        uint32_t failed = 0;     // columns whose chain met infinity in this lane
        fe acc;
        fe_one(acc);
        jacz P1;
        bool ok = true;
        for (int t = 0; t < kw; t++) {
            const int dg = t * a.dpc + place, len = chain_len(dg, more);
            aff B, S;
            if (place == 0) {
                load_aff(S, Bc, nl, (size_t)(c0 + t) * a.l + j);
                fe_canon(S.x, S.x);
                fe_canon(S.y, S.y);
                if (aff_is_inf(S)) atinf |= 1u << t;
                B = S;
                aff_to_mont(B);
            } else {
                lp_load_aff(B, base, t, lane);
                if (aff_is_inf(B)) atinf |= 1u << t;
                S = B;
                aff_from_mont(S);
            }
            if ((atinf >> t) & 1u) {
                fe_zero(S.x);
                fe_zero(S.y);
                aff_generator(B);
            }
            int o;
            uint4* hb = half_at(dg, o);
            lp_store_aff(hb, 1 << o, lane, S);
            if (len < 2) continue;
            const bool goes_on = cross && upper(dg);
            if (!goes_on) {
                P1.X = B.x;
                P1.Y = B.y;
                fe_one(P1.ZZ);
                fe_one(P1.ZZZ);
                ok = true;
            }
            uint4* rt = rat + (size_t)t * (size_t)(1 << (a.w < 4 ? a.w : 4)) * 128;
            // Entry e is (e + 1) times the point: X and Y to its place, ZZ's and
            // ZZZ's factors to slot e.  The first step is a doubling.
#pragma unroll 1
            for (int e = 1; e < len; e++) {
                uint4* xy = chain_row(dg, t, e, len, more, hb, o) + lane;
                uint4* f = rt + (size_t)e * 128 + lane;
                fe r2, r3;
                if (SIGNED && e == 8 && lower(dg)) {
                    jacz_dbl_ratio(P1, r2, r3);
                    if (fe_is_zero(P1.ZZ)) ok = false;
                } else {
                    jacz_madd_ratio_t<PAIRS == 2 ? PCMM_CROSS_INLINE : PAIRS == 1 ? PCMM_SIGNED_INLINE : PCMM_DIGIT_INLINE>(P1, B, r2, r3, ok, false);
                }
                if (goes_on && e == 1 && ((atinf >> (t - 1)) & 1u)) {
                    // Nothing to go on from: the upper column's own multiples.
                    P1.X = B.x;
                    P1.Y = B.y;
                    fe_one(P1.ZZ);
                    fe_one(P1.ZZZ);
                    fe_one(r2);
                    fe_one(r3);
                }
                xy[0] = fe_lo(P1.X);
                xy[32] = fe_hi(P1.X);
                xy[64] = fe_lo(P1.Y);
                xy[96] = fe_hi(P1.Y);
                f[0] = fe_lo(r2);
                f[32] = fe_hi(r2);
                f[64] = fe_lo(r3);
                f[96] = fe_hi(r3);
            }
            if (cross && lower(dg) && t + 1 < kw) continue;
            // The chain's product ZZ ZZZ for the shared inversion; ZZ and ZZZ
            // wait in slot 0, whose factors would be 1.
            aff zz;
            zz.x = P1.ZZ;
            zz.y = P1.ZZZ;
            if (!ok) {
                failed |= (goes_on ? 3u << (t - 1) : 1u << t);
                fe_one(zz.x);
                fe_one(zz.y);
            }
            lp_store_aff(rt, 0, lane, zz);
            lp_store_fe(pref, t, lane, acc);
            acc = fmul(acc, fmul(zz.x, zz.y));
        }
        if (a.w == 1) break;                    // no chains: nothing to invert
        __syncwarp();
        sm[tid] = fe_lo(acc);
        sm[128 + tid] = fe_hi(acc);
        __syncthreads();
        if (warp == (turn & 3u)) fold_inverse128(sm);
        turn++;
        __syncthreads();
        fe inv;
        fe_from_quads(inv, sm[tid], sm[128 + tid]);
        fe zi, zzi;                             // ZZ^-1 and ZZZ^-1 of the entry
        for (int t = kw - 1; t >= 0; t--) {
            const int dg = t * a.dpc + place, len = chain_len(dg, more);
            if (len < 2) continue;
            const uint4* rt = rat + (size_t)t * (size_t)(1 << (a.w < 4 ? a.w : 4)) * 128;
            const bool began = cross && lower(dg) && t + 1 < kw;   // the upper digit went on from here
            if (!began) {
                aff zz;
                fe pr;
                lp_load_aff(zz, rt, 0, lane);
                lp_load_fe(pr, pref, t, lane);
                const fe i5 = fmul(inv, pr);
                inv = fmul(inv, fmul(zz.x, zz.y));
                zi = fmul(i5, zz.y);
                zzi = fmul(i5, zz.x);
            }
            int o;
            uint4* hb = half_at(dg, o);
            for (int e = len - 1; e >= 1; e--) {
                const bool last = more && e == len - 1;
                uint4* row = chain_row(dg, t, e, len, more, hb, o);
                if (!began && (more ? e == len - 2 : e == len - 1)) {
                    // From here on the products with X and Y are standard.
                    fe_from_mont(zi, zi);
                    fe_from_mont(zzi, zzi);
                }
                aff Q, r;
                lp_load_aff(Q, row, 0, lane);
                Q.x = fmul(Q.x, zi);
                Q.y = fmul(Q.y, zzi);
                if (failed) {
                    if ((failed >> t) & 1u) {
                        aff B;
                        lp_load_aff(B, hb, 1 << o, lane);
                        aff_to_mont(B);
                        if (cross && upper(dg)) {
                            aff A;
                            int ol;
                            uint4* lb = half_at(dg - 1, ol);
                            lp_load_aff(A, lb, 1 << ol, lane);
                            aff_to_mont(A);
                            load_aff(B, Bc, nl, (size_t)(c0 + t) * a.l + j);
                            aff_to_mont(B);
                            Q = small_sum(A, B, (uint32_t)e);
                        } else {
                            Q = small_multiple(B, last ? 16u : (uint32_t)(e + 1));
                        }
                        if (!last) aff_from_mont(Q);
                    }
                }
                if (last) {
                    lp_store_aff(row, 0, lane, Q);
                    if (upper(dg)) {
                        aff_from_mont(Q);
                        row = spare(dg);
                    }
                }
                if (!last || upper(dg)) {
                    fe_canon(Q.x, Q.x);
                    fe_canon(Q.y, Q.y);
                    if ((atinf >> t) & 1u) {
                        fe_zero(Q.x);
                        fe_zero(Q.y);
                    }
                    lp_store_aff(row, 0, lane, Q);
                }
                lp_load_aff(r, rt, e, lane);
                zi = fmul(zi, r.x);
                zzi = fmul(zzi, r.y);
            }
            if (began && ((atinf >> (t + 1)) & 1u)) {
                // v infinity + 8 P0.
                aff Q;
                lp_load_aff(Q, hb, 8 << o, lane);
                int ou;
                uint4* ub = half_at(dg + 1, ou);
                for (int v = 1; v < 16; v++) lp_store_aff(chain_row(dg + 1, t + 1, v, 16, more, ub, ou), 0, lane, Q);
            }
        }
    }

    // 2. The halves' tables, one more digit of each half a round.
    const int nlow = a.ns, nhigh = a.nd - a.ns;
    for (int r = 1; r < nlow || r < nhigh; r++) {
        // Low half: digit r at bit oL; high half: digit ns + r at bit oH.
        // Pair index i of a half: (v - 1) 2^o + g; (v - 1) 8 + (g - 1) of
        // signed pairs, v 8 + (g - 1) across two columns (of which the upper
        // one may be missing: v = 0).
        int o[2] = {0, 0}, n[2] = {0, 0};
#pragma unroll
        for (int hf = 0; hf < 2; hf++) {
            const int dg = hf ? a.ns + r : r;
            if (r < (hf ? nhigh : nlow) && dg / a.dpc < kw) {
                half_at(dg, o[hf]);
                n[hf] = r == 1 && sp[hf] ? 8 << digit_bits(a, dg) : ((1 << digit_bits(a, dg)) - 1) << o[hf];
            } else if (cross && r == 1 && sp[hf] && dg - 1 < kw) {
                n[hf] = 8;
            }
        }
        auto pick = [&](int i, int& g, int& v, uint4*& tab, const uint4*& pa) -> unsigned {
            const int hf = i >= n[0];
            const int cnt = hf ? n[1] : n[0];
            if (hf) i -= n[0];
            tab = hf ? high : half;
            if (r == 1 && (hf ? sp[1] : sp[0])) {
                const int top = cnt >> 3;
                g = (i & 7) + 1;
                if (cross) {
                    v = (i >> 3) * 16 + 8;
                    pa = tab + (size_t)v * 128;
                    return (g < 8 ? 1u : 0u) | (v > 8 ? 2u : 0u);
                }
                v = (i >> 3) + 1;
                pa = v == top ? (hf ? half : high) : tab + (size_t)v * (16 * 128);
                const unsigned want = (v < top ? 1u : 0u) | (g < 8 ? 2u : 0u);
                v *= 16;
                return want;
            }
            const int ob = hf ? o[1] : o[0];
            g = i & ((1 << ob) - 1);
            v = ((i >> ob) + 1) << ob;
            pa = tab + (size_t)v * 128;
            return g != 0;
        };
        auto pair = [&](int i, const uint4*& pa, const uint4*& pb) -> unsigned {
            int g, v;
            uint4* tab;
            const unsigned want = pick(i, g, v, tab, pa);
            pa += lane;
            pb = tab + (size_t)g * 128 + lane;
            return want;
        };
        auto put = [&](int i, int minus, const aff& S) {
            int g, v;
            uint4* tab;
            const uint4* pa;
            pick(i, g, v, tab, pa);
            lp_store_aff(tab, minus ? v - g : v + g, lane, S);
        };
        affine_batch<SIGNED, PAIRS == 1>(n[0] + n[1], pair, put, pref, sm, turn++);
    }

    // 3. The strip's entries.
    const size_t tbase = (size_t)s_local * a.emax;
    const uint32_t lanepos = (uint32_t)c * a.lp + j;
    auto store_table = [&](int e, const aff& q) {
        store_aff(a.table, a.table_points, (tbase + e) * (2u * a.lp) + lanepos, q);
    };
    const uint32_t lmask = (1u << a.hl) - 1u;
    if (two) {
        // The entry of each code, then the pairs that hold one: v, g and the
        // entries of z + g and z - g (255: none), z = 16 v, or 16 v + 8 across two
        // columns.
        uint8_t* rank = (uint8_t*)(sm + 256 + warp * 48);
        uint32_t* list = (uint32_t*)(rank + 256);
        ((uint2*)rank)[lane] = make_uint2(0xffffffffu, 0xffffffffu);
        __syncwarp();
        for (int e = lane; e < E; e += 32) rank[codes[e] & 255] = (uint8_t)e;
        __syncwarp();
        const int top = 1 << a.hh;
        int cnt = 0;
        for (int b = 0; b < top * 8; b += 32) {
            const int i = b + (int)lane, v = (i >> 3) + (cross ? 0 : 1), g = (i & 7) + 1;
            const int z = 16 * v + (cross ? 8 : 0);
            const uint32_t plus = (cross ? g < 8 : v < top) ? rank[(z + g) & 255] : 255u;
            const uint32_t minus = (cross ? v > 0 : g < 8) ? rank[(z - g) & 255] : 255u;
            const bool any = (plus & minus) != 255u;
            const unsigned mask = __ballot_sync(0xffffffffu, any);
            if (any) list[cnt + __popc(mask & ((1u << lane) - 1u))] = (uint32_t)v | (uint32_t)g << 8 | plus << 16 | minus << 24;
            cnt += __popc(mask);
        }
        __syncwarp();
        affine_batch<true, PAIRS == 1>(
            cnt,
            [&](int i, const uint4*& pa, const uint4*& pb) -> unsigned {
                const uint32_t x = list[i];
                const int v = x & 255;
                pa = (v == top ? half : cross && v == 0 ? half + 8 * 128 : high + (size_t)v * 128) + lane;
                pb = half + (size_t)((x >> 8) & 255u) * 128 + lane;
                return (((x >> 16) & 255u) != 255u ? 1u : 0u) | ((x >> 24) != 255u ? 2u : 0u);
            },
            [&](int i, int minus, const aff& S) {
                store_table((int)(minus ? list[i] >> 24 : (list[i] >> 16) & 255u), S);
            },
            pref, sm, turn);
    } else if (a.nd > 1) {
        affine_batch<false, PAIRS == 1>(
            E,
            [&](int e, const uint4*& pa, const uint4*& pb) -> unsigned {
                const uint32_t code = codes[e];
                pa = half + (size_t)(code & lmask) * 128 + lane;
                pb = high + (size_t)(code >> a.hl) * 128 + lane;
                return (code & lmask) && (code >> a.hl);
            },
            [&](int e, int, const aff& S) { store_table(e, S); },
            pref, sm, turn);
    }
    for (int e = 0; e < E; e++) {
        const uint32_t code = codes[e], u = code & lmask;
        if (two && cross ? (code >> a.hl ? u != 8 : u > 8) : u && ((code >> a.hl) || (two && u > 8))) continue;
        aff Q;
        lp_load_aff(Q, u && !(two && cross && (code >> a.hl)) ? half + (size_t)u * 128 : high + (size_t)(code >> a.hl) * 128, 0, lane);
        store_table(e, Q);
    }
}

// What a strip's table costs by chains of prefix sums (table_item) beyond its cost by
// digits. The digits' chains and the halves' tables are made whatever the
// strip holds, so strips of few distinct codes (sparse columns, columns of few
// values) are cheaper by chains, which cost what they hold. In tenths of the
// microseconds that one of 608 warp schedulers takes, fitted to 840 table times (w = 1
// to 16, strips of 1 to 6 columns, densities 0.003 to 1, columns of 1, 2 and 4 values);
// the chains count 1.05 times, so that close calls go by digits. Tables of 256 columns of 256
// (us) by digits and by chains: w = 8 with 3.6 values a column 841 and 659, w = 12
// with 50 3833 and 3224, with 101 4383 and 4415, w = 16 with 3.2 5477 and 1214.
__device__ __forceinline__ int strip_excess(int entries, const uint16_t* len, int columns, int w, const FewArgs& f) {
    static_assert(NLEV == 4, "a column's lengths are read as one ushort4");
    int chains = 0;
#pragma unroll 1
    for (int t = 0; t < columns; t++, len += NLEV) {
        const ushort4 q = *(const ushort4*)len;
        if (q.x) chains += 33 * (q.x - 1) + 36 * (q.y + q.z - 2) + 19 * (w - 1) * q.w + (w > 1 ? 144 : 0);
    }
    // f.fixed counts the chains' own constant, which an empty strip does not have.
    return entries > 0 ? chains - f.entry * entries - f.fixed : -(f.fixed + 184 + 80 * columns);
}

// Whether a pass's tables cost less by chains than by digits: the sum over its
// strips, so that one of the two kernels builds them all (block by block, each kernel
// took the time of a whole wave: 1024 x 256 x 256 at w = 16 with 21 values a column 7.3 ms,
// 4.5 as it is). All 128 threads of the block call; sm: 2 uint4.
static __device__ __noinline__ bool pass_few(const int32_t* nent, const uint16_t* col_len, int s0, int strips, int n, int k,
                                             int w, int emax, FewArgs f, uint4* sm) {
    long long sum = 0;
#pragma unroll 1
    for (int x = (int)threadIdx.x; x < strips; x += 128) {
        const int s = s0 + x, c0 = s * k, E = nent[s];
        sum += strip_excess(E < emax ? E : emax, col_len + (size_t)c0 * NLEV, c0 + k <= n ? k : n - c0, w, f);
    }
    __syncwarp();
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
    long long* part = (long long*)sm;
    if ((threadIdx.x & 31u) == 0) part[threadIdx.x >> 5] = sum;
    __syncthreads();
    sum = part[0] + part[1] + part[2] + part[3];
    __syncthreads();
    return sum < 0;
}

// The digits and halves of a strip code, and whether the digit build takes
// the tables of this layout.
inline bool digit_split(const Layout& L, TableArgs& a, FewArgs& few) {
    a.dpc = (L.w + 3) / 4;
    a.nd = L.k * a.dpc;
    a.ns = 1;
    a.hl = L.w;
    a.hh = 0;
    auto bits = [&](int d) { const int r = L.w - 4 * (d % a.dpc); return r < 4 ? r : 4; };
    long long best = a.nd == 1 ? 1LL << L.w : -1;
    int lo = 0;
    for (int x = 1; x < a.nd; x++) {
        lo += bits(x - 1);
        const int hi = L.w * L.k - lo;
        const long long size = (1LL << lo) + (1LL << hi);
        if (best < 0 || size < best) { best = size; a.ns = x; a.hl = lo; a.hh = hi; }
    }
    // The digit build takes every layout whose scratch holds its halves: up to
    // about 3.5 half entries for each entry of the strip. Table times (ms) by chains
    // and by digits, 256 columns of 256: w = 16 with 160 rows (halves 512) 8.99 and
    // 7.46, w = 12 with 128 rows (halves 272) 4.90 and 4.64, with 96 rows 4.21 and
    // 4.34; 200 x 64 at w = 14 with 100 rows (halves 320) 1.81 and 1.55; 256 x 64 at w
    // = 8 with 12 rows (halves 32) 0.332 and 0.289; one digit, 128 x 1 at w = 4 with
    // 10 rows 135 and 118 us.
    a.w = L.w;
    const bool any = (a.nd == 2 && signed_pair(a, 0, 2)) || signed_pair(a, 0, a.ns) || signed_pair(a, a.ns, a.nd);
    a.pairs = !any ? 0 : a.dpc > 1 ? 1 : 2;
    // Costs for strip_excess: the steps of the digits' chains, the halves' sums and
    // the inversions of a strip, its columns, and for each entry its sum by
    // digits less the sums of its parts by chains.
    const bool two = a.nd == 2 && signed_pair(a, 0, 2);
    const bool sp[2] = {two || signed_pair(a, 0, a.ns), signed_pair(a, a.ns, a.nd)};
    int steps = 0, digit_entries = 0;
    for (int d = 0; d < a.nd; d++) {
        const bool more = d % a.dpc + 1 < a.dpc;
        const bool lower = (sp[0] && d == 0) || (sp[1] && d == a.ns);
        const bool upper = (sp[0] && d == 1) || (sp[1] && d == a.ns + 1);
        const int all = 1 << digit_bits(a, d);
        steps += (lower ? (a.dpc == 1 ? 8 : 9) : all - (more || upper ? 0 : 1)) - 1;
        digit_entries += all;
    }
    const int sums = a.nd > 1 ? (1 << a.hl) + (1 << a.hh) - digit_entries : 0;
    const int rounds = (a.ns > a.nd - a.ns ? a.ns : a.nd - a.ns) - 1;
    const int inversions = (L.w > 1 ? a.dpc : 0) + rounds + (a.nd > 1 ? 1 : 0);
    few.fixed = (int)(38.8 * steps + 14.0 * (sums > 0 ? sums : 0) + 77.1 * inversions + 8.4 * L.k - 184.0);
    few.entry = (int)((a.nd > 1 ? 13.9 : 0.0) - (L.k > 1 ? 34.0 * (L.k * (1.0 - 1.0 / (1 << L.w)) - 1.0) : 0.0));
    const bool fits = digit_scratch(L.w, L.k, a.dpc, a.hl, a.hh, L.n1max, L.l2max, L.emax).total <= L.item_u4;
    // A second launch costs a small call 5 to 7 us (10 x 128 x 1 at w = 4 175 and
    // 182, 512 x 1 x 16384 814 and 821). There the time is the latency of one strip's
    // build, and that of the digits is short with one place of digits and no round
    // between it and the entries: 98 us where a nearly empty strip takes 44 by chains.
    few.either = fits;
    few.small = fits && (L.w == 1 || inversions > 2);
    return fits;
}

struct GatherArgs {
    int m, l, lp, span, nq, emax;
    int s0, nstrips_chunk;
    bool first;
    const uint4* table;
    size_t table_points;
    uint4* ctC;            // Jacobian ciphertext matrix m x l
    int parts;             // warps per output splitting the chunk's strips (1: accumulate into ctC)
    uint4* partial;        // parts > 1: Jacobian partial sums, parts matrices laid out like ctC
};

// Accumulation of one warp item (output row i, component c, 32 columns) over
// the strips of a chunk.  CG = true reads tables and accumulators through L2
// only (ld.global.cg): in the persistent batched kernel they were written by
// other SMs during the same launch.
template <bool CG>
__device__ __forceinline__ void gather_item(const GatherArgs& a, const PlanPtrs& P, long long gw) {
    // Rows innermost: the warps resident at a time cover every row of a few
    // column blocks, so each strip's table region is fetched once per block
    // while those warps walk the strips together.
    // With parts > 1 (small outputs), warp gw / (m nq) takes part p of
    // the chunk's strips and leaves its partial sum for combine_kernel.
    const unsigned lane = threadIdx.x & 31u;
    const long long per_part = (long long)a.m * a.nq;
    const int part = (int)(gw / per_part);
    gw %= per_part;
    const int i = (int)(gw % a.m);
    int c, j;
    const bool own = lane_chain((int)(gw / a.m), a.span, a.l, c, j);
    const size_t ml = (size_t)a.m * a.l;
    uint4* Cc = (a.parts > 1 ? a.partial + (size_t)part * 12 * ml : a.ctC) + (size_t)c * 6 * ml;
    // The running sum is kept as (X, Y, Z^2, Z^3): its mixed additions then
    // cost 8M + 2S, and Z itself is rebuilt once at the end.  The table
    // entries are standard, so Z^2 and Z^3 carry the factor R (ec.cuh).
    jacz acc;
    if (a.first || a.parts > 1) {
        jacz_set_inf(acc);
    } else {
        jac prev;
        if (CG) load_jac_cg(prev, Cc, ml, (size_t)i * a.l + j);
        else load_jac(prev, Cc, ml, (size_t)i * a.l + j);
        jac_to_mont(prev);
        jacz_from_jac(acc, prev);
        jacz_add_R(acc);
    }
    const uint16_t* rk = P.rank + (size_t)a.s0 * a.m + i;
    aff T;
    const int s_lo = (int)((long long)a.nstrips_chunk * part / a.parts);
    const int s_hi = (int)((long long)a.nstrips_chunk * (part + 1) / a.parts);
    const uint32_t lanepos = (uint32_t)c * a.lp + j;
    auto entry = [&](aff& Q, int sl, uint16_t code) {
        const size_t ti = ((size_t)sl * a.emax + code) * (2u * a.lp) + lanepos;
        if (CG) load_aff_cg(Q, a.table, a.table_points, ti);
        else load_aff(Q, a.table, a.table_points, ti);
    };
    int sl = s_lo;
#ifndef PCMM_DEBUG_BOUNDS
    if (a.first || a.parts > 1) {
        // The first entry starts the sum; if no second one follows, the sum is
        // that entry and leaves as it is, with Z = 1 (0 at infinity).
        while (sl < s_hi && rk[(size_t)sl * a.m] == NO_RANK) sl++;
        if (sl < s_hi) {
            entry(T, sl, rk[(size_t)sl * a.m]);
            sl++;
            while (sl < s_hi && rk[(size_t)sl * a.m] == NO_RANK) sl++;
            if (sl == s_hi) {
                jac out;
                out.X = T.x;
                out.Y = T.y;
                fe_zero(out.Z);
                out.Z.v[0] = aff_is_inf(T) ? 0u : 1u;
                if (a.parts > 1) jac_to_mont(out);
                if (own) store_jac(Cc, ml, (size_t)i * a.l + j, out);
                return;
            }
            if (!aff_is_inf(T)) {
                fe_to_mont(acc.X, T.x);
                fe_to_mont(acc.Y, T.y);
                fe_set_R2(acc.ZZ);
                fe_set_R2(acc.ZZZ);
            }
        }
    }
#endif
    for (; sl < s_hi; sl++) {
        const uint16_t code = rk[(size_t)sl * a.m];
        if (code == NO_RANK) continue;
#ifdef PCMM_DEBUG_BOUNDS
        if (code >= P.nent[a.s0 + sl]) {   // a rank past the strip's table
            atomicOr(P.status, DEV_ERR_BOUNDS);
            continue;
        }
#endif
        entry(T, sl, code);
        jacz_madd_t<PCMM_GATHER_INLINE, true>(acc, T);
    }
    if (own) {
        jac out;
        jacz_drop_R(acc);
        jac_from_jacz(out, acc);
        if (a.parts == 1) jac_from_mont(out);   // partial sums stay in the Montgomery domain
        store_jac(Cc, ml, (size_t)i * a.l + j, out);
    }
}

// Expected number of distinct non-zero values when m values are drawn
// uniformly from [0, 2^bits).
inline double expected_distinct_nonzero(int m, int bits) {
    const double V = ldexp(1.0, bits);
    const double present = V * (1.0 - pow(1.0 - 1.0 / V, (double)m));
    const double zero = 1.0 - pow(1.0 - 1.0 / V, (double)m);
    double d = present - zero;
    return d < 0 ? 0 : d;
}

// Modelled time of one PC-MM in field-multiplication units (a squaring
// counted as one) for strip width k.  Gather: one mixed addition (11) per
// row, strip and ciphertext chain with a non-zero code.  Table build: per
// column the level-1 prefix sums (mixed additions) and the level-N
// double-and-add (about 2w operations of 8); the normalisation (5 per entry,
// along the chain's ratios) of the strip table (k = 1) or of the column
// tables (k > 1); for k > 1 the
// tuple entries by affine additions (6 per further non-zero component).  The
// table work is weighted by 1.9, fitted to GB300 timings of the
// 1024 x 1024 x 256 product for every w and k with tables by chains, which
// issue their multiplications less efficiently than the gather.  Of tables by digits,
// which most are now, it says too much: at w = 1 seven columns take 7.9 ms, the
// chosen six 8.7.
inline double model_cost(int m, int n, int l, int w, int k) {
    const double MADD = 11, DBL = 8, NORM = 5, AFF = 6, TABLE_WEIGHT = 1.9;
    const double chains = 2.0 * l;
    const int nstrips = (n + k - 1) / k;
    const double n1 = expected_distinct_nonzero(m, w);
    const double E = k == 1 ? n1 : expected_distinct_nonzero(m, w * k);
    const double nz1 = 1.0 - ldexp(1.0, -w);
    const double col = n * chains * (n1 * MADD + 2.0 * w * DBL);
    const double norm = (k == 1 ? nstrips * E : n * n1) * chains * NORM;
    const double extra = k * nz1 - 1.0;
    const double tup = k > 1 ? nstrips * chains * E * (extra > 0 ? extra : 0.0) * AFF : 0.0;
    const double gather = (double)m * chains * nstrips * (1.0 - ldexp(1.0, -w * k)) * MADD;
    return gather + TABLE_WEIGHT * (col + norm + tup);
}


}  // namespace cussen
}  // namespace pcmm

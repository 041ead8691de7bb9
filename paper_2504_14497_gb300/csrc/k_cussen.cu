// Cussen's compression-reconstruction PC-MM (Algorithms 2 and 3) on sm_103a.
//
// Three kernels per pass over a chunk of column strips of A:
//
//  plan   (once per call, one CTA per strip; plaintext only)
//         For every column: level 1 = the distinct non-zero values sorted
//         ascending; for w < N its consecutive differences are sorted and
//         deduplicated into level w + 1, recording for every element of
//         level w its position in level w + 1 (the tracking pointers);
//         level N keeps its values.  A zero contributes the identity and is
//         dropped from every level.  For the strip: the code of every row
//         (its k entries packed w bits apiece), the sorted list of distinct
//         non-zero codes, and each row's rank in that list (0xFFFF for 0).
//  table  (one warp per strip and 32 ciphertext chains, lane_span)
//         Level N: the compressed values times the ciphertext point B_c^(kj)
//         by double-and-add (the ECSMs of Algorithm 3).  Levels N-1..1: each
//         element of level w is the entry of level w + 1 its tracking pointer
//         names, and a running prefix sum of points turns the multiples of
//         differences into the multiples of the level's sorted values.
//         Level 1 is the per-column table v B_c^(kj) over the distinct values
//         v of the column, a chain of mixed additions in (X, Y, Z^2, Z^3).
//         For strips of k > 1 columns, each distinct k-tuple adds its
//         columns' entries (affine additions, one shared inversion per
//         round).  The tables are normalised to affine coordinates in the
//         same kernel: level 2 by Montgomery's simultaneous inversion, the
//         level-1 chains by walking Z^-2 and Z^-3 back along the factors the
//         chain multiplied them by; the inversion is shared by the lanes of
//         a warp and, when the block's four warps follow one strip's plan,
//         by the whole block.  Wherever the scratch holds the tables of a
//         code's halves (most strips) and the pass's strips hold more than a
//         few codes (pass_few) the same entries are built digit by digit
//         in affine coordinates instead (table_block), from the values that
//         the compressed levels expand to.
//  gather (one warp per output row i and 32 ciphertext chains)
//         C_ij += T_s[rank_s(i)] for every strip s: the "un-sort and re-insert
//         duplicates" step of Algorithm 2 fused with the accumulation of
//         Algorithm 3, one mixed addition per strip into an accumulator in
//         (X, Y, Z^2, Z^3).  The rank is the same for the whole warp (one
//         broadcast load); the 32 lanes' table entries are adjacent, so the
//         four 16-byte loads per point are coalesced.  Small outputs split
//         their strips over several warps (combine_kernel adds the parts).
#include <cuda_runtime.h>

#include "cussen_core.cuh"
#include "profiler.cuh"

using namespace pcmm;
using namespace pcmm::cussen;

// Minimum resident blocks per SM requested from the compiler (its register
// budget).  Measured on GB300: the gather is pipe-bound and wants the
// registers (w = 4, 1024 x 1024 x 256: 23.9 ms at 4 blocks, 25.1 at 5); the
// chains of the table build wait on their scratch and spill traffic, so more
// resident warps pay despite more spilling (at the multiplication of that
// time, 46.3 ms a step of four widths at 4 blocks, 45.0 at 7, 47.3 at 8).
// Build-time tunables.
#ifndef PCMM_GATHER_MINBLOCKS
#define PCMM_GATHER_MINBLOCKS 4
#endif
#ifndef PCMM_TABLE_MINBLOCKS
#define PCMM_TABLE_MINBLOCKS 7
#endif

namespace {

template <class TA>
__global__ void __launch_bounds__(PLAN_THREADS) plan_kernel(const TA* __restrict__ A, int m, int n, int w,
                                                            int k, PlanPtrs P) {
    plan_strip(A, m, n, w, k, P, blockIdx.x);
}

template <int BLOCKS>
__global__ void __launch_bounds__(128, BLOCKS) table_kernel(TableArgs a, PlanPtrs P, FewArgs f) {
    const long long item = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nitems = (long long)a.nstrips_chunk * a.nq;
    if (f.either) {
        __shared__ uint4 sm[2];
        if (!pass_few(P.nent, P.col_len, a.s0, a.nstrips_chunk, a.n, a.k, a.w, a.emax, f, sm)) return;
    }
    if (item >= nitems) return;
    table_item(a, P, item, a.scratch + (size_t)item * a.item_u4);
}

// table_kernel by digits (table_block): two thirds of the multiplications and
// hardly any spills, so it is faster than the chains and wants registers more
// than warps. Table times of 1024 x 1024 x 256 (ms), chains and digits at 3, 4,
// 5 and 6 blocks per SM: w = 8 21.5 / 10.9, 10.4, 10.4, 10.9; w = 4 8.3 / 5.5,
// 5.3, 5.7, 6.0; 512 x 512 x 256, w = 16: 36.6 / 24.0, 22.1, 23.1, 25.4 (before canonical
// forms moved behind a test, which took 2% off at 4).
#ifndef PCMM_DIGIT_MINBLOCKS
#define PCMM_DIGIT_MINBLOCKS 4
#endif
// Up to two blocks per SM the tables are bound by the latency of one warp per
// scheduler or two, and are built by copies of the kernels that the register file
// holds twice per SM (no spills). Table of 10 x 128 x 1 (w = 4) 119 -> 104 us, 512 x
// 1 x 16384 158 -> 141 us, by chains (10 x 160 x 15, w = 7) 243 -> 211 us; with up to four
// blocks per SM the copies lose (256 x 784 x 64 1.01 -> 1.35 ms).
constexpr unsigned FEW_BLOCKS = 2 * 152;
template <int PAIRS, int BLOCKS>
__global__ void __launch_bounds__(128, BLOCKS) digit_table_kernel(TableArgs a, PlanPtrs P, FewArgs f) {
    __shared__ uint4 sm[DIGIT_SHARED_U4];
    const long long item = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const bool valid = item < (long long)a.nstrips_chunk * a.nq;
    // As a jump out of the kernel, a return cost the tables of w = 16 3% (spills).
    if (f.either && pass_few(P.nent, P.col_len, a.s0, a.nstrips_chunk, a.n, a.k, a.w, a.emax, f, sm)) asm volatile("exit;");
    uint4* scratch = a.scratch + (valid ? (size_t)item : (size_t)0) * a.item_u4;
    table_block<PAIRS>(a, P, item, valid, scratch, sm);
}

__global__ void __launch_bounds__(128, PCMM_GATHER_MINBLOCKS) gather_kernel(GatherArgs a, PlanPtrs P) {
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (gw >= (long long)a.m * a.nq * a.parts) return;
    gather_item<false>(a, P, gw);
}

// Adds the parts partial sums (Montgomery domain) of every output point (and,
// after the first pass, the accumulated value) into ctC: G = 2^logG lanes a point
// add every G-th part each, and their sums as a tree. One lane a point waits for
// its chain of additions: with as many lanes as give two warps per scheduler, 66
// x 750 x 14 (w = 7, 32 parts) takes 40 us for 162, 29 x 926 x 86 (w = 4) 74 for
// 172; with four warps 76 and 66.
__global__ void __launch_bounds__(128) combine_kernel(const uint4* __restrict__ partial, int parts, int logG,
                                                      uint4* __restrict__ ctC, size_t ml, bool first) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int G = 1 << logG, p = (int)t & (G - 1);
    const bool valid = (t >> logG) < 2 * ml;
    const size_t o = valid ? t >> logG : 0;
    const size_t c = o >= ml, idx = o - c * ml;
    uint4* Cc = ctC + c * 6 * ml;
    jac acc;
    jac_set_inf(acc);
    for (int x = p; x < parts; x += G) {
        jac Q;
        load_jac(Q, partial + (size_t)x * 12 * ml + c * 6 * ml, ml, idx);
        jac_add(acc, Q);
    }
    __syncwarp();
    for (int d = G / 2; d >= 1; d >>= 1) {
        jac Q;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            Q.X.v[i] = __shfl_down_sync(0xffffffffu, acc.X.v[i], d);
            Q.Y.v[i] = __shfl_down_sync(0xffffffffu, acc.Y.v[i], d);
            Q.Z.v[i] = __shfl_down_sync(0xffffffffu, acc.Z.v[i], d);
        }
        if (p < d) jac_add(acc, Q);
        __syncwarp();
    }
    if (!valid || p) return;
    if (!first) {
        jac prev;
        load_jac(prev, Cc, ml, idx);
        jac_to_mont(prev);
        jac_add(acc, prev);
    }
    jac_from_mont(acc);
    store_jac(Cc, ml, idx, acc);
}

// Gather of a product of one strip: every output is its row's table entry (Z
// = 1) or infinity, a copy bound by memory. One warp per row and 32 chains. At 512 x
// 1 x 16384 (w = 4) it takes 241 us, where gather_kernel at its 128 registers keeps
// too few loads in flight (514 us).
__global__ void __launch_bounds__(128) gather_copy_kernel(GatherArgs a, PlanPtrs P) {
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (gw >= (long long)a.m * a.nq) return;
    const int i = (int)(gw % a.m);
    int c, j;
    if (!lane_chain((int)(gw / a.m), a.span, a.l, c, j)) return;
    const size_t ml = (size_t)a.m * a.l;
    aff T;
    fe_zero(T.x);
    fe_zero(T.y);
    const uint16_t code = P.rank[(size_t)a.s0 * a.m + i];
    if (code != NO_RANK) {
#ifdef PCMM_DEBUG_BOUNDS
        if (code >= P.nent[a.s0]) {   // a rank past the strip's table
            atomicOr(P.status, DEV_ERR_BOUNDS);
            return;
        }
#endif
        load_aff(T, a.table, a.table_points, ((size_t)code * 2 + c) * a.lp + j);
    }
    jac out;
    out.X = T.x;
    out.Y = T.y;
    fe_zero(out.Z);
    out.Z.v[0] = aff_is_inf(T) ? 0u : 1u;
    store_jac(a.ctC + (size_t)c * 6 * ml, ml, (size_t)i * a.l + j, out);
}

}  // namespace

extern "C" int pcmm_cussen_choose_k(int m, int n, int l, int w) {
    if (m < 1 || n < 1 || l < 1 || w < 1 || w > PCMM_MAX_W16) return 0;
    // A wider strip must win by 3%: its tables and scratch grow with 2^(w k).
    int best = 1;
    double bc = model_cost(m, n, l, w, 1);
    for (int k = 2; w * k <= PCMM_MAX_WK && k <= n; k++) {
        double c = model_cost(m, n, l, w, k);
        if (c < 0.97 * bc) { bc = c; best = k; }
    }
    return best;
}

// Table items (warps, counted without packing) per pass come in whole waves of
// the chains' table kernel on a 152-SM GB300 (PCMM_TABLE_MINBLOCKS blocks of 4 warps
// per SM): four waves when one pass's scratch and tables fit in PASS_BYTES_CAP, else
// as many whole waves as fit, at least one.  With chains, whole-wave passes
// measured 3 ms per headline step faster than passes of 4096 items (at 4 blocks
// per SM).  The digit kernel's waves are of 2432 items and its scratch is smaller, so
// its last wave is partly empty; the sizes of workspaces follow from this rule.
#ifndef PCMM_TARGET_WAVES
#define PCMM_TARGET_WAVES 4
#endif
static const size_t WAVE_ITEMS = 152 * PCMM_TABLE_MINBLOCKS * 4;
static const size_t TARGET_WAVES = PCMM_TARGET_WAVES;
static const size_t PASS_BYTES_CAP = (size_t)16 << 30;

namespace {
size_t default_strips(const Layout& L);
}

namespace {

template <class TA>
pcmm_status launch_plan(const Layout& L, const TA* A, const PlanPtrs& P, cudaStream_t st) {
    if (cudaMemsetAsync(P.status, 0, 4, st) != cudaSuccess) return PCMM_ECUDA;
    {
        ProfScope ps(KID_PLAN, st);
        plan_kernel<TA><<<L.nstrips, PLAN_THREADS, 0, st>>>(A, L.m, L.n, L.w, L.k, P);
    }
    PCMM_CUDA_CHECK_LAUNCH();
    return PCMM_OK;
}

// Warps per output for the gather of a pass of S strips: when the outputs
// alone give fewer than GATHER_WARPS_TARGET warps (about five waves of the
// gather on 152 SMs; both components' warps counted without packing, up to twice the
// warps there are for l <= 16), each output's strips are split into up to 32 parts of
// at least part_strips strips, and a combine kernel adds the partial sums
// (one full addition per part against at least part_strips mixed additions).
// Parts go down to 4 strips while all of them still leave the 608 schedulers
// with two warps each at most: such a gather takes as long as one part's
// chain, and the tree that adds the parts is short (10 x 128 x 1 at w = 4: 51 +
// 41 us with 8 parts of 16 strips added in a row, 22 + 29 us with 32 of 4).
const long long GATHER_WARPS_TARGET = 12288;
const long long SCHEDULERS = 608;

int part_strips(const Layout& L, size_t S) {
    return (long long)L.m * 2 * L.njb * (long long)(S / 4) <= 2 * SCHEDULERS ? 4 : 16;
}

int gather_parts(const Layout& L, size_t S, int least) {
    const long long warps = (long long)L.m * 2 * L.njb;
    if (warps >= GATHER_WARPS_TARGET) return 1;
    long long parts = (GATHER_WARPS_TARGET + warps - 1) / warps;
    const long long by_strips = (long long)S / least;
    if (parts > by_strips) parts = by_strips;
    if (parts > 32) parts = 32;
    return parts < 1 ? 1 : (int)parts;
}

int gather_parts(const Layout& L, size_t S) { return gather_parts(L, S, part_strips(L, S)); }

size_t partial_bytes(const Layout& L, int parts) {
    return parts > 1 ? align256((size_t)parts * 2 * L.m * L.l * 96) : 0;
}

// Table build and gather over chunks of S strips, using the scratch area at
// `chunk` (S * per_strip_bytes bytes) and, when parts > 1, the partial sums
// at `partial` (partial_bytes(L, parts) bytes).
pcmm_status launch_exec(const Layout& L, const PlanPtrs& P, const uint32_t* ctB, uint32_t* ctC,
                        uint8_t* chunk, size_t S, uint8_t* partial, int parts, cudaStream_t st) {
    uint4* scratch = (uint4*)chunk;
    uint4* table = (uint4*)(chunk + align256(S * L.items_per_strip * L.item_u4 * 16));
    const size_t ml = (size_t)L.m * L.l;
    TableArgs split;
    FewArgs fa;
    const bool digits = digit_split(L, split, fa);
    for (int s0 = 0; s0 < L.nstrips; s0 += (int)S) {
        const int sc = (int)((size_t)(L.nstrips - s0) < S ? (size_t)(L.nstrips - s0) : S);
        TableArgs ta = split;
        ta.ctB = (const uint4*)ctB;
        ta.m = L.m; ta.n = L.n; ta.l = L.l; ta.w = L.w; ta.k = L.k;
        ta.lp = L.lp; ta.span = lane_span(L.l); ta.nq = lane_blocks(L.l); ta.n1max = L.n1max; ta.l2max = L.l2max; ta.emax = L.emax;
        ta.s0 = s0; ta.nstrips_chunk = sc;
        ta.scratch = scratch;
        ta.item_u4 = L.item_u4;
        ta.table = table;
        ta.table_points = S * L.table_points_per_strip;
        // Four consecutive items (one 128-thread block) belong to one strip
        // exactly when a strip has a multiple of 4 items; then every block is
        // full and its warps follow the same plan, and share inversions.
        ta.bshare = (ta.nq % 4) == 0;
        const long long items = (long long)sc * ta.nq;
        const unsigned blocks = (unsigned)((items + 3) / 4);
        const bool few = blocks <= FEW_BLOCKS;
        FewArgs f = fa;
        f.either = few ? fa.small : fa.either;
        if (digits) {
            ProfScope ps(KID_TABLE, st);
            auto* kernel = few ? digit_table_kernel<0, 1> : digit_table_kernel<0, PCMM_DIGIT_MINBLOCKS>;
            if (split.pairs == 1) kernel = few ? digit_table_kernel<1, 1> : digit_table_kernel<1, PCMM_DIGIT_MINBLOCKS>;
            if (split.pairs == 2) kernel = few ? digit_table_kernel<2, 1> : digit_table_kernel<2, PCMM_DIGIT_MINBLOCKS>;
            kernel<<<blocks, 128, 0, st>>>(ta, P, f);
            PCMM_CUDA_CHECK_LAUNCH();
        }
        if (!digits || f.either) {   // which of the two builds the tables is decided on the device
            ProfScope ps(KID_TABLE, st);
            auto* kernel = few ? table_kernel<1> : table_kernel<PCMM_TABLE_MINBLOCKS>;
            kernel<<<blocks, 128, 0, st>>>(ta, P, f);
        }
        PCMM_CUDA_CHECK_LAUNCH();
        GatherArgs ga;
        ga.m = L.m; ga.l = L.l; ga.lp = L.lp; ga.span = ta.span; ga.nq = ta.nq; ga.emax = L.emax;
        ga.s0 = s0; ga.nstrips_chunk = sc;
        ga.first = (s0 == 0);
        ga.table = table;
        ga.table_points = ta.table_points;
        ga.ctC = (uint4*)ctC;
        // A short last chunk may take fewer parts than the buffer holds.
        int pc = sc / part_strips(L, S);
        pc = pc < 1 ? 1 : pc < parts ? pc : parts;
        ga.parts = pc;
        ga.partial = (uint4*)partial;
        const long long warps = (long long)L.m * ga.nq * pc;
        {
            ProfScope ps(KID_GATHER, st);
            if (ga.first && sc == 1) gather_copy_kernel<<<(unsigned)((warps + 3) / 4), 128, 0, st>>>(ga, P);
            else gather_kernel<<<(unsigned)((warps + 3) / 4), 128, 0, st>>>(ga, P);
        }
        PCMM_CUDA_CHECK_LAUNCH();
        if (pc > 1) {
            ProfScope ps(KID_COMBINE, st);
            int logG = 0;
            while ((1 << logG) < pc && logG < 5 && ((2 * ml) << (logG + 1)) <= (size_t)2 * SCHEDULERS * 32) logG++;
            combine_kernel<<<(unsigned)((((2 * ml) << logG) + 127) / 128), 128, 0, st>>>(
                (const uint4*)partial, pc, logG, (uint4*)ctC, ml, s0 == 0);
        }
        PCMM_CUDA_CHECK_LAUNCH();
    }
    return PCMM_OK;
}

size_t default_strips(const Layout& L) {
    const size_t ips = L.items_per_strip;
    const size_t cap = PASS_BYTES_CAP / L.per_strip_bytes;   // strips within the byte cap
    size_t waves = TARGET_WAVES;
    while (waves > 1 && waves * WAVE_ITEMS / ips > cap) waves--;
    size_t S = waves * WAVE_ITEMS / ips;                      // whole strips within the waves
    if (S > (size_t)L.nstrips) S = L.nstrips;
    return S < 1 ? 1 : S;
}

// Bytes of execution workspace (beyond the plan) the default configuration
// uses: the gather's partial sums, then passes of default_strips strips.
size_t default_exec_bytes(const Layout& L) {
    const size_t S = default_strips(L);
    return partial_bytes(L, gather_parts(L, S)) + S * L.per_strip_bytes;
}

// Splits `avail` bytes of execution workspace into the partial sums (when
// the gather splits its strips) and passes of S strips; the partial sums are
// dropped when both do not fit, and made of parts of at least 16 strips where
// the room of smaller parts would cost passes: 73 x 41 x 63 (w = 1, k = 3) in a
// workspace for its 14 strips and no partial sums took 14 passes, 977 us, with
// parts of 4, and takes one, 111 us, without. False when not even one strip
// fits.
bool exec_space(const Layout& L, size_t avail, size_t& S, int& parts, size_t& pbytes) {
    if (avail < L.per_strip_bytes) return false;
    const size_t S0 = default_strips(L);
    size_t passes = 0;
    for (int least = 16; least >= part_strips(L, S0); least -= 12) {
        int p = gather_parts(L, S0, least);
        size_t pb = partial_bytes(L, p);
        if (p > 1 && avail < pb + L.per_strip_bytes) {
            p = 1;
            pb = 0;
        }
        size_t s = (avail - pb) / L.per_strip_bytes;
        if (s > (size_t)L.nstrips) s = L.nstrips;
        const size_t n = (L.nstrips + s - 1) / s;
        if (passes && n > passes) break;
        passes = n;
        S = s;
        parts = p;
        pbytes = pb;
    }
    const int ps = gather_parts(L, S);
    if (ps < parts) parts = ps;
    return true;
}

}  // namespace

namespace {

template <class TA>
pcmm_status cussen_call(const TA* A, int m, int n, int w, const uint32_t* ctB, int l, uint32_t* ctC, int k,
                        void* ws, size_t ws_bytes, pcmm_stream_t stream) {
    if (!A || !ctB || !ctC || !ws || ((uintptr_t)ws & 255u)) return PCMM_EINVAL;
    if (m < 1 || n < 1 || l < 1 || w < 1 || w > 8 * (int)sizeof(TA)) return PCMM_EINVAL;
    if (k == 0) k = pcmm_cussen_choose_k(m, n, l, w);
    Layout L;
    if (!make_layout(L, m, n, l, w, k)) return PCMM_EINVAL;
    if (ws_bytes < L.plan_bytes) return PCMM_ENOMEM;
    size_t S, pbytes;
    int parts;
    if (!exec_space(L, ws_bytes - L.plan_bytes, S, parts, pbytes)) return PCMM_ENOMEM;
    cudaStream_t st = (cudaStream_t)stream;
    PlanPtrs P = plan_ptrs(L, ws);
    pcmm_status rc = launch_plan(L, A, P, st);
    if (rc != PCMM_OK) return rc;
    uint8_t* partial = (uint8_t*)ws + L.plan_bytes;
    return launch_exec(L, P, ctB, ctC, partial + pbytes, S, partial, parts, st);
}

}  // namespace

extern "C" size_t pcmm_cussen_workspace_bytes_for(int m, int n, int l, int w, int k, int strips) {
    Layout L;
    if (k < 1 || strips < 1 || !make_layout(L, m, n, l, w, k)) return 0;
    const size_t S = (size_t)strips < (size_t)L.nstrips ? (size_t)strips : (size_t)L.nstrips;
    // Room for the gather's partial sums as the default pass sizes them
    // (exec_space reserves them first, then fits the strips).
    return L.plan_bytes + partial_bytes(L, gather_parts(L, default_strips(L))) + S * L.per_strip_bytes;
}

extern "C" size_t pcmm_cussen_workspace_bytes(int m, int n, int l, int w, int k) {
    if (k == 0) k = pcmm_cussen_choose_k(m, n, l, w);
    Layout L;
    if (!make_layout(L, m, n, l, w, k)) return 0;
    return L.plan_bytes + default_exec_bytes(L);
}

extern "C" size_t pcmm_workspace_bytes(int op, int m, int n, int l, int w, int k) {
    const bool shape_ok = m >= 1 && n >= 1 && l >= 1 && w >= 1 && w <= PCMM_MAX_W16;
    size_t b = 0;
    switch (op) {
        case PCMM_OP_ENCRYPT:
            return pcmm_encrypt_workspace_bytes();
        case PCMM_OP_SCHOOLBOOK:
        case PCMM_OP_NORMALIZE:
            return shape_ok ? 0 : PCMM_WS_INVALID;
        case PCMM_OP_CUSSEN:
            b = pcmm_cussen_workspace_bytes(m, n, l, w, k);
            break;
        case PCMM_OP_CUSSEN_PLAN:
            b = pcmm_cussen_plan_bytes(m, n, w, k ? k : pcmm_cussen_choose_k(m, n, l, w));
            break;
        case PCMM_OP_CUSSEN_EXEC:
            b = pcmm_cussen_exec_bytes(m, n, l, w, k ? k : pcmm_cussen_choose_k(m, n, l, w));
            break;
        case PCMM_OP_STRASSEN:
            b = pcmm_strassen_workspace_bytes(m, n, l, w, k);
            break;
        default:
            return PCMM_WS_INVALID;
    }
    return (shape_ok && b) ? b : PCMM_WS_INVALID;
}

extern "C" pcmm_status pcmm_cussen(const uint8_t* A, int m, int n, int w, const uint32_t* ctB, int l,
                                   uint32_t* ctC, int k, void* ws, size_t ws_bytes,
                                   pcmm_stream_t stream) {
    return cussen_call(A, m, n, w, ctB, l, ctC, k, ws, ws_bytes, stream);
}

extern "C" pcmm_status pcmm_cussen16(const uint16_t* A, int m, int n, int w, const uint32_t* ctB, int l,
                                     uint32_t* ctC, int k, void* ws, size_t ws_bytes,
                                     pcmm_stream_t stream) {
    return cussen_call(A, m, n, w, ctB, l, ctC, k, ws, ws_bytes, stream);
}

extern "C" size_t pcmm_cussen_plan_bytes(int m, int n, int w, int k) {
    Layout L;
    if (!make_layout(L, m, n, 1, w, k)) return 0;
    return L.plan_bytes;
}

extern "C" pcmm_status pcmm_cussen_plan(const uint8_t* A, int m, int n, int w, int k, void* plan,
                                        size_t plan_bytes, pcmm_stream_t stream) {
    if (!A || !plan || ((uintptr_t)plan & 255u) || w > PCMM_MAX_W) return PCMM_EINVAL;
    Layout L;
    if (!make_layout(L, m, n, 1, w, k)) return PCMM_EINVAL;
    if (plan_bytes < L.plan_bytes) return PCMM_ENOMEM;
    return launch_plan(L, A, plan_ptrs(L, plan), (cudaStream_t)stream);
}

extern "C" size_t pcmm_cussen_exec_bytes(int m, int n, int l, int w, int k) {
    Layout L;
    if (!make_layout(L, m, n, l, w, k)) return 0;
    return default_exec_bytes(L);
}

extern "C" pcmm_status pcmm_cussen_execute(const void* plan, int m, int n, int w, int k,
                                           const uint32_t* ctB, int l, uint32_t* ctC, void* ws,
                                           size_t ws_bytes, pcmm_stream_t stream) {
    if (!plan || !ctB || !ctC || !ws || ((uintptr_t)plan & 255u) || ((uintptr_t)ws & 255u))
        return PCMM_EINVAL;
    Layout L;
    if (!make_layout(L, m, n, l, w, k)) return PCMM_EINVAL;
    size_t S, pbytes;
    int parts;
    if (!exec_space(L, ws_bytes, S, parts, pbytes)) return PCMM_ENOMEM;
    return launch_exec(L, plan_ptrs(L, const_cast<void*>(plan)), ctB, ctC, (uint8_t*)ws + pbytes, S,
                       (uint8_t*)ws, parts, (cudaStream_t)stream);
}

extern "C" pcmm_status pcmm_workspace_status(const void* ws, uint32_t* status_host, pcmm_stream_t stream) {
    if (!ws || !status_host) return PCMM_EINVAL;
    if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return PCMM_ECUDA;
    if (cudaMemcpy(status_host, ws, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return PCMM_ECUDA;
    return PCMM_OK;
}

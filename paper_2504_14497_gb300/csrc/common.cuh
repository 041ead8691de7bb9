// Helpers shared by the PC-MM kernels: status codes, the bounded device
// wait, batched inversion (Montgomery's simultaneous-inversion trick with
// warp-shuffle prefix products, optionally shared by the four warps of a
// block), warp-level affine normalisation, and the lane-planar scratch
// layout.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/pcmm.h"
#include "ec.cuh"

namespace pcmm {

// Error bits a kernel may raise in a device status word.
enum : uint32_t {
    DEV_ERR_A_RANGE = 1u << 0,  // an entry of A is >= 2^w
    DEV_ERR_PLAN = 1u << 1,     // a plan size exceeded its bound
    DEV_ERR_TIMEOUT = 1u << 2,  // a bounded device-side wait gave up
    DEV_ERR_BOUNDS = 1u << 3,   // a plan index outside its table (PCMM_DEBUG_BOUNDS builds)
};

// Waits until *ctr >= target, polling with short sleeps, for at most about
// 2^22 polls (roughly a second).  Gives up early when another warp has
// already raised DEV_ERR_TIMEOUT in *status; raises it itself when the bound
// runs out.  Returns whether the target was reached.  Call from one lane.
__device__ __forceinline__ bool wait_at_least(const int* ctr, int target, uint32_t* status) {
    for (int it = 0; it < (1 << 22); it++) {
        if (*(volatile const int*)ctr >= target) {
            __threadfence();
            return true;
        }
        if (*(volatile const uint32_t*)status & DEV_ERR_TIMEOUT) return false;
        __nanosleep(256);
    }
    atomicOr(status, DEV_ERR_TIMEOUT);
    return false;
}

__device__ __forceinline__ fe fe_shfl_up(const fe& a, unsigned d) {
    fe r;
#pragma unroll
    for (int i = 0; i < 8; i++) r.v[i] = __shfl_up_sync(0xffffffffu, a.v[i], d);
    return r;
}

__device__ __forceinline__ fe fe_shfl_down(const fe& a, unsigned d) {
    fe r;
#pragma unroll
    for (int i = 0; i < 8; i++) r.v[i] = __shfl_down_sync(0xffffffffu, a.v[i], d);
    return r;
}

__device__ __forceinline__ fe fe_shfl(const fe& a, int src) {
    fe r;
#pragma unroll
    for (int i = 0; i < 8; i++) r.v[i] = __shfl_sync(0xffffffffu, a.v[i], src);
    return r;
}

// a^-1 (Montgomery domain; 0 gives 0) of a value that all 32 lanes hold; all
// of them must call.
//
// Division steps (Bernstein and Yang, "Fast constant-time gcd computation
// and modular inversion", 2019) in batches of 30, with delta = k + 1/2 and several
// steps at once as in the variable-time inversion of libsecp256k1
// (src/modinv32_impl.h): from f = p, g = a a batch
// reads only the low words of f and g and yields integers u, v, q, r with
//   (f, g) <- (u f + v g, q f + r g) / 2^30,
// and the same map, with a multiple of p that makes the division exact, keeps
// d a = C f and e a = C g (mod p), starting from d = 0, e = C = R^2.  When g
// reaches 0 (after about 530 steps; 590 at most from that delta, 741 from the
// paper's, and the loop allows 750), f = +-1 and d = +-R^2 / a.
// A step with delta = k + 1/2 > 0 and g odd takes (f, g) <- (g, (g - f) / 2),
// delta <- 1 - delta; any other (f, g) <- (f, (g + (g mod 2) f) / 2), delta <-
// delta + 1.  Runs of the second kind are taken at once: w f with w = -g / f
// mod 2^j clears j low bits of g (j at most -k, the steps until delta turns
// positive, and at most 6, the precision of the inverse of f used).
//
// The four updates run in four lanes side by side (eight groups of four do
// the same): lane 0 of a group holds f, lane 1 g, lane 2 d, lane 3 e, each
// with a copy of its partner's, as nine signed limbs of 30 bits.  p is sparse
// in that radix, -1 + 2^6 2^90 + 2^12 2^180 - 2^14 2^210 + 2^16 2^240, so the
// multiple of p is the low limb itself and four shifted additions.  d and e
// grow by at most p a batch: 26 p at the end.
//
// Bound by its serial chain in one warp: 18 batches with about 96 rounds of
// the inner loop in all. Normalising 10 ciphertexts, which waits on one
// inversion, takes 33 us, against 76 us with a binary extended Euclid that
// every lane repeats on full-width values.  A product of factors that are all 1
// (points that are still affine, digits without a chain) is returned at once, as
// that Euclid did: the baby steps of 256 messages take 19 us, not 25.
static __device__ __noinline__ fe warp_uniform_inv(fe a) {
    const unsigned lane = threadIdx.x & 31u;
    const int M30 = 0x3fffffff;
    const unsigned all = 0xffffffffu;
    fe_canon(a, a);
    if (fe_is_one(a)) return a;
    // The limbs of this lane's value W and its partner's V.
    int W[9], V[9];
    {
        fe pm, r2;
        pm.v[0] = pm.v[1] = pm.v[2] = 0xffffffffu;
        pm.v[3] = pm.v[4] = pm.v[5] = 0u;
        pm.v[6] = 1u;
        pm.v[7] = 0xffffffffu;
        fe_set_R2(r2);
        const unsigned who = lane & 3u;
        uint32_t x[9], y[9];
#pragma unroll
        for (int i = 0; i < 8; i++) {
            x[i] = who == 0u ? pm.v[i] : who == 1u ? a.v[i] : who == 2u ? 0u : r2.v[i];
            y[i] = who == 0u ? a.v[i] : who == 1u ? pm.v[i] : who == 2u ? r2.v[i] : 0u;
        }
        x[8] = y[8] = 0u;
#pragma unroll
        for (int i = 0; i < 9; i++) {
            const int w = (30 * i) >> 5, sh = (30 * i) & 31;
            W[i] = (int)(__funnelshift_r(x[w], w < 8 ? x[w + 1] : 0u, sh) & (uint32_t)M30);
            V[i] = (int)(__funnelshift_r(y[w], w < 8 ? y[w + 1] : 0u, sh) & (uint32_t)M30);
        }
    }
    const int mdmask = (lane & 2u) ? M30 : 0;      // only d and e take multiples of p
    int k = 0;                                     // delta - 1/2
    for (int batch = 0; batch < 25; batch++) {
        // Low words of f and g, in every lane.
        const uint32_t low = (uint32_t)W[0] | ((uint32_t)W[1] << 30);
        uint32_t f = __shfl_sync(all, low, 0), g = __shfl_sync(all, low, 1);
        int u = 1, v = 0, q = 0, r = 1, left = 30;
        for (;;) {
            const int z = __ffs((int)(g | (1u << left))) - 1;
            g >>= z;
            u = (int)((uint32_t)u << z);
            v = (int)((uint32_t)v << z);
            k += z;
            left -= z;
            if (left == 0) break;
            if (k >= 0) {
                const uint32_t t = f;
                f = g;
                g = 0u - t;
                const int tu = u, tv = v;
                u = q;
                v = r;
                q = -tu;
                r = -tv;
                k = -k - 1;
            }
            int j = -k < left ? -k : left;
            j = j < 6 ? j : 6;
            const uint32_t w = (g * f * (f * f - 2u)) & ((1u << j) - 1u);
            g += w * f;
            q += (int)w * u;
            r += (int)w * v;
        }
        // W <- (A W + B V + md p) / 2^30.
        const int A = (lane & 1u) ? r : u, B = (lane & 1u) ? q : v;
        long long acc = (long long)A * W[0] + (long long)B * V[0];
        const int md = (int)acc & mdmask;
        acc >>= 30;
#pragma unroll
        for (int i = 1; i < 9; i++) {
            acc += (long long)A * W[i] + (long long)B * V[i];
            if (i == 3) acc += (long long)md << 6;
            if (i == 6) acc += (long long)md << 12;
            if (i == 7) acc -= (long long)md << 14;
            if (i == 8) acc += (long long)md << 16;
            W[i - 1] = (int)acc & M30;
            acc >>= 30;
        }
        W[8] = (int)acc;
        int nz = 0;
#pragma unroll
        for (int i = 0; i < 9; i++) {
            nz |= W[i];
            V[i] = __shfl_xor_sync(all, W[i], 1);
        }
        if (!__shfl_sync(all, nz, 1)) break;
    }
    // f = +-1 (p when a = 0, and d is then 0): the sign is that of the top limb.
    const int neg = __shfl_sync(all, W[8], 0) < 0 ? -1 : 0;
    // +-d + 32 p > 0, carried into limbs of 30 bits (top limb below 2^22), then
    // into nine words.
    uint32_t n[9];
    long long acc = 0;
#pragma unroll
    for (int i = 0; i < 9; i++) {
        const int x = __shfl_sync(all, W[i], 2);
        acc += (x ^ neg) - neg;
        acc += i == 0 ? -32 : i == 3 ? 32 << 6 : i == 6 ? 32 << 12 : i == 7 ? -(32 << 14) : i == 8 ? 32 << 16 : 0;
        n[i] = i < 8 ? (uint32_t)acc & (uint32_t)M30 : (uint32_t)acc;
        acc >>= 30;
    }
    fe lo, hi;
#pragma unroll
    for (int i = 0; i < 8; i++) {
        // Bits 32 i .. 32 i + 31 lie in limbs b and b + 1.
        const int b = (32 * i) / 30, sh = (32 * i) % 30;
        lo.v[i] = (n[b] >> sh) | (n[b + 1] << (30 - sh));
    }
    // The value is lo + top 2^256 with top < 2^7; top 2^256 = top K (mod p).
    const uint32_t top = n[8] >> 16;
    fe_zero(hi);
    hi.v[0] = top;
    fe r2;
    fe_set_R2(r2);
    hi = fmul(hi, r2);                             // top R = top 2^256
    fe_add(lo, lo, hi);
    return lo;
}

// Given each lane's value t (non-zero), returns t^-1 using one field
// inversion for the whole warp: inclusive prefix and suffix products over
// the lanes by shuffles, the inverse of the warp total, and
// t^-1 = total^-1 * (product of the other lanes).  All 32 lanes must call.
__device__ __forceinline__ void warp_inverse(fe& tinv, const fe& t) {
    const unsigned lane = threadIdx.x & 31u;
    fe pre = t, suf = t, o;
#pragma unroll
    for (unsigned d = 1; d < 32; d <<= 1) {
        o = fe_shfl_up(pre, d);
        if (lane >= d) pre = fmul(pre, o);
    }
#pragma unroll
    for (unsigned d = 1; d < 32; d <<= 1) {
        o = fe_shfl_down(suf, d);
        if (lane + d < 32u) suf = fmul(suf, o);
    }
    fe total = fe_shfl(pre, 31);
    fe pex = fe_shfl_up(pre, 1);    // product of lanes below
    fe sex = fe_shfl_down(suf, 1);  // product of lanes above
    if (lane == 0) fe_one(pex);
    if (lane == 31) fe_one(sex);
    fe inv = warp_uniform_inv(total);
    inv = fmul(inv, pex);
    tinv = fmul(inv, sex);
}

// warp_inverse with one field inversion shared by the four warps of a
// 128-thread block: each warp's total goes to shared
// memory, warp 0 inverts the product of the four and hands each warp the
// inverse of its total.  All 128 threads of the block must call, in the same
// order as every other block-level call (blockDim.x must be 128).
static __device__ __noinline__ fe block4_inverse(fe t) {
    __shared__ fe sh_tot[4];
    __shared__ fe sh_inv[4];
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    fe pre = t, suf = t, o;
#pragma unroll
    for (unsigned d = 1; d < 32; d <<= 1) {
        o = fe_shfl_up(pre, d);
        if (lane >= d) pre = fmul(pre, o);
    }
#pragma unroll
    for (unsigned d = 1; d < 32; d <<= 1) {
        o = fe_shfl_down(suf, d);
        if (lane + d < 32u) suf = fmul(suf, o);
    }
    fe total = fe_shfl(pre, 31);
    fe pex = fe_shfl_up(pre, 1);
    fe sex = fe_shfl_down(suf, 1);
    if (lane == 0) fe_one(pex);
    if (lane == 31) fe_one(sex);
    if (lane == 0) sh_tot[warp] = total;
    __syncthreads();
    if (warp == 0) {
        const fe p01 = fmul(sh_tot[0], sh_tot[1]);
        const fe p012 = fmul(p01, sh_tot[2]);
        const fe i = warp_uniform_inv(fmul(p012, sh_tot[3]));
        const fe i3 = fmul(i, p012);                 // total_3^-1
        const fe i012 = fmul(i, sh_tot[3]);          // (t0 t1 t2)^-1
        const fe i2 = fmul(i012, p01);               // total_2^-1
        const fe i01 = fmul(i012, sh_tot[2]);        // (t0 t1)^-1
        const fe i1 = fmul(i01, sh_tot[0]);
        const fe i0 = fmul(i01, sh_tot[1]);
        if (lane == 0) {
            sh_inv[0] = i0;
            sh_inv[1] = i1;
            sh_inv[2] = i2;
            sh_inv[3] = i3;
        }
    }
    __syncthreads();
    fe inv = sh_inv[warp];
    inv = fmul(inv, pex);
    return fmul(inv, sex);
}

// The inverses of 128 non-zero values, one per thread of a 128-thread block,
// in place in shared memory (low quads sm[0..127], high quads sm[128..255]),
// by one warp: each lane folds four of the values, the lanes fold theirs by
// a butterfly of which every lane keeps its partners' products, one field
// inversion, and the same way back: 19 multiplications and an inversion of
// one warp while the other blocks of the SM have the pipes. Call with one
// whole warp, between two block barriers.
static __device__ __noinline__ void fold_inverse128(uint4* sm) {
    const unsigned lane = threadIdx.x & 31u;
    fe t[4], sib[5];
#pragma unroll
    for (int w = 0; w < 4; w++) fe_from_quads(t[w], sm[32 * w + lane], sm[128 + 32 * w + lane]);
    const fe p1 = fmul(t[0], t[1]);
    const fe p2 = fmul(p1, t[2]);
    fe cur = fmul(p2, t[3]);
#pragma unroll
    for (int k = 0; k < 5; k++) {
#pragma unroll
        for (int i = 0; i < 8; i++) sib[k].v[i] = __shfl_xor_sync(0xffffffffu, cur.v[i], 1 << k);
        cur = fmul(cur, sib[k]);
    }
    fe inv = warp_uniform_inv(cur);
#pragma unroll
    for (int k = 4; k >= 0; k--) inv = fmul(inv, sib[k]);
    fe r = fmul(inv, p2);
    sm[96 + lane] = fe_lo(r);
    sm[128 + 96 + lane] = fe_hi(r);
    inv = fmul(inv, t[3]);
    r = fmul(inv, p1);
    sm[64 + lane] = fe_lo(r);
    sm[128 + 64 + lane] = fe_hi(r);
    inv = fmul(inv, t[2]);
    r = fmul(inv, t[0]);
    sm[32 + lane] = fe_lo(r);
    sm[128 + 32 + lane] = fe_hi(r);
    r = fmul(inv, t[1]);
    sm[lane] = fe_lo(r);
    sm[128 + lane] = fe_hi(r);
}

// t^-1 per lane: block4_inverse when `shared` (then all 128 threads of the
// block must call), warp_inverse otherwise.
__device__ __forceinline__ void group_inverse(fe& tinv, const fe& t, bool shared) {
    if (shared) tinv = block4_inverse(t);
    else warp_inverse(tinv, t);
}

// Whether x holds on every lane of the warp or, with `shared`, on every
// thread of the block (then all threads of the block must call).
__device__ __forceinline__ bool group_all(bool x, bool shared) {
    __syncwarp();   // lanes may come from different branches; a block barrier wants the warp whole
    return shared ? __syncthreads_and(x) != 0 : __all_sync(0xffffffffu, x);
}

// Normalise E Jacobian points held in each lane's registers to affine
// coordinates; infinity (Z = 0) becomes (0, 0).  One inversion per
// warp for 32 * E points.  All 32 lanes must call.
template <int E>
__device__ __forceinline__ void warp_normalize_regs(aff out[E], const jac P[E]) {
    fe pref[E];
    fe acc;
    fe_one(acc);
#pragma unroll
    for (int e = 0; e < E; e++) {
        fe z = P[e].Z;
        if (fe_is_zero(z)) fe_one(z);
        acc = fmul(acc, z);
        pref[e] = acc;
    }
    fe inv;
    warp_inverse(inv, acc);
#pragma unroll
    for (int e = E - 1; e >= 0; e--) {
        fe zinv;
        if (e > 0) zinv = fmul(inv, pref[e - 1]);
        else zinv = inv;
        fe z = P[e].Z;
        bool is_inf = fe_is_zero(z);
        if (is_inf) fe_one(z);
        inv = fmul(inv, z);
        if (is_inf) {
            fe_zero(out[e].x);
            fe_zero(out[e].y);
        } else {
            jac_to_aff_with_zinv(out[e], P[e], zinv);
        }
    }
}

// ---------------------------------------------------------------------------
// Lane-planar scratch: a per-warp array of E entries, each entry holding Q
// quads for each of the 32 lanes; quad q of entry e for lane L lives at
// uint4 index (e * Q + q) * 32 + L, so every access is a coalesced 512-byte
// warp transaction.
// ---------------------------------------------------------------------------

__device__ __forceinline__ void lp_store_jac(uint4* base, int e, unsigned lane, const jac& P) {
    uint4* b = base + (size_t)e * 6 * 32 + lane;
    b[0] = fe_lo(P.X);
    b[32] = fe_hi(P.X);
    b[64] = fe_lo(P.Y);
    b[96] = fe_hi(P.Y);
    b[128] = fe_lo(P.Z);
    b[160] = fe_hi(P.Z);
}

__device__ __forceinline__ void lp_load_jac(jac& P, const uint4* base, int e, unsigned lane) {
    const uint4* b = base + (size_t)e * 6 * 32 + lane;
    fe_from_quads(P.X, b[0], b[32]);
    fe_from_quads(P.Y, b[64], b[96]);
    fe_from_quads(P.Z, b[128], b[160]);
}

__device__ __forceinline__ void lp_load_z(fe& z, const uint4* base, int e, unsigned lane) {
    const uint4* b = base + (size_t)e * 6 * 32 + lane;
    fe_from_quads(z, b[128], b[160]);
}

__device__ __forceinline__ void lp_store_fe(uint4* base, int e, unsigned lane, const fe& a) {
    uint4* b = base + (size_t)e * 2 * 32 + lane;
    b[0] = fe_lo(a);
    b[32] = fe_hi(a);
}

__device__ __forceinline__ void lp_load_fe(fe& a, const uint4* base, int e, unsigned lane) {
    const uint4* b = base + (size_t)e * 2 * 32 + lane;
    fe_from_quads(a, b[0], b[32]);
}

}  // namespace pcmm

#define PCMM_CUDA_CHECK_LAUNCH()                                   \
    do {                                                           \
        cudaError_t _e = cudaGetLastError();                       \
        if (_e != cudaSuccess) return PCMM_ECUDA;                  \
    } while (0)

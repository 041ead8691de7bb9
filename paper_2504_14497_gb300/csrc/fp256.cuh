// Prime-field arithmetic in F_p for NIST P-256, p = 2^256 - 2^224 + 2^192 + 2^96 - 1
// (Section 4.1), on sm_103a.
//
// Representation: 8 x 32-bit little-endian limbs held in registers, in the
// MONTGOMERY domain with R = 2^256: the field element x is held as x R mod p.
// Values are kept WEAKLY reduced: any integer in [0, 2^256) that is congruent
// to x R (so 0 may appear as 0 or as p).  fe_canon() gives the unique
// representative below p.  Everything outside the kernels (inputs, strip
// tables, results, comb tables) is standard: fe_to_mont and fe_from_mont
// convert at the kernels' loads and stores, or the conversion is folded into
// a factor that is there anyway (see jacz in ec.cuh).
//
// Multiplication: 8x8-limb operand scanning, one row per limb of b, with the
// products of even and odd word positions in two accumulators, so that every
// limb product is one 64-bit multiply-add with carry in and out (a mad.lo.cc /
// madc.hi.cc pair) and almost no separate carry additions are left: 64 wide
// multiply-adds and 24 ALU additions.  Measured per warp and scheduler at
// eight warps each: a wide multiply-add takes 4.2 cycles of the FMA pipe
// (30 a clock and SM; a low-half one 2.1) and an addition with carry 2.1 of
// the ALU pipe, so a product is bound by 270 FMA cycles.  Adding each row's
// running word as a zero-extended 64-bit addend and folding the high halves
// in with addc took a register move per product beside 57 additions:
// 385 cycles a product against 290, 530 a multiplication against 437.
// Squaring: 28 cross products, doubled, plus 8 diagonal squares.  Products
// and reductions also live in out-of-line functions (fmul, fsqr), which the
// table builds call: a call moves its operands on the pipe that multiplies, but
// their code inlined at every site outgrows the instruction cache.  Loops of
// one addition or doubling inline them (gather, encryption, decryption).
//
// Reduction of the 512-bit product t to t / R mod p: since p = -1 mod 2^96,
// the three lowest words q of t cancel against q p, which leaves (after the
// shift by 96 bits) t / 2^96 + q (2^160 - 2^128 + 2^96 + 1): with D = q (2^64
// - 2^32 + 1), five words from seven additions, one carry chain of eight adds
// (q, D).  Steps of 3, 3 and 2 words clear all eight: about 54 additions and
// no multiplications.  Measured per warp and scheduler: 102 cycles, against
// 205 for the special-form (Solinas) reduction of a standard residue, whose
// nine rearranged terms need 96 additions; a multiplication takes 330 cycles
// inlined and 336 called (437 and 448 with the special-form reduction), a
// squaring 262. The corrections by p and K take their words from the carry
// itself: with general masks the multiplication took 347 cycles and a
// subtraction 65 instead of 49.
#pragma once
#include <stdint.h>

namespace pcmm {

struct fe {
    uint32_t v[8];
};

// K = 2^256 mod p = 2^224 - 2^192 - 2^96 + 1, little-endian words.
#define PCMM_K0 0x00000001u
#define PCMM_K3 0xffffffffu
#define PCMM_K6 0xfffffffeu

__device__ __forceinline__ void fe_zero(fe& r) {
#pragma unroll
    for (int i = 0; i < 8; i++) r.v[i] = 0;
}

// The field element 1: R mod p = K.
__device__ __forceinline__ void fe_one(fe& r) {
    r.v[0] = PCMM_K0;
    r.v[1] = r.v[2] = 0;
    r.v[3] = r.v[4] = r.v[5] = PCMM_K3;
    r.v[6] = PCMM_K6;
    r.v[7] = 0;
}

// R^2 mod p and R^3 mod p.
__device__ __forceinline__ void fe_set_R2(fe& r) {
    r.v[0] = 3u; r.v[1] = 0u; r.v[2] = 0xffffffffu; r.v[3] = 0xfffffffbu;
    r.v[4] = 0xfffffffeu; r.v[5] = 0xffffffffu; r.v[6] = 0xfffffffdu; r.v[7] = 4u;
}
__device__ __forceinline__ void fe_set_R3(fe& r) {
    r.v[0] = 0x0000000au; r.v[1] = 0xfffffffdu; r.v[2] = 0xfffffff7u; r.v[3] = 0xffffffedu;
    r.v[4] = 0xfffffffcu; r.v[5] = 0x00000005u; r.v[6] = 0x00000001u; r.v[7] = 0x00000018u;
}

// r += p & m (m is 0 or 0xffffffff) modulo 2^256; returns the carry out. With
// words 3..5 of p zero and all others but word 6 full, m itself is the addend.
__device__ __forceinline__ uint32_t fe_add_p_masked(fe& r, uint32_t m) {
    uint32_t c;
    asm("add.cc.u32  %0, %0, %9;\n\t"
        "addc.cc.u32 %1, %1, %9;\n\t"
        "addc.cc.u32 %2, %2, %9;\n\t"
        "addc.cc.u32 %3, %3, 0;\n\t"
        "addc.cc.u32 %4, %4, 0;\n\t"
        "addc.cc.u32 %5, %5, 0;\n\t"
        "addc.cc.u32 %6, %6, %10;\n\t"
        "addc.cc.u32 %7, %7, %9;\n\t"
        "addc.u32    %8, 0, 0;"
        : "+r"(r.v[0]), "+r"(r.v[1]), "+r"(r.v[2]), "+r"(r.v[3]), "+r"(r.v[4]), "+r"(r.v[5]),
          "+r"(r.v[6]), "+r"(r.v[7]), "=r"(c)
        : "r"(m), "r"(m & 1u));
    return c;
}

// r -= c p (c is 0 or 1) modulo 2^256; returns 0xffffffff on a borrow, else 0.
__device__ __forceinline__ uint32_t fe_sub_p_times(fe& r, uint32_t c) {
    const uint32_t m = 0u - c;
    uint32_t b;
    asm("sub.cc.u32  %0, %0, %9;\n\t"
        "subc.cc.u32 %1, %1, %9;\n\t"
        "subc.cc.u32 %2, %2, %9;\n\t"
        "subc.cc.u32 %3, %3, 0;\n\t"
        "subc.cc.u32 %4, %4, 0;\n\t"
        "subc.cc.u32 %5, %5, 0;\n\t"
        "subc.cc.u32 %6, %6, %10;\n\t"
        "subc.cc.u32 %7, %7, %9;\n\t"
        "subc.u32    %8, 0, 0;"
        : "+r"(r.v[0]), "+r"(r.v[1]), "+r"(r.v[2]), "+r"(r.v[3]), "+r"(r.v[4]), "+r"(r.v[5]),
          "+r"(r.v[6]), "+r"(r.v[7]), "=r"(b)
        : "r"(m), "r"(c));
    return b;
}

// r = a + b mod p (weak). A carry out of 2^256 is paid for by subtracting p; in
// the rare case (about 2^-32) that this does not take the sum below 2^256, a
// second subtraction does.
__device__ __forceinline__ void fe_add(fe& r, const fe& a, const fe& b) {
    uint32_t c;
    asm("add.cc.u32  %0, %9, %17;\n\t"
        "addc.cc.u32 %1, %10, %18;\n\t"
        "addc.cc.u32 %2, %11, %19;\n\t"
        "addc.cc.u32 %3, %12, %20;\n\t"
        "addc.cc.u32 %4, %13, %21;\n\t"
        "addc.cc.u32 %5, %14, %22;\n\t"
        "addc.cc.u32 %6, %15, %23;\n\t"
        "addc.cc.u32 %7, %16, %24;\n\t"
        "addc.u32    %8, 0, 0;"
        : "=r"(r.v[0]), "=r"(r.v[1]), "=r"(r.v[2]), "=r"(r.v[3]), "=r"(r.v[4]), "=r"(r.v[5]),
          "=r"(r.v[6]), "=r"(r.v[7]), "=r"(c)
        : "r"(a.v[0]), "r"(a.v[1]), "r"(a.v[2]), "r"(a.v[3]), "r"(a.v[4]), "r"(a.v[5]),
          "r"(a.v[6]), "r"(a.v[7]), "r"(b.v[0]), "r"(b.v[1]), "r"(b.v[2]), "r"(b.v[3]),
          "r"(b.v[4]), "r"(b.v[5]), "r"(b.v[6]), "r"(b.v[7]));
    c += fe_sub_p_times(r, c);           // the net top word, 0 but for the rare case
    if (c) fe_sub_p_times(r, c);
}

// r = a - b mod p (weak). A borrow is paid for by adding p; in the rare case
// that the value stays negative (b - a > p, which needs b >= p) once more.
__device__ __forceinline__ void fe_sub(fe& r, const fe& a, const fe& b) {
    uint32_t bw;
    asm("sub.cc.u32  %0, %9, %17;\n\t"
        "subc.cc.u32 %1, %10, %18;\n\t"
        "subc.cc.u32 %2, %11, %19;\n\t"
        "subc.cc.u32 %3, %12, %20;\n\t"
        "subc.cc.u32 %4, %13, %21;\n\t"
        "subc.cc.u32 %5, %14, %22;\n\t"
        "subc.cc.u32 %6, %15, %23;\n\t"
        "subc.cc.u32 %7, %16, %24;\n\t"
        "subc.u32    %8, 0, 0;"
        : "=r"(r.v[0]), "=r"(r.v[1]), "=r"(r.v[2]), "=r"(r.v[3]), "=r"(r.v[4]), "=r"(r.v[5]),
          "=r"(r.v[6]), "=r"(r.v[7]), "=r"(bw)
        : "r"(a.v[0]), "r"(a.v[1]), "r"(a.v[2]), "r"(a.v[3]), "r"(a.v[4]), "r"(a.v[5]),
          "r"(a.v[6]), "r"(a.v[7]), "r"(b.v[0]), "r"(b.v[1]), "r"(b.v[2]), "r"(b.v[3]),
          "r"(b.v[4]), "r"(b.v[5]), "r"(b.v[6]), "r"(b.v[7]));
    bw += fe_add_p_masked(r, bw);
    if (bw) fe_add_p_masked(r, bw);
}

// r = a - b mod p for b <= p (canonical, say): one addition of p always does.
__device__ __forceinline__ void fe_sub_canon(fe& r, const fe& a, const fe& b) {
    uint32_t bw;
    asm("sub.cc.u32  %0, %9, %17;\n\t"
        "subc.cc.u32 %1, %10, %18;\n\t"
        "subc.cc.u32 %2, %11, %19;\n\t"
        "subc.cc.u32 %3, %12, %20;\n\t"
        "subc.cc.u32 %4, %13, %21;\n\t"
        "subc.cc.u32 %5, %14, %22;\n\t"
        "subc.cc.u32 %6, %15, %23;\n\t"
        "subc.cc.u32 %7, %16, %24;\n\t"
        "subc.u32    %8, 0, 0;"
        : "=r"(r.v[0]), "=r"(r.v[1]), "=r"(r.v[2]), "=r"(r.v[3]), "=r"(r.v[4]), "=r"(r.v[5]),
          "=r"(r.v[6]), "=r"(r.v[7]), "=r"(bw)
        : "r"(a.v[0]), "r"(a.v[1]), "r"(a.v[2]), "r"(a.v[3]), "r"(a.v[4]), "r"(a.v[5]),
          "r"(a.v[6]), "r"(a.v[7]), "r"(b.v[0]), "r"(b.v[1]), "r"(b.v[2]), "r"(b.v[3]),
          "r"(b.v[4]), "r"(b.v[5]), "r"(b.v[6]), "r"(b.v[7]));
    asm("add.cc.u32  %0, %0, %8;\n\t"
        "addc.cc.u32 %1, %1, %8;\n\t"
        "addc.cc.u32 %2, %2, %8;\n\t"
        "addc.cc.u32 %3, %3, 0;\n\t"
        "addc.cc.u32 %4, %4, 0;\n\t"
        "addc.cc.u32 %5, %5, 0;\n\t"
        "addc.cc.u32 %6, %6, %9;\n\t"
        "addc.u32    %7, %7, %8;"
        : "+r"(r.v[0]), "+r"(r.v[1]), "+r"(r.v[2]), "+r"(r.v[3]), "+r"(r.v[4]), "+r"(r.v[5]),
          "+r"(r.v[6]), "+r"(r.v[7])
        : "r"(bw), "r"(bw & 1u));
}

__device__ __forceinline__ void fe_dbl(fe& r, const fe& a) { fe_add(r, a, a); }

// Canonical representative in [0, p): subtract p once if a >= p.
__device__ __forceinline__ void fe_canon(fe& r, const fe& a) {
    fe t;
    uint32_t bw;
    asm("sub.cc.u32  %0, %9, 0xffffffff;\n\t"
        "subc.cc.u32 %1, %10, 0xffffffff;\n\t"
        "subc.cc.u32 %2, %11, 0xffffffff;\n\t"
        "subc.cc.u32 %3, %12, 0;\n\t"
        "subc.cc.u32 %4, %13, 0;\n\t"
        "subc.cc.u32 %5, %14, 0;\n\t"
        "subc.cc.u32 %6, %15, 1;\n\t"
        "subc.cc.u32 %7, %16, 0xffffffff;\n\t"
        "subc.u32    %8, 0, 0;"
        : "=r"(t.v[0]), "=r"(t.v[1]), "=r"(t.v[2]), "=r"(t.v[3]), "=r"(t.v[4]), "=r"(t.v[5]),
          "=r"(t.v[6]), "=r"(t.v[7]), "=r"(bw)
        : "r"(a.v[0]), "r"(a.v[1]), "r"(a.v[2]), "r"(a.v[3]), "r"(a.v[4]), "r"(a.v[5]),
          "r"(a.v[6]), "r"(a.v[7]));
    // bw = 0xffffffff when a < p: keep a.
#pragma unroll
    for (int i = 0; i < 8; i++) r.v[i] = (a.v[i] & bw) | (t.v[i] & ~bw);
}

// True when a = 0 (mod p), i.e. a is 0 or p.
__device__ __forceinline__ bool fe_is_zero(const fe& a) {
    uint32_t z = a.v[0] | a.v[1] | a.v[2] | a.v[3] | a.v[4] | a.v[5] | a.v[6] | a.v[7];
    uint32_t q = (a.v[0] ^ 0xffffffffu) | (a.v[1] ^ 0xffffffffu) | (a.v[2] ^ 0xffffffffu) |
                 a.v[3] | a.v[4] | a.v[5] | (a.v[6] ^ 1u) | (a.v[7] ^ 0xffffffffu);
    return (z == 0u) | (q == 0u);
}

// True when a = b (mod p).
__device__ __forceinline__ bool fe_equal(const fe& a, const fe& b) {
    fe d;
    fe_sub(d, a, b);
    return fe_is_zero(d);
}

// Whether a holds exactly the canonical words of 1 (the congruent value
// above p, which weakly reduced arithmetic could produce, is not recognised;
// callers use this only to skip work when it says yes).
__device__ __forceinline__ bool fe_is_one(const fe& a) {
    uint32_t z = (a.v[0] ^ PCMM_K0) | a.v[1] | a.v[2] | (a.v[3] ^ PCMM_K3) | (a.v[4] ^ PCMM_K3) |
                 (a.v[5] ^ PCMM_K3) | (a.v[6] ^ PCMM_K6) | a.v[7];
    return z == 0u;
}

// r = t / R mod p (weak) for any 512-bit t; t is clobbered.
__device__ __forceinline__ void fe_reduce(fe& r, uint32_t t[16]) {
    uint32_t D1, D2, D3, D4, c;
    // Words 0..2 (q): D = q (2^64 - 2^32 + 1) = (q0, D1, D2, D3, D4), then
    // words 3..10 += (q0, q1, q2, q0, D1, D2, D3, D4), carry c into word 11.
    asm("add.cc.u32  %1, %6, %4;\n\t"
        "addc.cc.u32 %2, %5, 0;\n\t"
        "addc.u32    %3, %6, 0;\n\t"
        "sub.cc.u32  %0, %5, %4;\n\t"
        "subc.cc.u32 %1, %1, %5;\n\t"
        "subc.cc.u32 %2, %2, %6;\n\t"
        "subc.u32    %3, %3, 0;"
        : "=&r"(D1), "=&r"(D2), "=&r"(D3), "=&r"(D4)
        : "r"(t[0]), "r"(t[1]), "r"(t[2]));
    asm("add.cc.u32  %0, %0, %9;\n\t"
        "addc.cc.u32 %1, %1, %10;\n\t"
        "addc.cc.u32 %2, %2, %11;\n\t"
        "addc.cc.u32 %3, %3, %9;\n\t"
        "addc.cc.u32 %4, %4, %12;\n\t"
        "addc.cc.u32 %5, %5, %13;\n\t"
        "addc.cc.u32 %6, %6, %14;\n\t"
        "addc.cc.u32 %7, %7, %15;\n\t"
        "addc.u32    %8, 0, 0;"
        : "+r"(t[3]), "+r"(t[4]), "+r"(t[5]), "+r"(t[6]), "+r"(t[7]), "+r"(t[8]), "+r"(t[9]), "+r"(t[10]),
          "=r"(c)
        : "r"(t[0]), "r"(t[1]), "r"(t[2]), "r"(D1), "r"(D2), "r"(D3), "r"(D4));
    // Words 3..5: the same, with the carry c (word 11) joining D2; D stays
    // below 2^160 with it.  New carry c into word 14.
    asm("add.cc.u32  %1, %7, 0xffffffff;\n\t"
        "addc.cc.u32 %1, %6, %4;\n\t"
        "addc.cc.u32 %2, %5, 0;\n\t"
        "addc.u32    %3, %6, 0;\n\t"
        "sub.cc.u32  %0, %5, %4;\n\t"
        "subc.cc.u32 %1, %1, %5;\n\t"
        "subc.cc.u32 %2, %2, %6;\n\t"
        "subc.u32    %3, %3, 0;"
        : "=&r"(D1), "=&r"(D2), "=&r"(D3), "=&r"(D4)
        : "r"(t[3]), "r"(t[4]), "r"(t[5]), "r"(c));
    asm("add.cc.u32  %0, %0, %9;\n\t"
        "addc.cc.u32 %1, %1, %10;\n\t"
        "addc.cc.u32 %2, %2, %11;\n\t"
        "addc.cc.u32 %3, %3, %9;\n\t"
        "addc.cc.u32 %4, %4, %12;\n\t"
        "addc.cc.u32 %5, %5, %13;\n\t"
        "addc.cc.u32 %6, %6, %14;\n\t"
        "addc.cc.u32 %7, %7, %15;\n\t"
        "addc.u32    %8, 0, 0;"
        : "+r"(t[6]), "+r"(t[7]), "+r"(t[8]), "+r"(t[9]), "+r"(t[10]), "+r"(t[11]), "+r"(t[12]), "+r"(t[13]),
          "=r"(c)
        : "r"(t[3]), "r"(t[4]), "r"(t[5]), "r"(D1), "r"(D2), "r"(D3), "r"(D4));
    // Words 6, 7: D = (q0, D1, D2, D3) with the carry c (word 14) added to D2,
    // then words 9..15 += (q0, q1, 0, q0, D1, D2, D3), carry c.
    asm("sub.cc.u32  %0, %4, %3;\n\t"
        "subc.cc.u32 %1, %3, %4;\n\t"
        "subc.u32    %2, %4, 0;\n\t"
        "add.cc.u32  %1, %1, %5;\n\t"
        "addc.u32    %2, %2, 0;"
        : "=&r"(D1), "=&r"(D2), "=&r"(D3)
        : "r"(t[6]), "r"(t[7]), "r"(c));
    asm("add.cc.u32  %0, %0, %8;\n\t"
        "addc.cc.u32 %1, %1, %9;\n\t"
        "addc.cc.u32 %2, %2, 0;\n\t"
        "addc.cc.u32 %3, %3, %8;\n\t"
        "addc.cc.u32 %4, %4, %10;\n\t"
        "addc.cc.u32 %5, %5, %11;\n\t"
        "addc.cc.u32 %6, %6, %12;\n\t"
        "addc.u32    %7, 0, 0;"
        : "+r"(t[9]), "+r"(t[10]), "+r"(t[11]), "+r"(t[12]), "+r"(t[13]), "+r"(t[14]), "+r"(t[15]), "=r"(c)
        : "r"(t[6]), "r"(t[7]), "r"(D1), "r"(D2), "r"(D3));
    // The value (t + q p) / R is below 2^256 + p: on a carry add K once (and
    // drop the carry), with c itself and -c as the words of c K.
#pragma unroll
    for (int i = 0; i < 8; i++) r.v[i] = t[8 + i];
    const uint32_t n = 0u - c;
    asm("add.cc.u32  %0, %0, %8;\n\t"
        "addc.cc.u32 %1, %1, 0;\n\t"
        "addc.cc.u32 %2, %2, 0;\n\t"
        "addc.cc.u32 %3, %3, %9;\n\t"
        "addc.cc.u32 %4, %4, %9;\n\t"
        "addc.cc.u32 %5, %5, %9;\n\t"
        "addc.cc.u32 %6, %6, %10;\n\t"
        "addc.u32    %7, %7, 0;"
        : "+r"(r.v[0]), "+r"(r.v[1]), "+r"(r.v[2]), "+r"(r.v[3]), "+r"(r.v[4]), "+r"(r.v[5]),
          "+r"(r.v[6]), "+r"(r.v[7])
        : "r"(c), "r"(n), "r"(n << 1));
}

// Rows of fused wide multiply-adds.  A 64-bit product a_j b_i lands on words
// i + j and i + j + 1; products whose i + j has one parity tile the word
// positions without overlap, so a row's four even (or four odd) products join
// one carry chain of mad.lo.cc / madc.hi.cc pairs, and each pair is a single
// 64-bit multiply-add with carry in and out.

// e[0..7] = the four products of a row (nothing accumulated yet).
__device__ __forceinline__ void row_first(uint32_t* e, uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3,
                                          uint32_t b) {
    uint64_t p = (uint64_t)x0 * b;
    e[0] = (uint32_t)p; e[1] = (uint32_t)(p >> 32);
    p = (uint64_t)x1 * b;
    e[2] = (uint32_t)p; e[3] = (uint32_t)(p >> 32);
    p = (uint64_t)x2 * b;
    e[4] = (uint32_t)p; e[5] = (uint32_t)(p >> 32);
    p = (uint64_t)x3 * b;
    e[6] = (uint32_t)p; e[7] = (uint32_t)(p >> 32);
}

// e[0..7] += the four products; the carry out becomes e[8].
__device__ __forceinline__ void row_carry(uint32_t* e, uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3,
                                          uint32_t b) {
    asm("mad.lo.cc.u32 %0, %9, %13, %0;\n\tmadc.hi.cc.u32 %1, %9, %13, %1;\n\t"
        "madc.lo.cc.u32 %2, %10, %13, %2;\n\tmadc.hi.cc.u32 %3, %10, %13, %3;\n\t"
        "madc.lo.cc.u32 %4, %11, %13, %4;\n\tmadc.hi.cc.u32 %5, %11, %13, %5;\n\t"
        "madc.lo.cc.u32 %6, %12, %13, %6;\n\tmadc.hi.cc.u32 %7, %12, %13, %7;\n\t"
        "addc.u32 %8, 0, 0;"
        : "+r"(e[0]), "+r"(e[1]), "+r"(e[2]), "+r"(e[3]), "+r"(e[4]), "+r"(e[5]), "+r"(e[6]), "+r"(e[7]),
          "=r"(e[8])
        : "r"(x0), "r"(x1), "r"(x2), "r"(x3), "r"(b));
}

// e[0..6] += the four products, whose top word becomes e[7]: e[7] was not
// written before and e[6] held at most a carry, so nothing carries out.
__device__ __forceinline__ void row_top(uint32_t* e, uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3,
                                        uint32_t b) {
    asm("mad.lo.cc.u32 %0, %8, %12, %0;\n\tmadc.hi.cc.u32 %1, %8, %12, %1;\n\t"
        "madc.lo.cc.u32 %2, %9, %12, %2;\n\tmadc.hi.cc.u32 %3, %9, %12, %3;\n\t"
        "madc.lo.cc.u32 %4, %10, %12, %4;\n\tmadc.hi.cc.u32 %5, %10, %12, %5;\n\t"
        "madc.lo.cc.u32 %6, %11, %12, %6;\n\tmadc.hi.u32 %7, %11, %12, 0;"
        : "+r"(e[0]), "+r"(e[1]), "+r"(e[2]), "+r"(e[3]), "+r"(e[4]), "+r"(e[5]), "+r"(e[6]), "=r"(e[7])
        : "r"(x0), "r"(x1), "r"(x2), "r"(x3), "r"(b));
}

// t[0..15] = a * b: e collects the products at even word positions, o those
// at odd positions (one word lower), and t = e + 2^32 o.
__device__ __forceinline__ void mul_wide(uint32_t t[16], const fe& a, const fe& b) {
    uint32_t e[16], o[15];
    row_first(e, a.v[0], a.v[2], a.v[4], a.v[6], b.v[0]);
    row_first(o, a.v[1], a.v[3], a.v[5], a.v[7], b.v[0]);
    e[8] = 0;
#pragma unroll
    for (int i = 1; i < 8; i++) {
        if (i & 1) {
            row_top(e + i + 1, a.v[1], a.v[3], a.v[5], a.v[7], b.v[i]);
            row_carry(o + i - 1, a.v[0], a.v[2], a.v[4], a.v[6], b.v[i]);
        } else {
            row_carry(e + i, a.v[0], a.v[2], a.v[4], a.v[6], b.v[i]);
            row_top(o + i, a.v[1], a.v[3], a.v[5], a.v[7], b.v[i]);
        }
    }
    t[0] = e[0];
    asm("add.cc.u32  %0, %15, %30;\n\taddc.cc.u32 %1, %16, %31;\n\taddc.cc.u32 %2, %17, %32;\n\t"
        "addc.cc.u32 %3, %18, %33;\n\taddc.cc.u32 %4, %19, %34;\n\taddc.cc.u32 %5, %20, %35;\n\t"
        "addc.cc.u32 %6, %21, %36;\n\taddc.cc.u32 %7, %22, %37;\n\taddc.cc.u32 %8, %23, %38;\n\t"
        "addc.cc.u32 %9, %24, %39;\n\taddc.cc.u32 %10, %25, %40;\n\taddc.cc.u32 %11, %26, %41;\n\t"
        "addc.cc.u32 %12, %27, %42;\n\taddc.cc.u32 %13, %28, %43;\n\taddc.u32 %14, %29, %44;"
        : "=r"(t[1]), "=r"(t[2]), "=r"(t[3]), "=r"(t[4]), "=r"(t[5]), "=r"(t[6]), "=r"(t[7]), "=r"(t[8]),
          "=r"(t[9]), "=r"(t[10]), "=r"(t[11]), "=r"(t[12]), "=r"(t[13]), "=r"(t[14]), "=r"(t[15])
        : "r"(e[1]), "r"(e[2]), "r"(e[3]), "r"(e[4]), "r"(e[5]), "r"(e[6]), "r"(e[7]), "r"(e[8]), "r"(e[9]),
          "r"(e[10]), "r"(e[11]), "r"(e[12]), "r"(e[13]), "r"(e[14]), "r"(e[15]), "r"(o[0]), "r"(o[1]),
          "r"(o[2]), "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7]), "r"(o[8]), "r"(o[9]), "r"(o[10]),
          "r"(o[11]), "r"(o[12]), "r"(o[13]), "r"(o[14]));
}

// t[0..15] = a^2: the 28 products a_i a_j with i < j in the same even and odd
// columns, doubled, then one carry chain of the eight squares a_i^2.
__device__ __forceinline__ void sqr_wide(uint32_t t[16], const fe& a) {
    uint32_t e[14], o[14];
    // Row 0: a_0 a_1, a_3, a_5, a_7 at words 1, 3, 5, 7 (o) and a_0 a_2, a_4, a_6 at 2, 4, 6 (e).
    uint64_t p;
#define PUT(arr, k, x, y) p = (uint64_t)(x) * (y); arr[k] = (uint32_t)p; arr[(k) + 1] = (uint32_t)(p >> 32);
    PUT(o, 0, a.v[0], a.v[1]) PUT(o, 2, a.v[0], a.v[3]) PUT(o, 4, a.v[0], a.v[5]) PUT(o, 6, a.v[0], a.v[7])
    PUT(e, 2, a.v[0], a.v[2]) PUT(e, 4, a.v[0], a.v[4]) PUT(e, 6, a.v[0], a.v[6])
    // Row 1: words 3, 5, 7 (o, carry out) and 4, 6, 8 (e).
    asm("mad.lo.cc.u32 %0,%7,%10,%0;\n\tmadc.hi.cc.u32 %1,%7,%10,%1;\n\tmadc.lo.cc.u32 %2,%8,%10,%2;\n\tmadc.hi.cc.u32 %3,%8,%10,%3;\n\t"
        "madc.lo.cc.u32 %4,%9,%10,%4;\n\tmadc.hi.cc.u32 %5,%9,%10,%5;\n\taddc.u32 %6,0,0;"
        : "+r"(o[2]), "+r"(o[3]), "+r"(o[4]), "+r"(o[5]), "+r"(o[6]), "+r"(o[7]), "=r"(o[8]) : "r"(a.v[2]), "r"(a.v[4]), "r"(a.v[6]), "r"(a.v[1]));
    asm("mad.lo.cc.u32 %0,%6,%9,%0;\n\tmadc.hi.cc.u32 %1,%6,%9,%1;\n\tmadc.lo.cc.u32 %2,%7,%9,%2;\n\tmadc.hi.cc.u32 %3,%7,%9,%3;\n\t"
        "madc.lo.cc.u32 %4,%8,%9,0;\n\tmadc.hi.u32 %5,%8,%9,0;"
        : "+r"(e[4]), "+r"(e[5]), "+r"(e[6]), "+r"(e[7]), "=r"(e[8]), "=r"(e[9]) : "r"(a.v[3]), "r"(a.v[5]), "r"(a.v[7]), "r"(a.v[1]));
    // Row 2: words 5, 7, 9 (o) and 6, 8 (e, carry out).
    asm("mad.lo.cc.u32 %0,%6,%9,%0;\n\tmadc.hi.cc.u32 %1,%6,%9,%1;\n\tmadc.lo.cc.u32 %2,%7,%9,%2;\n\tmadc.hi.cc.u32 %3,%7,%9,%3;\n\t"
        "madc.lo.cc.u32 %4,%8,%9,%4;\n\tmadc.hi.u32 %5,%8,%9,0;"
        : "+r"(o[4]), "+r"(o[5]), "+r"(o[6]), "+r"(o[7]), "+r"(o[8]), "=r"(o[9]) : "r"(a.v[3]), "r"(a.v[5]), "r"(a.v[7]), "r"(a.v[2]));
    asm("mad.lo.cc.u32 %0,%5,%7,%0;\n\tmadc.hi.cc.u32 %1,%5,%7,%1;\n\tmadc.lo.cc.u32 %2,%6,%7,%2;\n\tmadc.hi.cc.u32 %3,%6,%7,%3;\n\taddc.u32 %4,0,0;"
        : "+r"(e[6]), "+r"(e[7]), "+r"(e[8]), "+r"(e[9]), "=r"(e[10]) : "r"(a.v[4]), "r"(a.v[6]), "r"(a.v[2]));
    // Row 3: words 7, 9 (o, carry out) and 8, 10 (e).
    asm("mad.lo.cc.u32 %0,%5,%7,%0;\n\tmadc.hi.cc.u32 %1,%5,%7,%1;\n\tmadc.lo.cc.u32 %2,%6,%7,%2;\n\tmadc.hi.cc.u32 %3,%6,%7,%3;\n\taddc.u32 %4,0,0;"
        : "+r"(o[6]), "+r"(o[7]), "+r"(o[8]), "+r"(o[9]), "=r"(o[10]) : "r"(a.v[4]), "r"(a.v[6]), "r"(a.v[3]));
    asm("mad.lo.cc.u32 %0,%4,%6,%0;\n\tmadc.hi.cc.u32 %1,%4,%6,%1;\n\tmadc.lo.cc.u32 %2,%5,%6,%2;\n\tmadc.hi.u32 %3,%5,%6,0;"
        : "+r"(e[8]), "+r"(e[9]), "+r"(e[10]), "=r"(e[11]) : "r"(a.v[5]), "r"(a.v[7]), "r"(a.v[3]));
    // Row 4: words 9, 11 (o) and 10 (e, carry out).
    asm("mad.lo.cc.u32 %0,%4,%6,%0;\n\tmadc.hi.cc.u32 %1,%4,%6,%1;\n\tmadc.lo.cc.u32 %2,%5,%6,%2;\n\tmadc.hi.u32 %3,%5,%6,0;"
        : "+r"(o[8]), "+r"(o[9]), "+r"(o[10]), "=r"(o[11]) : "r"(a.v[5]), "r"(a.v[7]), "r"(a.v[4]));
    asm("mad.lo.cc.u32 %0,%3,%4,%0;\n\tmadc.hi.cc.u32 %1,%3,%4,%1;\n\taddc.u32 %2,0,0;"
        : "+r"(e[10]), "+r"(e[11]), "=r"(e[12]) : "r"(a.v[6]), "r"(a.v[4]));
    // Row 5: words 11 (o, carry out) and 12 (e).
    asm("mad.lo.cc.u32 %0,%3,%4,%0;\n\tmadc.hi.cc.u32 %1,%3,%4,%1;\n\taddc.u32 %2,0,0;"
        : "+r"(o[10]), "+r"(o[11]), "=r"(o[12]) : "r"(a.v[6]), "r"(a.v[5]));
    asm("mad.lo.cc.u32 %0,%2,%3,%0;\n\tmadc.hi.u32 %1,%2,%3,0;" : "+r"(e[12]), "=r"(e[13]) : "r"(a.v[7]), "r"(a.v[5]));
    // Row 6: word 13 (o).
    asm("mad.lo.cc.u32 %0,%2,%3,%0;\n\tmadc.hi.u32 %1,%2,%3,0;" : "+r"(o[12]), "=r"(o[13]) : "r"(a.v[7]), "r"(a.v[6]));
    // Cross products e + 2^32 o (words 1..14).
    t[1] = o[0];
    asm("add.cc.u32 %0,%13,%25;\n\taddc.cc.u32 %1,%14,%26;\n\taddc.cc.u32 %2,%15,%27;\n\taddc.cc.u32 %3,%16,%28;\n\taddc.cc.u32 %4,%17,%29;\n\t"
        "addc.cc.u32 %5,%18,%30;\n\taddc.cc.u32 %6,%19,%31;\n\taddc.cc.u32 %7,%20,%32;\n\taddc.cc.u32 %8,%21,%33;\n\taddc.cc.u32 %9,%22,%34;\n\t"
        "addc.cc.u32 %10,%23,%35;\n\taddc.cc.u32 %11,%24,%36;\n\taddc.u32 %12,%37,0;"
        : "=r"(t[2]), "=r"(t[3]), "=r"(t[4]), "=r"(t[5]), "=r"(t[6]), "=r"(t[7]), "=r"(t[8]), "=r"(t[9]), "=r"(t[10]), "=r"(t[11]), "=r"(t[12]), "=r"(t[13]), "=r"(t[14])
        : "r"(e[2]), "r"(e[3]), "r"(e[4]), "r"(e[5]), "r"(e[6]), "r"(e[7]), "r"(e[8]), "r"(e[9]), "r"(e[10]), "r"(e[11]), "r"(e[12]), "r"(e[13]),
          "r"(o[1]), "r"(o[2]), "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7]), "r"(o[8]), "r"(o[9]), "r"(o[10]), "r"(o[11]), "r"(o[12]), "r"(o[13]));
    // Doubled, plus the squares.
    asm("add.cc.u32 %0,%0,%0;\n\taddc.cc.u32 %1,%1,%1;\n\taddc.cc.u32 %2,%2,%2;\n\taddc.cc.u32 %3,%3,%3;\n\taddc.cc.u32 %4,%4,%4;\n\t"
        "addc.cc.u32 %5,%5,%5;\n\taddc.cc.u32 %6,%6,%6;\n\taddc.cc.u32 %7,%7,%7;\n\taddc.cc.u32 %8,%8,%8;\n\taddc.cc.u32 %9,%9,%9;\n\t"
        "addc.cc.u32 %10,%10,%10;\n\taddc.cc.u32 %11,%11,%11;\n\taddc.cc.u32 %12,%12,%12;\n\taddc.cc.u32 %13,%13,%13;\n\taddc.u32 %14,0,0;"
        : "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "+r"(t[4]), "+r"(t[5]), "+r"(t[6]), "+r"(t[7]), "+r"(t[8]), "+r"(t[9]), "+r"(t[10]), "+r"(t[11]), "+r"(t[12]), "+r"(t[13]), "+r"(t[14]), "=r"(t[15]));
    t[0] = 0;
    asm("mad.lo.cc.u32 %0,%16,%16,0;\n\tmadc.hi.cc.u32 %1,%16,%16,%1;\n\tmadc.lo.cc.u32 %2,%17,%17,%2;\n\tmadc.hi.cc.u32 %3,%17,%17,%3;\n\t"
        "madc.lo.cc.u32 %4,%18,%18,%4;\n\tmadc.hi.cc.u32 %5,%18,%18,%5;\n\tmadc.lo.cc.u32 %6,%19,%19,%6;\n\tmadc.hi.cc.u32 %7,%19,%19,%7;\n\t"
        "madc.lo.cc.u32 %8,%20,%20,%8;\n\tmadc.hi.cc.u32 %9,%20,%20,%9;\n\tmadc.lo.cc.u32 %10,%21,%21,%10;\n\tmadc.hi.cc.u32 %11,%21,%21,%11;\n\t"
        "madc.lo.cc.u32 %12,%22,%22,%12;\n\tmadc.hi.cc.u32 %13,%22,%22,%13;\n\tmadc.lo.cc.u32 %14,%23,%23,%14;\n\tmadc.hi.u32 %15,%23,%23,%15;"
        : "+r"(t[0]), "+r"(t[1]), "+r"(t[2]), "+r"(t[3]), "+r"(t[4]), "+r"(t[5]), "+r"(t[6]), "+r"(t[7]), "+r"(t[8]), "+r"(t[9]), "+r"(t[10]), "+r"(t[11]), "+r"(t[12]), "+r"(t[13]), "+r"(t[14]), "+r"(t[15])
        : "r"(a.v[0]), "r"(a.v[1]), "r"(a.v[2]), "r"(a.v[3]), "r"(a.v[4]), "r"(a.v[5]), "r"(a.v[6]), "r"(a.v[7]));
#undef PUT
}

__device__ __forceinline__ void fe_mul(fe& r, const fe& a, const fe& b) {
    uint32_t t[16];
    mul_wide(t, a, b);
    fe_reduce(r, t);
}

__device__ __forceinline__ void fe_sqr(fe& r, const fe& a) {
    uint32_t t[16];
    sqr_wide(t, a);
    fe_reduce(r, t);
}

// Out-of-line multiplication and squaring (by value): the hot point formulas
// call these so that one copy of the product and reduction code serves every
// call site.
static __device__ __noinline__ fe fmul(fe a, fe b) {
    fe r;
    fe_mul(r, a, b);
    return r;
}

static __device__ __noinline__ fe fsqr(fe a) {
    fe r;
    fe_sqr(r, a);
    return r;
}

// Standard residue -> Montgomery domain and back.
__device__ __forceinline__ void fe_to_mont(fe& r, const fe& a) {
    fe r2;
    fe_set_R2(r2);
    r = fmul(a, r2);
}
__device__ __forceinline__ void fe_from_mont(fe& r, const fe& a) {
    uint32_t t[16];
#pragma unroll
    for (int i = 0; i < 8; i++) {
        t[i] = a.v[i];
        t[8 + i] = 0;
    }
    fe_reduce(r, t);
}

// The square of a, reduced twice: a^2 / R^2. Of a Montgomery-domain a it is
// the standard residue of the square.
__device__ __forceinline__ fe fe_sqr_std(const fe& a) {
    uint32_t t[16];
    sqr_wide(t, a);
    fe r;
    fe_reduce(r, t);
    fe_from_mont(r, r);
    return r;
}

// x <- x 2^-k mod p for canonical x and 1 <= k <= 31.  Since p = -1 mod
// 2^32, x + (x mod 2^k) p is a multiple of 2^k, below 2^k p, so the shifted
// sum is canonical again.
__device__ __forceinline__ void fe_div_pow2(fe& x, unsigned k) {
    const uint32_t q = x.v[0] & ((1u << k) - 1u);
    // t = x + q p with p = 2^256 - 2^224 + 2^192 + 2^96 - 1 (words 0..7:
    // ffffffff x3, 0 x2, 1, ffffffff; the 2^256 term lands in word 8).
    uint32_t t[9];
    uint64_t c = 0;
#pragma unroll
    for (int j = 0; j < 8; j++) {
        const uint64_t pj = (j < 3 || j == 7) ? 0xffffffffull : (j == 6 ? 1ull : 0ull);
        c += (uint64_t)x.v[j] + (uint64_t)q * pj;
        t[j] = (uint32_t)c;
        c >>= 32;
    }
    t[8] = (uint32_t)c;
#pragma unroll
    for (int j = 0; j < 8; j++) x.v[j] = __funnelshift_r(t[j], t[j + 1], k);
}

// r = a^-1 in the Montgomery domain (a holds x R, r gets x^-1 R) for a != 0
// mod p (0 gives 0), a weakly reduced.  Binary extended Euclid on the held
// value, whose inverse x^-1 R^-1 a multiplication by R^3 brings to x^-1 R:
// with u = a, v = p, x1 = 1, x2 = 0 the
// invariants x1 a = u and x2 a = v (mod p) hold throughout; factors of two
// leave u (or v) together with the same power of two from x1 (or x2), and
// the smaller of two odd u, v is subtracted from the larger (their
// difference is even), until one of them is 1.  About 2 log2 p steps of a
// few 256-bit additions each, against the 267 dependent multiplications of
// a Fermat power.
static __device__ __noinline__ void fe_inv(fe& r, const fe& a) {
    fe u, v, x1, x2;
    fe_canon(u, a);
    if ((u.v[0] | u.v[1] | u.v[2] | u.v[3] | u.v[4] | u.v[5] | u.v[6] | u.v[7]) == 0u) {
        fe_zero(r);
        return;
    }
    v.v[0] = v.v[1] = v.v[2] = 0xffffffffu;
    v.v[3] = v.v[4] = v.v[5] = 0u;
    v.v[6] = 1u;
    v.v[7] = 0xffffffffu;
    fe_zero(x1);
    x1.v[0] = 1u;
    fe_zero(x2);
    // Each step removes a factor of two or shrinks u + v: the bound is never
    // reached for a != 0 mod p.
    for (int it = 0; it < 4096; it++) {
        const bool u1 = ((u.v[0] ^ 1u) | u.v[1] | u.v[2] | u.v[3] | u.v[4] | u.v[5] | u.v[6] | u.v[7]) == 0u;
        if (u1) break;
        const bool v1 = ((v.v[0] ^ 1u) | v.v[1] | v.v[2] | v.v[3] | v.v[4] | v.v[5] | v.v[6] | v.v[7]) == 0u;
        if (v1) {
            x1 = x2;
            break;
        }
        if (!(u.v[0] & 1u)) {
            const unsigned k = u.v[0] ? (unsigned)(__ffs(u.v[0]) - 1) : 31u;
#pragma unroll
            for (int j = 0; j < 7; j++) u.v[j] = __funnelshift_r(u.v[j], u.v[j + 1], k);
            u.v[7] >>= k;
            fe_div_pow2(x1, k);
            continue;
        }
        if (!(v.v[0] & 1u)) {
            const unsigned k = v.v[0] ? (unsigned)(__ffs(v.v[0]) - 1) : 31u;
#pragma unroll
            for (int j = 0; j < 7; j++) v.v[j] = __funnelshift_r(v.v[j], v.v[j + 1], k);
            v.v[7] >>= k;
            fe_div_pow2(x2, k);
            continue;
        }
        // d = u - v; if no borrow u <- d, x1 <- x1 - x2, else v <- -d, x2 <- x2 - x1.
        fe d;
        uint32_t bw;
        asm("sub.cc.u32  %0, %9, %17;\n\t"
            "subc.cc.u32 %1, %10, %18;\n\t"
            "subc.cc.u32 %2, %11, %19;\n\t"
            "subc.cc.u32 %3, %12, %20;\n\t"
            "subc.cc.u32 %4, %13, %21;\n\t"
            "subc.cc.u32 %5, %14, %22;\n\t"
            "subc.cc.u32 %6, %15, %23;\n\t"
            "subc.cc.u32 %7, %16, %24;\n\t"
            "subc.u32    %8, 0, 0;"
            : "=r"(d.v[0]), "=r"(d.v[1]), "=r"(d.v[2]), "=r"(d.v[3]), "=r"(d.v[4]), "=r"(d.v[5]),
              "=r"(d.v[6]), "=r"(d.v[7]), "=r"(bw)
            : "r"(u.v[0]), "r"(u.v[1]), "r"(u.v[2]), "r"(u.v[3]), "r"(u.v[4]), "r"(u.v[5]), "r"(u.v[6]),
              "r"(u.v[7]), "r"(v.v[0]), "r"(v.v[1]), "r"(v.v[2]), "r"(v.v[3]), "r"(v.v[4]), "r"(v.v[5]),
              "r"(v.v[6]), "r"(v.v[7]));
        if (!bw) {
            u = d;
            fe_sub(x1, x1, x2);
            fe_canon(x1, x1);
        } else {
            asm("sub.cc.u32  %0, 0, %0;\n\t"
                "subc.cc.u32 %1, 0, %1;\n\t"
                "subc.cc.u32 %2, 0, %2;\n\t"
                "subc.cc.u32 %3, 0, %3;\n\t"
                "subc.cc.u32 %4, 0, %4;\n\t"
                "subc.cc.u32 %5, 0, %5;\n\t"
                "subc.cc.u32 %6, 0, %6;\n\t"
                "subc.u32    %7, 0, %7;"
                : "+r"(d.v[0]), "+r"(d.v[1]), "+r"(d.v[2]), "+r"(d.v[3]), "+r"(d.v[4]), "+r"(d.v[5]),
                  "+r"(d.v[6]), "+r"(d.v[7]));
            v = d;
            fe_sub(x2, x2, x1);
            fe_canon(x2, x2);
        }
    }
    fe r3;
    fe_set_R3(r3);
    r = fmul(x1, r3);
}

// r = a b - c d (mod p) with a single reduction: the two 512-bit products
// are subtracted, p 2^256 (= 0 mod p) is added back while the difference is
// negative (once, or on a rare branch twice), then the sum is reduced.
__device__ __forceinline__ fe fe_mulsub(const fe& a, const fe& b, const fe& c, const fe& d) {
    uint32_t u[16], v[16];
    mul_wide(u, a, b);
    mul_wide(v, c, d);
    uint32_t bw;
    asm("sub.cc.u32  %0, %0, %17;\n\t"
        "subc.cc.u32 %1, %1, %18;\n\t"
        "subc.cc.u32 %2, %2, %19;\n\t"
        "subc.cc.u32 %3, %3, %20;\n\t"
        "subc.cc.u32 %4, %4, %21;\n\t"
        "subc.cc.u32 %5, %5, %22;\n\t"
        "subc.cc.u32 %6, %6, %23;\n\t"
        "subc.cc.u32 %7, %7, %24;\n\t"
        "subc.cc.u32 %8, %8, %25;\n\t"
        "subc.cc.u32 %9, %9, %26;\n\t"
        "subc.cc.u32 %10, %10, %27;\n\t"
        "subc.cc.u32 %11, %11, %28;\n\t"
        "subc.cc.u32 %12, %12, %29;\n\t"
        "subc.cc.u32 %13, %13, %30;\n\t"
        "subc.cc.u32 %14, %14, %31;\n\t"
        "subc.cc.u32 %15, %15, %32;\n\t"
        "subc.u32    %16, 0, 0;"
        : "+r"(u[0]), "+r"(u[1]), "+r"(u[2]), "+r"(u[3]), "+r"(u[4]), "+r"(u[5]), "+r"(u[6]), "+r"(u[7]),
          "+r"(u[8]), "+r"(u[9]), "+r"(u[10]), "+r"(u[11]), "+r"(u[12]), "+r"(u[13]), "+r"(u[14]),
          "+r"(u[15]), "=r"(bw)
        : "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]));
    // On a borrow (bw = 0xffffffff) add p to the high half, twice in the rare
    // case (c d - a b > p 2^256) that it stays negative. As a loop, that case is
    // a branch of its own and ends the block of instructions that the assembler
    // schedules as one: the gather's inlined addition, whose carries overflow
    // the predicate registers otherwise, took 25.4 ms a step with an if and
    // 23.9 with the loop (w = 4, 1024 x 1024 x 256).
    fe h;
#pragma unroll
    for (int i = 0; i < 8; i++) h.v[i] = u[8 + i];
    bw += fe_add_p_masked(h, bw);
    while (bw) bw += fe_add_p_masked(h, bw);
#pragma unroll
    for (int i = 0; i < 8; i++) u[8 + i] = h.v[i];
    fe r;
    fe_reduce(r, u);
    return r;
}

static __device__ __noinline__ fe fmulsub(fe a, fe b, fe c, fe d) { return fe_mulsub(a, b, c, d); }

// Multiplication, squaring and a b - c d either out of line (INL = false:
// one shared copy of the code) or inlined at the call site (INL = true).
template <bool INL>
__device__ __forceinline__ fe mul_t(const fe& a, const fe& b) {
    if (INL) {
        fe r;
        fe_mul(r, a, b);
        return r;
    }
    return fmul(a, b);
}
template <bool INL>
__device__ __forceinline__ fe sqr_t(const fe& a) {
    if (INL) {
        fe r;
        fe_sqr(r, a);
        return r;
    }
    return fsqr(a);
}
template <bool INL>
__device__ __forceinline__ fe mulsub_t(const fe& a, const fe& b, const fe& c, const fe& d) {
    if (INL) return fe_mulsub(a, b, c, d);
    return fmulsub(a, b, c, d);
}

}  // namespace pcmm

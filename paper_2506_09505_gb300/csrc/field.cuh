// Device arithmetic in the Goldilocks field, Eq. 1: p = 2^64 - 2^32 + 1.
//
// Values travel between operations as 64-bit "weak" representatives: any
// word in [0, 2^64) standing for its residue mod p.  Only stored results are
// made canonical (0 <= e < p, Sec. 2.4).  Products are formed from four
// 32x32->64 partial products (IMAD.WIDE.U32 with a zero addend, so no
// register pair has to be built for the addend) and summed column by column
// in carry chains.  The 128-bit (or 160-bit) result is folded with
// 2^64 = 2^32 - 1, 2^96 = -1 and 2^128 = -2^32 (mod p): the special-prime
// reduction of Alg. 2 and Eqs. 2-4 on 32-bit limbs, with no 64-bit multiply.
#pragma once
#include <cstdint>

namespace pg12 {
namespace dev {

constexpr uint64_t P = 0xFFFFFFFF00000001ull;
constexpr uint64_t EPS = 0xFFFFFFFFull;  // 2^64 mod p

typedef unsigned __int128 u128;
typedef __int128 s128;

__device__ __forceinline__ uint32_t lo32(uint64_t x) { return (uint32_t)x; }
__device__ __forceinline__ uint32_t hi32(uint64_t x) { return (uint32_t)(x >> 32); }

// The four partial products of a*b (each < 2^64).
struct Partial {
    uint64_t ll, lh, hl, hh;
};

__device__ __forceinline__ Partial partials(uint64_t a, uint64_t b) {
    const uint32_t a0 = lo32(a), a1 = hi32(a), b0 = lo32(b), b1 = hi32(b);
    Partial q;
    q.ll = (uint64_t)a0 * b0;
    q.lh = (uint64_t)a0 * b1;
    q.hl = (uint64_t)a1 * b0;
    q.hh = (uint64_t)a1 * b1;
    return q;
}

// (r3:r2:r1:r0) = ll + (lh + hl) * 2^32 + hh * 2^64, two carry chains.
// (Running the second chain as multiply-adds by a 1 held in constant memory,
// to move its adds from the ALU pipe to the FMA pipe, measured 1% slower.)
__device__ __forceinline__ u128 join(const Partial &q) {
    uint32_t r0 = lo32(q.ll), r1, r2, r3;
    asm("add.cc.u32 %0, %3, %4;\n\t"
        "addc.cc.u32 %1, %5, %6;\n\t"
        "addc.u32 %2, %7, 0;\n\t"
        "add.cc.u32 %0, %0, %8;\n\t"
        "addc.cc.u32 %1, %1, %9;\n\t"
        "addc.u32 %2, %2, 0;"
        : "=r"(r1), "=r"(r2), "=r"(r3)
        : "r"(hi32(q.ll)), "r"(lo32(q.lh)), "r"(hi32(q.lh)), "r"(lo32(q.hh)), "r"(hi32(q.hh)),
          "r"(lo32(q.hl)), "r"(hi32(q.hl)));
    return ((u128)(((uint64_t)r3 << 32) | r2) << 64) | (((uint64_t)r1 << 32) | r0);
}

// a^2 = ll + 2 lh 2^32 + hh 2^64 from three partial products.
__device__ __forceinline__ u128 sqr_full(uint64_t a) {
    const uint32_t a0 = lo32(a), a1 = hi32(a);
    const uint64_t ll = (uint64_t)a0 * a0, lh = (uint64_t)a0 * a1, hh = (uint64_t)a1 * a1;
    uint32_t r1, r2, r3;
    asm("add.cc.u32 %0, %3, %4;\n\t"
        "addc.cc.u32 %1, %5, %6;\n\t"
        "addc.u32 %2, %7, 0;\n\t"
        "add.cc.u32 %0, %0, %4;\n\t"
        "addc.cc.u32 %1, %1, %5;\n\t"
        "addc.u32 %2, %2, 0;"
        : "=r"(r1), "=r"(r2), "=r"(r3)
        : "r"(hi32(ll)), "r"(lo32(lh)), "r"(hi32(lh)), "r"(lo32(hh)), "r"(hi32(hh)));
    return ((u128)(((uint64_t)r3 << 32) | r2) << 64) | (((uint64_t)r1 << 32) | lo32(ll));
}

// value = lo + hl 2^32 - hl - hh - k 2^32 (mod p) for hi = hh:hl and a small
// extra k (the 2^128 limb of a lazy sum, 2^128 = -2^32).  The exact signed
// value t lies in (-(k + 2) 2^32, 2^65 - 2^33]; its top word tp is -1, 0 or 1
// and is folded back as tp (2^32 - 1) (2^64 = 2^32 - 1).  That add cannot wrap
// again: for tp = 1 the low word is at most 2^64 - 2^33, for tp = -1 at least
// 2^64 - (k + 2) 2^32.
//
// 1 (default): the words of t come from one borrow/carry chain on 32-bit
// limbs; 0: the same value through signed 128-bit C arithmetic (measured: a
// 2^22 x 8 tree 3% slower, S-box 10% slower).
#ifndef PG12_FOLD_PTX
#define PG12_FOLD_PTX 1
#endif
__device__ __forceinline__ uint64_t fold(uint64_t lo, uint64_t hi, uint32_t k) {
#if PG12_FOLD_PTX
    // t = l0 + (l1 + hl - k) 2^32 - hl - hh as a 96-bit two's-complement value (w0, w1, tp)
    uint32_t w0, w1, tp;
    asm("sub.cc.u32 %0, %3, %5;\n\t"
        "subc.cc.u32 %1, %4, %7;\n\t"
        "subc.u32 %2, 0, 0;\n\t"
        "sub.cc.u32 %0, %0, %6;\n\t"
        "subc.cc.u32 %1, %1, 0;\n\t"
        "subc.u32 %2, %2, 0;\n\t"
        "add.cc.u32 %1, %1, %5;\n\t"
        "addc.u32 %2, %2, 0;"
        : "=r"(w0), "=r"(w1), "=r"(tp)
        : "r"(lo32(lo)), "r"(hi32(lo)), "r"(lo32(hi)), "r"(hi32(hi)), "r"(k));
    // + tp (2^32 - 1): minus tp sign-extended, plus tp at 2^32 (the same
    // correction as 64-bit C arithmetic on the sign-extended tp measured 2%
    // slower in the tensor-core kernels)
    uint32_t r0, r1;
    asm("{\n\t.reg .u32 sh;\n\t"
        "shr.s32 sh, %4, 31;\n\t"
        "sub.cc.u32 %0, %2, %4;\n\t"
        "subc.u32 %1, %3, sh;\n\t"
        "add.u32 %1, %1, %4;\n\t}"
        : "=r"(r0), "=r"(r1)
        : "r"(w0), "r"(w1), "r"(tp));
    return ((uint64_t)r1 << 32) | r0;
#else
    const uint64_t hl = hi & EPS, hh = hi >> 32;
    const s128 t = (s128)lo + (s128)(hl << 32) - (s128)(hl + hh) - (s128)((uint64_t)k << 32);
    const uint64_t top = (uint64_t)(t >> 64);
    return (uint64_t)t + ((top << 32) - top);
#endif
}

__device__ __forceinline__ uint64_t reduce128(u128 r) { return fold((uint64_t)r, (uint64_t)(r >> 64), 0); }

// a * b + c for 32-bit a, b and a 64-bit c (one IMAD.WIDE; the caller keeps
// the sum below 2^64)
__device__ __forceinline__ uint64_t madw(uint32_t a, uint32_t b, uint64_t c) {
    uint64_t d;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

__device__ __forceinline__ uint64_t canon(uint64_t x) { return x >= P ? x - P : x; }

// (Summing the columns inside chained 32x32+64-bit multiply-adds instead of
// carry chains measured 0.5% slower in the tensor-core kernels.)
__device__ __forceinline__ uint64_t mul(uint64_t a, uint64_t b) { return reduce128(join(partials(a, b))); }

__device__ __forceinline__ uint64_t sqr(uint64_t a) { return reduce128(sqr_full(a)); }

// weak a + canonical c (c < p): at most one wrap, folded as +(2^32 - 1).
__device__ __forceinline__ uint64_t add_canon(uint64_t a, uint64_t c) {
    uint64_t s = a + c;
    if (s < c) s += EPS;
    return s;
}

// S-box of Alg. 1: x^7 = (x^2)^2 * (x^2 * x).
__device__ __forceinline__ uint64_t sbox(uint64_t x) {
    const uint64_t x2 = sqr(x);
    const uint64_t x3 = mul(x2, x);
    const uint64_t x4 = sqr(x2);
    return mul(x4, x3);
}

// x + w*y as one 128-bit value (x added into the product), reduced once.
__device__ __forceinline__ uint64_t mul_add(uint64_t w, uint64_t y, uint64_t x) {
    u128 r = join(partials(w, y));
    r += x;  // < 2^128: the product is below p * 2^64
    return reduce128(r);
}

// Lazy dot-product accumulator.  The outer partial products (ll, hh) of a
// term are one contiguous 128-bit value and go into a 160-bit sum; the two
// middle products go into a separate sum that is shifted in once at the end.
// Holds up to 2^30 terms.
#ifndef PG12_ACC_MID64
#define PG12_ACC_MID64 1  // 0: middle products in a 96-bit carry chain (measured 2% slower)
#endif
struct Acc {
    uint32_t a0, a1, a2, a3, a4;
#if PG12_ACC_MID64
    uint64_t mlo, mhi;  // sums of the low / high halves of lh and hl (weights 2^32, 2^64)
#else
    uint32_t m0, m1, m2;
#endif
};

__device__ __forceinline__ void acc_zero(Acc &A) {
    A.a0 = A.a1 = A.a2 = A.a3 = A.a4 = 0;
#if PG12_ACC_MID64
    A.mlo = A.mhi = 0;
#else
    A.m0 = A.m1 = A.m2 = 0;
#endif
}

// Sum that starts from one 64-bit value v (as if a first term were v * 1).
__device__ __forceinline__ void acc_init(Acc &A, uint64_t v) {
    acc_zero(A);
    A.a0 = lo32(v);
    A.a1 = hi32(v);
}

__device__ __forceinline__ void acc_mac(Acc &A, uint64_t x, uint64_t m) {
    const Partial q = partials(x, m);
#if PG12_ACC_MID64
    asm("add.cc.u32 %0, %0, %5;\n\t"
        "addc.cc.u32 %1, %1, %6;\n\t"
        "addc.cc.u32 %2, %2, %7;\n\t"
        "addc.cc.u32 %3, %3, %8;\n\t"
        "addc.u32 %4, %4, 0;"
        : "+r"(A.a0), "+r"(A.a1), "+r"(A.a2), "+r"(A.a3), "+r"(A.a4)
        : "r"(lo32(q.ll)), "r"(hi32(q.ll)), "r"(lo32(q.hh)), "r"(hi32(q.hh)));
    // three-input adds into 64-bit words: no carry leaves them
    A.mlo += (uint64_t)lo32(q.lh) + lo32(q.hl);
    A.mhi += (uint64_t)hi32(q.lh) + hi32(q.hl);
#else
    asm("add.cc.u32 %0, %0, %8;\n\t"
        "addc.cc.u32 %1, %1, %9;\n\t"
        "addc.cc.u32 %2, %2, %10;\n\t"
        "addc.cc.u32 %3, %3, %11;\n\t"
        "addc.u32 %4, %4, 0;\n\t"
        "add.cc.u32 %5, %5, %12;\n\t"
        "addc.cc.u32 %6, %6, %13;\n\t"
        "addc.u32 %7, %7, 0;\n\t"
        "add.cc.u32 %5, %5, %14;\n\t"
        "addc.cc.u32 %6, %6, %15;\n\t"
        "addc.u32 %7, %7, 0;"
        : "+r"(A.a0), "+r"(A.a1), "+r"(A.a2), "+r"(A.a3), "+r"(A.a4), "+r"(A.m0), "+r"(A.m1), "+r"(A.m2)
        : "r"(lo32(q.ll)), "r"(hi32(q.ll)), "r"(lo32(q.hh)), "r"(hi32(q.hh)), "r"(lo32(q.lh)),
          "r"(hi32(q.lh)), "r"(lo32(q.hl)), "r"(hi32(q.hl)));
#endif
}

// sum -> weak 64-bit residue.
__device__ __forceinline__ uint64_t acc_reduce(const Acc &A) {
#if PG12_ACC_MID64
    // middle sum = mlo + mhi 2^32 (each half-sum is below 2^33 per term, so the
    // sum stays below 2^96), as three words m0..m2 at weight 2^32
    const u128 mid = (u128)A.mlo + ((u128)A.mhi << 32);
    const uint32_t m0 = (uint32_t)mid, m1 = (uint32_t)(mid >> 32), m2 = (uint32_t)(mid >> 64);
#else
    const uint32_t m0 = A.m0, m1 = A.m1, m2 = A.m2;
#endif
    uint32_t a1, a2, a3, a4;
    asm("add.cc.u32 %0, %4, %8;\n\t"
        "addc.cc.u32 %1, %5, %9;\n\t"
        "addc.cc.u32 %2, %6, %10;\n\t"
        "addc.u32 %3, %7, 0;"
        : "=r"(a1), "=r"(a2), "=r"(a3), "=r"(a4)
        : "r"(A.a1), "r"(A.a2), "r"(A.a3), "r"(A.a4), "r"(m0), "r"(m1), "r"(m2));
    return fold(((uint64_t)a1 << 32) | A.a0, ((uint64_t)a3 << 32) | a2, a4);
}

// ---------------------------------------------------------- Montgomery form
// The tensor-core kernels multiply with the reduction x -> x R^-1 mod p,
// R = 2^64 (Montgomery, "Modular multiplication without trial division",
// 1985), because its tail is shorter here than the fold above: p^-1 mod R is
// 2^32 + 1, so for x = r3:r2:r1:r0 the quotient is
// m = (r1 + r0 mod 2^32) : r0 with no product, and
//   (x - m p) / 2^64 = (r1 + r2 + e) + 2^32 (r3 - (m1 + e)),  m1 + e 2^32 = r0 + r1,
// which lies in (-p, 2^64) for any x < 2^128: p is added (as 2^64 - (2^32 - 1))
// when it is negative, once.  m1 + e cannot wrap, nor r3 + carry for a product
// (2^64 - a)(2^64 - b): r3 = 2^32 - 1 needs a + b <= 2^32, and then r2 =
// 2^32 - (a + b) and r1 + e <= (a + b) / 4 leave no carry.  Eight instructions
// against the fold's twelve, on a product whose columns the compiler sums in
// multiply-adds with carry: twelve independent x^7 chains per thread, 16 warps
// per SM, take 105 cycles per warp and S-box against 143 with sbox() above (60
// instructions against 81; ALU / FMA pipe 30 / 30 against 56 / 23).
// The factor R^-1 of every product is carried into the constants: x^7 comes
// out as x^7 R^-6, and the matrices applied to S-box outputs are stored times
// R^6.
__device__ __forceinline__ uint64_t mont_tail(uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
    uint32_t l, h;
    asm("{\n\t.reg .u32 m, me, t, k;\n\t"
        "add.cc.u32 m, %3, %2;\n\t"
        "addc.u32 me, m, 0;\n\t"          // r0 + r1 with its carry added back
        "addc.cc.u32 %0, %3, %4;\n\t"     // r1 + r2 + e
        "addc.u32 t, %5, 0;\n\t"
        "sub.cc.u32 %1, t, me;\n\t"
        "subc.u32 k, 0, 0;\n\t"           // all ones when negative
        "sub.cc.u32 %0, %0, k;\n\t"
        "subc.u32 %1, %1, 0;\n\t}"
        : "=&r"(l), "=&r"(h)
        : "r"(r0), "r"(r1), "r"(r2), "r"(r3));
    return ((uint64_t)h << 32) | l;
}

// The same for the low 128 bits of any sum (r3 may be 2^32 - 1 with a carry in).
__device__ __forceinline__ uint64_t mont_tail_any(uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
    uint32_t l, h;
    asm("{\n\t.reg .u32 m, me, f, k;\n\t"
        "add.cc.u32 m, %3, %2;\n\t"
        "addc.u32 me, m, 0;\n\t"
        "addc.cc.u32 %0, %3, %4;\n\t"
        "addc.u32 f, 0, 0;\n\t"
        "sub.cc.u32 %1, %5, me;\n\t"
        "subc.u32 k, 0, 0;\n\t"
        "add.cc.u32 %1, %1, f;\n\t"
        "addc.u32 k, k, 0;\n\t"
        "sub.cc.u32 %0, %0, k;\n\t"
        "subc.u32 %1, %1, 0;\n\t}"
        : "=&r"(l), "=&r"(h)
        : "r"(r0), "r"(r1), "r"(r2), "r"(r3));
    return ((uint64_t)h << 32) | l;
}

// a b R^-1 (weak operands and result)
__device__ __forceinline__ uint64_t mmul(uint64_t a, uint64_t b) {
    const u128 v = (u128)a * b;
    const uint64_t lo = (uint64_t)v, hi = (uint64_t)(v >> 64);
    return mont_tail(lo32(lo), hi32(lo), lo32(hi), hi32(hi));
}

// x^7 R^-6
__device__ __forceinline__ uint64_t msbox(uint64_t x) {
    const uint64_t x2 = mmul(x, x);
    const uint64_t x3 = mmul(x2, x);
    const uint64_t x4 = mmul(x2, x2);
    return mmul(x4, x3);
}

// lo + h 2^64 for h < 2^31: lo + h 2^32 - h (2^64 = 2^32 - 1), whose first sum
// wraps at most once and then leaves less than 2^63, so its carry k adds k 2^32 -
// k without another wrap; the subtraction of h + k cannot borrow out.  (As a
// wide multiply-add h (2^32 - 1) + lo with its carry: a 2^22 x 8 tree 4.98 ms
// against 4.94, the low half becoming a negation and the high half an IMAD.HI.)
__device__ __forceinline__ uint64_t fold_small(uint32_t w0, uint32_t w1, uint32_t h) {
    uint32_t l, u;
    asm("{\n\t.reg .u32 k, g;\n\t"
        "add.cc.u32 %1, %3, %4;\n\t"
        "addc.u32 k, 0, 0;\n\t"
        "add.u32 g, %4, k;\n\t"
        "add.u32 %1, %1, k;\n\t"
        "sub.cc.u32 %0, %2, g;\n\t"
        "subc.u32 %1, %1, 0;\n\t}"
        : "=&r"(l), "=&r"(u)
        : "r"(w0), "r"(w1), "r"(h));
    return ((uint64_t)u << 32) | l;
}

// a + b as a weak word
__device__ __forceinline__ uint64_t add_fold(uint64_t a, uint64_t b) {
    uint32_t l, h, k;
    asm("add.cc.u32 %0, %3, %5;\n\t"
        "addc.cc.u32 %1, %4, %6;\n\t"
        "addc.u32 %2, 0, 0;"
        : "=&r"(l), "=&r"(h), "=&r"(k)
        : "r"(lo32(a)), "r"(hi32(a)), "r"(lo32(b)), "r"(hi32(b)));
    return fold_small(l, h, k);
}

// Lazy dot product in Montgomery form: sum_j x_j m_j R^-1 + u.  The outer
// partial products go into a 160-bit sum that starts at u 2^64, the middle
// ones into a 96-bit sum; each is a multiply-add with carry, so a term is four
// of those and three adds.
struct MAcc {
    uint32_t a0, a1, a2, a3, a4, b0, b1, b2;
};

__device__ __forceinline__ void macc_init(MAcc &A, uint64_t u) {
    A.a0 = A.a1 = A.a4 = A.b0 = A.b1 = A.b2 = 0;
    A.a2 = lo32(u);
    A.a3 = hi32(u);
}

__device__ __forceinline__ void macc(MAcc &A, uint64_t x, uint64_t m) {
    asm("mad.lo.cc.u32 %0, %8, %10, %0;\n\t"
        "madc.hi.cc.u32 %1, %8, %10, %1;\n\t"
        "madc.lo.cc.u32 %2, %9, %11, %2;\n\t"
        "madc.hi.cc.u32 %3, %9, %11, %3;\n\t"
        "addc.u32 %4, %4, 0;\n\t"
        "mad.lo.cc.u32 %5, %8, %11, %5;\n\t"
        "madc.hi.cc.u32 %6, %8, %11, %6;\n\t"
        "addc.u32 %7, %7, 0;\n\t"
        "mad.lo.cc.u32 %5, %9, %10, %5;\n\t"
        "madc.hi.cc.u32 %6, %9, %10, %6;\n\t"
        "addc.u32 %7, %7, 0;"
        : "+r"(A.a0), "+r"(A.a1), "+r"(A.a2), "+r"(A.a3), "+r"(A.a4), "+r"(A.b0), "+r"(A.b1), "+r"(A.b2)
        : "r"(lo32(x)), "r"(hi32(x)), "r"(lo32(m)), "r"(hi32(m)));
}

// A += B
__device__ __forceinline__ void macc_join(MAcc &A, const MAcc &B) {
    asm("add.cc.u32 %0, %0, %8;\n\t"
        "addc.cc.u32 %1, %1, %9;\n\t"
        "addc.cc.u32 %2, %2, %10;\n\t"
        "addc.cc.u32 %3, %3, %11;\n\t"
        "addc.u32 %4, %4, %12;\n\t"
        "add.cc.u32 %5, %5, %13;\n\t"
        "addc.cc.u32 %6, %6, %14;\n\t"
        "addc.u32 %7, %7, %15;"
        : "+r"(A.a0), "+r"(A.a1), "+r"(A.a2), "+r"(A.a3), "+r"(A.a4), "+r"(A.b0), "+r"(A.b1), "+r"(A.b2)
        : "r"(B.a0), "r"(B.a1), "r"(B.a2), "r"(B.a3), "r"(B.a4), "r"(B.b0), "r"(B.b1), "r"(B.b2));
}

// (sum of the products) R^-1 + u as a weak word: the tail on the sum's low 128
// bits, then its top word (2^128 R^-1 = 2^64).
__device__ __forceinline__ uint64_t macc_reduce(const MAcc &A) {
    uint32_t a1, a2, a3, a4;
    asm("add.cc.u32 %0, %4, %8;\n\t"
        "addc.cc.u32 %1, %5, %9;\n\t"
        "addc.cc.u32 %2, %6, %10;\n\t"
        "addc.u32 %3, %7, 0;"
        : "=&r"(a1), "=&r"(a2), "=&r"(a3), "=&r"(a4)
        : "r"(A.a1), "r"(A.a2), "r"(A.a3), "r"(A.a4), "r"(A.b0), "r"(A.b1), "r"(A.b2));
    const uint64_t v = mont_tail_any(A.a0, a1, a2, a3);
    return fold_small(lo32(v), hi32(v), a4);
}

}  // namespace dev
}  // namespace pg12

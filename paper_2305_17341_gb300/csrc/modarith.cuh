// modarith.cuh -- 64-bit modular arithmetic for residues of primes q < 2^60.
//
// Every RNS limb of the paper's full-RNS CKKS (App. A) is a polynomial with
// coefficients mod a prime q_i = 1 mod 2N.  All arithmetic stays exact.
//   * Shoup multiplication by a precomputed constant w (w' = floor(w 2^64 / q)):
//     one 64x64 high product and two low products, result in [0, 2q).
//   * Montgomery reduction (R = 2^64) of a 128-bit value x < q R, used for
//     products of two variable operands and for lazily accumulated sums of
//     products (sum of up to 15 products of residues < q stays below q R).
#pragma once
#include <cstdint>

typedef unsigned long long u64;
typedef long long i64;
typedef unsigned int u32;

// Programmatic dependent launch.  A kernel that calls pdl_trigger lets the next
// kernel of the stream start as soon as all its own CTAs run, if that kernel
// was launched for it (the NTT passes are): its CTAs take free SMs, form their
// indexes and stage their tables, and pdl_wait holds them until every earlier
// kernel has finished and its writes are visible.  Nothing that an earlier
// kernel writes is touched before pdl_wait, and in every launch some CTA calls
// it, with work or without: the kernel after it waits for this grid alone.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

struct ModQ {
    u64 q;       // the prime
    u64 qinv;    // -q^-1 mod 2^64 (Montgomery)
    u64 r2;      // 2^128 mod q
    u64 twoq;
    u64 wone;    // floor(2^64 / q): the Shoup companion of 1
};

// Constants of the float-quotient product (fq_mul below) for a prime
// 2^36 <= q < 1.5 2^40 (on = 0 for the others).
struct ModF {
    u64 nQ;      // -(q 2^22) mod 2^64
    u64 cst;     // kFqBits (q 2^22) mod 2^64
    u64 nq;      // -q split for a signed multiply-add: low word signed, high word the rest
    float qi;    // 2^32 / q
    u32 on;
};
// 1.5 2^23: adding it to a float |v| <= 2^22 rounds v to an integer that
// sits in the low mantissa bits, as_int(v + kFqMagic) = kFqBits + round(v).
#define FQ_MAGIC 12582912.0f
constexpr u32 kFqBits = 0x4B400000u;

__device__ __forceinline__ u64 mulhi64(u64 a, u64 b) { return __umul64hi(a, b); }

// a * w mod q, lazily in [0, 2q), for any a < 2^64.
__device__ __forceinline__ u64 shoup_lazy(u64 a, u64 w, u64 wp, u64 q) {
    u64 h = mulhi64(a, wp);
    return a * w - h * q;
}

// High word of the 128-bit product a b from three of its four 32 x 32
// partial products: dropping al bl and the low halves of ah bl and al bh
// loses less than 3 units of 2^64, so the result is the exact high word
// minus 0, 1 or 2.
__device__ __forceinline__ u64 mulhi64_trunc(u64 a, u64 b) {
    const u32 al = (u32)a, ah = (u32)(a >> 32), bl = (u32)b, bh = (u32)(b >> 32);
    return (u64)ah * bh + __umulhi(ah, bl) + __umulhi(al, bh);
}

// a * w mod q in [0, 4q) for any a < 2^64 and q < 2^62: Shoup's product with
// the truncated quotient (exact quotient minus at most 2).
__device__ __forceinline__ u64 shoup_lazy4(u64 a, u64 w, u64 wp, u64 q) {
    return a * w - mulhi64_trunc(a, wp) * q;
}

__device__ __forceinline__ u64 shoup(u64 a, u64 w, u64 wp, u64 q) {
    u64 r = shoup_lazy(a, w, wp, q);
    return r >= q ? r - q : r;
}

// a mod q for any 64-bit a: Shoup's product by 1 lands in [0, 2q), then one
// conditional subtraction.
__device__ __forceinline__ u64 reduce_any(u64 a, u64 q, u64 wone) {
    u64 r = a - mulhi64(a, wone) * q;
    return r >= q ? r - q : r;
}

__device__ __forceinline__ u64 reduce4q(u64 a, u64 q) {
    a = a >= 2 * q ? a - 2 * q : a;
    return a >= q ? a - q : a;
}

__device__ __forceinline__ u64 addmod(u64 a, u64 b, u64 q) {
    u64 s = a + b;
    return s >= q ? s - q : s;
}

__device__ __forceinline__ u64 submod(u64 a, u64 b, u64 q) { return a >= b ? a - b : a + q - b; }

// 128-bit accumulator
struct U128 {
    u64 lo, hi;
};

__device__ __forceinline__ void mac128(U128 &acc, u64 a, u64 b) {
    u64 lo = a * b;
    u64 hi = mulhi64(a, b);
    u64 nlo = acc.lo + lo;
    acc.hi += hi + (nlo < lo ? 1ull : 0ull);
    acc.lo = nlo;
}

// acc += a b for residues a, b < q < 2^60, keeping acc below q 2^64 (the
// Montgomery reduction's input bound) however many terms are summed: each
// product is below q 2^60, so after it the high word is below q + q/16 + 1,
// and subtracting q 2^64 (a multiple of q) once restores the bound.
__device__ __forceinline__ void mac128_q(U128 &acc, u64 a, u64 b, u64 q) {
    mac128(acc, a, b);
    if (acc.hi >= q) acc.hi -= q;
}

// -------------------------------------------------- float-quotient product
// y w mod q for the 40-bit limbs, with the quotient taken as two FP32 digits
// instead of one 64-bit high product: the high products are what bounds the
// butterfly (IMAD.HI and IMAD.WIDE issue at half the rate of IMAD), while
// the FP32 multiply-adds run on the FMA lanes that integer code leaves idle.
//
// w is centred, |w| <= q/2, with wq = w / (q 2^8); y is signed, |y| <= 17.5 q.
//   ha = round((y >> 14) wq)              ~ y w / (q 2^22)
//   P  = y w - ha (q 2^22)                exact mod 2^64
//   hb = round((P >> 32) 2^32 / q)
//   t  = P - hb q
// For q < 1.5 2^40: |y w / q| <= 8.75 q, so |ha| < 2^21.72 and its error is
// below 0.5 + 2^21.72 2^-23 < 0.92 (y and wq each carry a half unit of 2^-24),
// |P| <= 0.92 2^22 q < 2^62.5 fits a signed word; |hb| <= 2^21.9, its error
// is below 0.5 + 2^21.9 2^-23 + 2^32/q <= 0.97 (q >= 2^40), and for smaller
// q, where the first two terms shrink with q and 2^32/q <= 2^-4 (q >= 2^36),
// below 0.97 too: |t| < q, t signed.  16 butterfly stages from |x| <= q stay
// below 16.6 q, a difference u - x of the fused epilogues below 17.5 q.  18 instructions per butterfly against 21.6 with the truncated
// Shoup quotient, 1406 against 1000 G butterflies/s with register operands.
// The products are written as a wide product and an add in one statement:
// the compiler then emits one multiply-add without the moves that a wide
// multiply-add on separately built register pairs costs.
__device__ __forceinline__ u64 fq_madw(u32 a, u32 b, u64 c) {
    u64 r;
    asm("mul.wide.u32 %0, %1, %2;\n\tadd.u64 %0, %0, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
__device__ __forceinline__ u64 fq_madws(int a, int b, u64 c) {
    u64 r;
    asm("mul.wide.s32 %0, %1, %2;\n\tadd.u64 %0, %0, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
__device__ __forceinline__ u32 fq_madl(u32 a, u32 b, u32 c) {
    u32 r;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}
// P - round(P / q) q for a signed word P (|P| < 2^62.5): |result| < q.
__device__ __forceinline__ u64 fq_low(u32 p0, u32 p1, const ModF &m) {
    const int hb = __float_as_int(__fmaf_rn(__int2float_rn((int)p1), m.qi, FQ_MAGIC)) - (int)kFqBits;
    const u64 r = fq_madws(hb, (int)(u32)m.nq, ((u64)p1 << 32) | p0);
    return ((u64)fq_madl((u32)hb, (u32)(m.nq >> 32), (u32)(r >> 32)) << 32) | (u32)r;
}
// tw: x = w (centred, signed), y = the bits of wq
__device__ __forceinline__ u64 fq_mul(u64 y, const ulonglong2 tw, const ModF &m) {
    const u32 y0 = (u32)y, y1 = (u32)(y >> 32), w0 = (u32)tw.x, w1 = (u32)(tw.x >> 32);
    const float yf = __int2float_rn((int)__funnelshift_r(y0, y1, 14));
    const u32 ha = __float_as_uint(__fmaf_rn(yf, __uint_as_float((u32)tw.y), FQ_MAGIC));
    u64 a = fq_madw(y0, w0, m.cst);
    a = fq_madw(ha, (u32)m.nQ, a);
    const u32 h = fq_madl(ha, (u32)(m.nQ >> 32), fq_madl(y0, w1, fq_madl(y1, w0, (u32)(a >> 32))));
    return fq_low((u32)a, h, m);
}
// Factor of a 64-bit unsigned source: y w = (low word of y) lo + (high word)
// hi with lo = w, hi = w 2^32 mod q, both centred; .y the bits of w / (q 2^22).
// For sources below 2^41 `lo` is instead a factor of fq_mul (see FqDot::narrow).
struct FqPair {
    ulonglong2 lo, hi;
};
// Sum of products y_i w_i + e modulo a prime with ModF constants, with one
// quotient for the sum (its two digits, as in fq_mul): 3 or 4 wide or low
// multiply-adds per word of y against 14 multiply slots for a Shoup product.
// Bound: sum |y_i w_i| + e below 2^42 q (get), in at most ten words.  Four narrow
// sources (y < 2^41, |w| <= q/2) or five wide ones and e < q stay below it; so do
// the sums of lin_row (relin.cu), which derives its own case.
struct FqDot {
    u64 a;
    float s;
    FqDot() = default;
    __device__ __forceinline__ FqDot(u64 e, const ModF &m) : a(e + m.cst), s(0.0f) {}
    __device__ __forceinline__ void word(u32 y, const ulonglong2 w) {
        s = __fmaf_rn(__uint2float_rn(y), __uint_as_float((u32)w.y), s);
        a = fq_madw(y, (u32)w.x, a);
        a = ((u64)fq_madl(y, (u32)(w.x >> 32), (u32)(a >> 32)) << 32) | (u32)a;
    }
    __device__ __forceinline__ void wide(u64 y, const FqPair &w) {
        word((u32)y, w.lo);
        word((u32)(y >> 32), w.hi);
    }
    __device__ __forceinline__ void narrow(u64 y, const ulonglong2 w) {
        const u32 y0 = (u32)y, y1 = (u32)(y >> 32), w0 = (u32)w.x, w1 = (u32)(w.x >> 32);
        s = __fmaf_rn(__int2float_rn((int)__funnelshift_r(y0, y1, 14)), __uint_as_float((u32)w.y), s);
        a = fq_madw(y0, w0, a);
        a = ((u64)fq_madl(y0, w1, fq_madl(y1, w0, (u32)(a >> 32))) << 32) | (u32)a;
    }
    // the residue in [0, q): for a sum below 2^42 q, |ha| <= 2^20 is off by less
    // than 0.78 with 4 words and, below 2^41.2 q, 0.92 with 10: half a unit, 2^-5
    // for each addition to the estimate, 2^-23 |ha| for the rounding of the words
    // and factors, 2^-9 a word for the 14 bits cut off.  |P| < 2^62.5, |t| < q
    __device__ __forceinline__ u64 get(u64 q, const ModF &m) const;
};

// a signed value |v| < q to [0, q)
__device__ __forceinline__ u64 fq_pos(u64 v, u64 q) { return v + ((u64)((i64)v >> 63) & q); }
__device__ __forceinline__ u64 FqDot::get(u64 q, const ModF &m) const {
    const u32 ha = __float_as_uint(s + FQ_MAGIC);
    const u64 r = fq_madw(ha, (u32)m.nQ, a);
    return fq_pos(fq_low((u32)r, fq_madl(ha, (u32)(m.nQ >> 32), (u32)(r >> 32)), m), q);
}
// any signed |v| <= 17.5 q to |result| <= 0.57 q
__device__ __forceinline__ u64 fq_red(u64 v, const ModF &m) { return fq_low((u32)v, (u32)(v >> 32), m); }

// Montgomery REDC with the prime and -q^-1 mod 2^64 given directly.
__device__ __forceinline__ u64 redc_q(u64 lo, u64 hi, u64 q, u64 qinv) {
    const u64 t = lo * qinv;
    const u64 r = hi + mulhi64(t, q) + (lo != 0 ? 1ull : 0ull);
    return r >= q ? r - q : r;
}

// Montgomery REDC: x * 2^-64 mod q for x < q 2^64, result in [0, q).
__device__ __forceinline__ u64 redc(u64 lo, u64 hi, const ModQ &m) {
    u64 t = lo * m.qinv;
    u64 mh = mulhi64(t, m.q);
    u64 r = hi + mh + (lo != 0 ? 1ull : 0ull);
    return r >= m.q ? r - m.q : r;
}

// a * b mod q for two residues (double REDC with R^2).
__device__ __forceinline__ u64 mulmod(u64 a, u64 b, const ModQ &m) {
    u64 t = redc(a * b, mulhi64(a, b), m);           // a b R^-1
    return redc(t * m.r2, mulhi64(t, m.r2), m);      // a b
}

// a * bM mod q where bM = b R mod q is in Montgomery form.
__device__ __forceinline__ u64 mulmont(u64 a, u64 bM, const ModQ &m) {
    return redc(a * bM, mulhi64(a, bM), m);
}

// (hi 2^64 + lo) mod q for any 128-bit value.
__device__ __forceinline__ u64 mod128(u64 hi, u64 lo, const ModQ &m) {
    u64 h = hi % m.q, l = lo % m.q;
    u64 t = redc(l, h, m);                           // (h R + l) R^-1
    return redc(t * m.r2, mulhi64(t, m.r2), m);      // t R
}

// signed integer -> residue
__device__ __forceinline__ u64 from_signed(i64 x, u64 q) {
    if (x >= 0) return ((u64)x) % q;
    u64 r = ((u64)(-x)) % q;
    return r ? q - r : 0;
}

// kernels.cuh -- device code shared by the conversion kernels.
#pragma once
#include <algorithm>

#include "he_internal.h"

namespace he {

// e = floor(S / P) for S = sum_j y[j] (P/p_j): S < A P < 2^(64 A).
template <int A>
__device__ __forceinline__ int md_overflow(const u64 (&y)[A], const MdExact &k) {
    if constexpr (A == 1) {
        return 0;
    } else {
        u64 s[A];
#pragma unroll
        for (int i = 0; i < A; i++) s[i] = 0;
#pragma unroll
        for (int j = 0; j < A; j++) {
            u64 carry = 0;
#pragma unroll
            for (int i = 0; i < A - 1; i++) {
                const u64 lo = y[j] * k.phat[j][i], hi = __umul64hi(y[j], k.phat[j][i]);
                u64 t = s[i] + lo;
                u64 cy = t < lo ? 1ull : 0ull;
                t += carry;
                cy += t < carry ? 1ull : 0ull;
                s[i] = t;
                carry = hi + cy;   // hi < 2^62
            }
            s[A - 1] += carry;     // the partial sums stay below S
        }
        int e = 0;
#pragma unroll
        for (int m = 0; m < A - 1; m++) {
            int cmp = 0;
#pragma unroll
            for (int i = A - 1; i >= 0; i--)
                if (cmp == 0) cmp = s[i] > k.kP[m][i] ? 1 : (s[i] < k.kP[m][i] ? -1 : 0);
            e += cmp >= 0 ? 1 : 0;
        }
        return e;
    }
}

// Sum of products v k of residues v < q and centred k modulo a prime with ModF
// constants: the sum mod 2^64 and, as a float, sum (v >> 14)(k >> 14).  Of at most
// lim + 1 products (12 below 1.1 2^40, else 7) the estimate of the quotient in
// units of 2^22 q is off by less than 1.65 (1.2): half a unit, half a unit of
// 2^-24 for each conversion, and the same for each addition of a partial sum of
// up to as many times q / 2^23; then |sum - ha 2^22 q| < 2^62.9 fits a signed
// word.  Longer sums are folded to |.| < 1.5 q in between.
struct FqMacC {
    float c;     // 2^6 / q
    int lim;     // products between folds
    int Ql;      // -(q 2^22) with a signed low word
    u32 Qh;
    __device__ __forceinline__ FqMacC(const ModF &m, u64 q)
        : c(m.qi * 1.4901161193847656e-08f), lim(q < (1126ull << 30) ? 11 : 6), Ql((int)(u32)m.nQ),
          Qh((u32)(m.nQ >> 32) + ((u32)m.nQ >> 31)) {}
};
struct FqMac {
    u32 a0, a1;
    float s;
    __device__ __forceinline__ static float part(u64 v) {
        return __int2float_rn((int)__funnelshift_r((u32)v, (u32)(v >> 32), 14));
    }
    __device__ __forceinline__ void add(u64 v, float vf, u64 k, float kf) {
        s = __fmaf_rn(vf, kf, s);
        asm("mad.lo.cc.u32 %0, %2, %4, %0;\n\tmadc.hi.u32 %1, %2, %4, %1;\n\t"
            "mad.lo.u32 %1, %3, %4, %1;\n\tmad.lo.u32 %1, %2, %5, %1;"
            : "+r"(a0), "+r"(a1)
            : "r"((u32)v), "r"((u32)(v >> 32)), "r"((u32)k), "r"((u32)(k >> 32)));
    }
    // |result| < 1.5 q: the second digit is off by half a unit, a quarter each for
    // the rounding of h and of the product, 0.41 for that of 1/q
    __device__ __forceinline__ void fold(const FqMacC &c, const ModF &m) {
        const int ha = __float2int_rn(s * c.c);
        u64 r = fq_madws(ha, c.Ql, ((u64)a1 << 32) | a0);
        const u32 h = fq_madl((u32)ha, c.Qh, (u32)(r >> 32));
        const int hb = __float2int_rn(__int2float_rn((int)h) * m.qi);
        r = fq_madws(hb, (int)(u32)m.nq, ((u64)h << 32) | (u32)r);
        a0 = (u32)r, a1 = fq_madl((u32)hb, (u32)(m.nq >> 32), (u32)(r >> 32));
        s = 0.0f;
    }
    __device__ __forceinline__ u64 get(const FqMacC &c, u64 q, const ModF &m) {
        fold(c, m);
        return fq_pos(fq_low(a0, a1, m), q);
    }
};
// Sum of products of residues below 2^60 and its Montgomery reduction: up to 256
// products stay below 2^128, so only the end reduces the high word.
struct WideMac {
    u32 w0, w1, w2, w3;
    __device__ __forceinline__ void add(u64 a, u64 b) {
        asm("mad.lo.cc.u32 %0, %4, %6, %0;\n\tmadc.hi.cc.u32 %1, %4, %6, %1;\n\t"
            "madc.lo.cc.u32 %2, %5, %7, %2;\n\tmadc.hi.u32 %3, %5, %7, %3;\n\t"
            "mad.lo.cc.u32 %1, %4, %7, %1;\n\tmadc.hi.cc.u32 %2, %4, %7, %2;\n\taddc.u32 %3, %3, 0;\n\t"
            "mad.lo.cc.u32 %1, %5, %6, %1;\n\tmadc.hi.cc.u32 %2, %5, %6, %2;\n\taddc.u32 %3, %3, 0;"
            : "+r"(w0), "+r"(w1), "+r"(w2), "+r"(w3)
            : "r"((u32)a), "r"((u32)(a >> 32)), "r"((u32)b), "r"((u32)(b >> 32)));
    }
    __device__ __forceinline__ u64 get(const ModQ &m) const {
        const u64 hi = reduce_any(((u64)w3 << 32) | w2, m.q, m.wone);
        return redc(((u64)w1 << 32) | w0, hi, m);
    }
};

// a factor of fq_mul from a centred word: the bits of w / (q 2^8), c = 2^6 / q
__device__ __forceinline__ ulonglong2 fq_svar(u64 w, float c) {
    return make_ulonglong2(w, __float_as_uint(__fmul_rn(FqMac::part(w), c)));
}

}  // namespace he

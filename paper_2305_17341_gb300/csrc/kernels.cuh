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

}  // namespace he

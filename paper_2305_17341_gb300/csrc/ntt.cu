// ntt.cu -- batched negacyclic number-theoretic transforms over RNS limbs.
//
// The polynomial products of full-RNS CKKS (App. A; "RNS and NTT domains",
// Sec. 3.2) are evaluated pointwise after a negacyclic NTT of every limb.
// Decompose and ModDown (Sec. 3.3) spend most of their time here.
//
// Forward: Cooley-Tukey with the 2N-th root psi merged in (twiddle psi^brv(k)),
// natural order in, bit-reversed order out; evaluation point of output j is
// psi^(2 brv(j) + 1).  Inverse: Gentleman-Sande with psi^-brv(k), bit-reversed
// in, natural out, times N^-1.  Harvey's lazy butterflies keep values in
// [0, 4q) (forward) / [0, 2q) (inverse) between stages; the output is in [0, q).
// Measured (1024 rows of N = 2^16, the chain 60 + 20 x 40, 2 x 60 bits):
// forward 721 -> 567 us, inverse 819 -> 618 us, of which the float-quotient
// butterfly gives about two thirds (721 -> 619), the twiddles in their order
// of use and the columns' single crossing of shared memory 619 -> 584, the
// compile-time column stride and the staged row twiddles the rest.  What bounds
// it: the FMA-heavy pipe (70 % busy in the column pass, 63 % in the row pass, 2024
// rows) at 23 and 28 instructions per butterfly, 18 of them arithmetic.
// The register-blocked kernels for logN 14..16 go lazier: on the 40-bit
// limbs (ModF::on) both directions run the signed float-quotient product of
// modarith.cuh; on other primes the forward skips the per-stage reduction
// below 2^57 and the inverse keeps values in [0, 4q), both with a
// truncated-quotient Shoup product.
//
// Each limb of N = N1 * N2 coefficients is transformed in two passes: pass 1
// runs the stages whose butterfly span is >= N2 on column tiles (elements with
// equal index mod N2, C columns per CTA, staged in shared memory); pass 2 runs
// the remaining log2(N2) stages on rows of N2 contiguous coefficients.  Both
// passes read and write HBM once.
#include <cstdio>
#include <cstring>
#include <algorithm>
#include <stdexcept>

#include "bulkcopy.cuh"
#include "he_internal.h"

namespace he {

__device__ __forceinline__ void bf_fwd(u64 &x, u64 &y, u64 w, u64 wp, u64 q) {
    u64 tq = 2 * q;
    u64 a = x >= tq ? x - tq : x;
    u64 t = shoup_lazy(y, w, wp, q);
    x = a + t;
    y = a - t + tq;
}

__device__ __forceinline__ void bf_inv(u64 &x, u64 &y, u64 w, u64 wp, u64 q) {
    u64 tq = 2 * q;
    u64 s = x + y;
    s = s >= tq ? s - tq : s;
    u64 d = x - y + tq;
    x = s;
    y = shoup_lazy(d, w, wp, q);
}

// Inverse butterfly on values in [0, 4q): s = x + y reduced below 4q,
// y' = w (x - y + 4q) with the truncated-quotient Shoup product, in [0, 4q)
// (8q < 2^64 for every prime below 2^61).
__device__ __forceinline__ void bf_inv4(u64 &x, u64 &y, u64 w, u64 wp, u64 q) {
    const u64 fq = 4 * q;
    u64 s = x + y;
    s = s >= fq ? s - fq : s;
    const u64 d = x - y + fq;
    x = s;
    y = shoup_lazy4(d, w, wp, q);
}

// ---------------------------------------------------------------- forward
__global__ void k_ntt_fwd_p1(u64 *data, RowMap rm, const ModQ *mods, const u64 *tw, const u64 *twp,
                             int logN, int logN1, int C) {
    extern __shared__ u64 sm[];
    const int N = 1 << logN, N1 = 1 << logN1, N2 = N >> logN1;
    const long row = blockIdx.y;
    const int pidx = rm.at(row);
    const u64 q = mods[pidx].q;
    u64 *base = data + row * (long)N + (long)blockIdx.x * C;
    const u64 *w = tw + (long)pidx * N, *wp = twp + (long)pidx * N;
    for (int e = threadIdx.x; e < N1 * C; e += blockDim.x) {
        int r = e / C, c = e - r * C;
        sm[e] = base[(long)r * N2 + c];
    }
    __syncthreads();
    for (int m = 1, t1 = N1 >> 1; m < N1; m <<= 1, t1 >>= 1) {
        for (int e = threadIdx.x; e < (N1 >> 1) * C; e += blockDim.x) {
            int b = e / C, c = e - b * C;
            int i = b / t1, k = b - i * t1;
            int hi = 2 * i * t1 + k;
            u64 x = sm[hi * C + c], y = sm[(hi + t1) * C + c];
            bf_fwd(x, y, w[m + i], wp[m + i], q);
            sm[hi * C + c] = x;
            sm[(hi + t1) * C + c] = y;
        }
        __syncthreads();
    }
    for (int e = threadIdx.x; e < N1 * C; e += blockDim.x) {
        int r = e / C, c = e - r * C;
        base[(long)r * N2 + c] = sm[e];
    }
}

__global__ void k_ntt_fwd_p2(u64 *data, RowMap rm, const ModQ *mods, const u64 *tw, const u64 *twp,
                             int logN, int logN1, int R) {
    extern __shared__ u64 sm[];
    const int N = 1 << logN, N1 = 1 << logN1, N2 = N >> logN1;
    const long row = blockIdx.y;
    const int pidx = rm.at(row);
    const u64 q = mods[pidx].q;
    const int hi0 = blockIdx.x * R;
    u64 *base = data + row * (long)N + (long)hi0 * N2;
    const u64 *w = tw + (long)pidx * N, *wp = twp + (long)pidx * N;
    for (int e = threadIdx.x; e < R * N2; e += blockDim.x) sm[e] = base[e];
    __syncthreads();
    const int half = N2 >> 1;
    for (int m = N1, t = N2 >> 1; t >= 1; m <<= 1, t >>= 1) {
        for (int e = threadIdx.x; e < R * half; e += blockDim.x) {
            int rr = e / half, b = e - rr * half;
            int il = b / t, k = b - il * t;
            int j = 2 * il * t + k;
            int gi = (hi0 + rr) * (N2 / (2 * t)) + il;
            u64 *s = sm + rr * N2;
            u64 x = s[j], y = s[j + t];
            bf_fwd(x, y, w[m + gi], wp[m + gi], q);
            s[j] = x;
            s[j + t] = y;
        }
        __syncthreads();
    }
    for (int e = threadIdx.x; e < R * N2; e += blockDim.x) base[e] = reduce4q(sm[e], q);
}

// ---------------------------------------------------------------- inverse
__global__ void k_ntt_inv_p2(u64 *data, RowMap rm, const ModQ *mods, const u64 *tw, const u64 *twp,
                             int logN, int logN1, int R) {
    extern __shared__ u64 sm[];
    const int N = 1 << logN, N1 = 1 << logN1, N2 = N >> logN1;
    const long row = blockIdx.y;
    const int pidx = rm.at(row);
    const u64 q = mods[pidx].q;
    const int hi0 = blockIdx.x * R;
    u64 *base = data + row * (long)N + (long)hi0 * N2;
    const u64 *w = tw + (long)pidx * N, *wp = twp + (long)pidx * N;
    for (int e = threadIdx.x; e < R * N2; e += blockDim.x) sm[e] = base[e];
    __syncthreads();
    const int half = N2 >> 1;
    for (int t = 1; t < N2; t <<= 1) {
        int m = N / (2 * t);
        for (int e = threadIdx.x; e < R * half; e += blockDim.x) {
            int rr = e / half, b = e - rr * half;
            int il = b / t, k = b - il * t;
            int j = 2 * il * t + k;
            int gi = (hi0 + rr) * (N2 / (2 * t)) + il;
            u64 *s = sm + rr * N2;
            u64 x = s[j], y = s[j + t];
            bf_inv(x, y, w[m + gi], wp[m + gi], q);
            s[j] = x;
            s[j + t] = y;
        }
        __syncthreads();
    }
    (void)N1;
    for (int e = threadIdx.x; e < R * N2; e += blockDim.x) base[e] = sm[e];
}

__global__ void k_ntt_inv_p1(u64 *data, RowMap rm, const ModQ *mods, const u64 *tw, const u64 *twp,
                             const u64 *ninv, int logN, int logN1, int C) {
    extern __shared__ u64 sm[];
    const int N = 1 << logN, N1 = 1 << logN1, N2 = N >> logN1;
    const long row = blockIdx.y;
    const int pidx = rm.at(row);
    const u64 q = mods[pidx].q;
    u64 *base = data + row * (long)N + (long)blockIdx.x * C;
    const u64 *w = tw + (long)pidx * N, *wp = twp + (long)pidx * N;
    for (int e = threadIdx.x; e < N1 * C; e += blockDim.x) {
        int r = e / C, c = e - r * C;
        sm[e] = base[(long)r * N2 + c];
    }
    __syncthreads();
    for (int t1 = 1; t1 < N1; t1 <<= 1) {
        int m = N1 / (2 * t1);
        for (int e = threadIdx.x; e < (N1 >> 1) * C; e += blockDim.x) {
            int b = e / C, c = e - b * C;
            int i = b / t1, k = b - i * t1;
            int hi = 2 * i * t1 + k;
            u64 x = sm[hi * C + c], y = sm[(hi + t1) * C + c];
            bf_inv(x, y, w[m + i], wp[m + i], q);
            sm[hi * C + c] = x;
            sm[(hi + t1) * C + c] = y;
        }
        __syncthreads();
    }
    const u64 ni = ninv[2 * pidx], nip = ninv[2 * pidx + 1];
    for (int e = threadIdx.x; e < N1 * C; e += blockDim.x) {
        int r = e / C, c = e - r * C;
        base[(long)r * N2 + c] = shoup(sm[e], ni, nip, q);
    }
}

// ------------------------------------------------- register-blocked passes
// One pass transforms W independent length-M sequences per CTA (M = 2^LM,
// 128 or 256).  Each of the T = M/16 threads of a sequence holds 16 elements:
// layout A = elements t + T k (k < 16), which covers the 4 stages with spans
// M/2 .. T in registers; a shared-memory transpose gives layout B = elements
// 16 t + k, which covers spans T/2 .. 1.  ROWS: sequences are rows of M
// contiguous coefficients (the last stages of a limb); otherwise columns
// with stride N/M (the first stages).  The twiddle of the butterfly at local
// span sp and local group i is psi^brv((M / 2sp) G + i), G = 1 for columns
// and G = N/M + row for rows.  Global accesses of rows are in layout A
// (coalesced along the row); columns are coalesced across the W sequences in
// either layout, so they load in A and store in B (the inverse the other way)
// and cross shared memory once.
//
// Twiddle tables (Ctx::d_psi2, d_ipsi2), per prime: 256 entries in natural
// order for the columns, then the M twiddles of every row sequence in the
// order of use: those of layout A at 8/s + j for distance s (shared by the
// sequence's threads), those of layout B as one run of T words per load (word
// t for thread t), so that a warp's load is contiguous.  In natural order the
// last stage's loads were 128 bytes apart between threads, 32 lines each.
// Rows keep each sequence contiguous in shared memory with one pad word per
// 16 (element r at r + r/16): both layouts are free of bank conflicts, and
// every access is a compile-time offset from a per-thread base (17 t + k in
// layout B, t + T k + k T/16 in layout A).
template <int LM, bool ROWS>
struct PassGeom {
    static constexpr int M = 1 << LM, T = M / 16, W = 256 / T;
    static constexpr int SM = ROWS ? W * (M + M / 16) : W * M;
    __device__ static __forceinline__ int sidx(int r, int w) {
        if (ROWS) return w * (M + M / 16) + r + (r >> 4);
        return r * W + w;
    }
};

// Forward butterfly without the reduction of x: x' = x + t, y' = x - t + 4q
// (t = w y mod q in [0, 4q), Shoup's product with the truncated quotient).
// Both outputs grow by less than 4q per stage, so from inputs below 4q the
// 16 stages of a limb stay below 68q < 2^64 for every prime below 2^57 (all
// the 40-bit levels); larger primes use bf_fwd.
__device__ __forceinline__ void bf_fwd_nored(u64 &x, u64 &y, u64 w, u64 wp, u64 q) {
    u64 t = shoup_lazy4(y, w, wp, q);
    u64 a = x;
    x = a + t;
    y = a - t + 4 * q;
}

// Arithmetic of a limb's butterflies, uniform over a CTA: reducing Shoup
// butterflies (primes from 2^57), lazy ones, or the signed float-quotient
// ones (x' = x + t, y' = x - t with |t| < q: 16 stages from |x| <= q stay
// below 17 q, the bound of fq_mul).
enum { AR_RED = 0, AR_LAZY = 1, AR_FQ = 2 };

template <int AR>
__device__ __forceinline__ void bf_fwd_ar(u64 &x, u64 &y, const ulonglong2 wv, u64 q, const ModF &f) {
    if constexpr (AR == AR_FQ) {
        const u64 t = fq_mul(y, wv, f), a = x;
        x = a + t;
        y = a - t;
    } else if constexpr (AR == AR_RED) {
        bf_fwd(x, y, wv.x, wv.y, q);
    } else {
        bf_fwd_nored(x, y, wv.x, wv.y, q);
    }
}

// the exact residue of a forward transform's last value
template <int AR>
__device__ __forceinline__ u64 fwd_residue(u64 s, u64 q, u64 wone, const ModF &f) {
    if constexpr (AR == AR_FQ) return fq_pos(fq_red(s, f), q);
    else if constexpr (AR == AR_RED) return reduce4q(s, q);
    else return reduce_any(s, q, wone);
}

__device__ __forceinline__ int ntt_arith(u64 q, const ModF &f) { return f.on ? AR_FQ : q >= (1ull << 57) ? AR_RED : AR_LAZY; }

// SubScale's value for the transform's last value s: (u - v) w (+ add) mod q
template <int AR>
__device__ __forceinline__ u64 subscale_value(const SubScale &ep, int r, u64 u, u64 s, u64 q, u64 wone, const ModF &f) {
    if constexpr (AR == AR_FQ) {
        return fq_pos(fq_mul(u - s, ep.wf[r], f), q);   // |u - s| <= 17.5 q
    } else {
        const ShoupPair wr = ep.w[r];
        return shoup(submod(u, fwd_residue<AR>(s, q, wone, f), q), wr.w, wr.wp, q);
    }
}

// The twiddles of one sequence (columns: of the prime): w in shared memory
// (STG) or in global memory.
template <int LM, bool ROWS, bool STG>
struct PassTw {
    typedef PassGeom<LM, ROWS> G_;
    const ulonglong2 *w;
    int t;
    __device__ __forceinline__ ulonglong2 at(int i) const {
        if constexpr (STG) return w[i];
        else return __ldg(w + i);
    }
    // distance s (8..1) in layout A, pair j
    __device__ __forceinline__ ulonglong2 a(int s, int j) const { return at(8 / s + j); }
    // span sp (T/2..1) in layout B, pair j
    __device__ __forceinline__ ulonglong2 b(int sp, int j) const {
        if (ROWS) return at(16 + (8 / sp - 1 - (G_::T == 8 ? 1 : 0) + j) * G_::T + t);
        return at(G_::M / (2 * sp) + t * (8 / sp) + j);
    }
};


// The 8 stages of one pass: 4 in registers in layout A, a shared-memory
// transpose, 4 (3 for M = 128) in layout B, leaving the words in x.
template <int LM, bool ROWS, bool STG, int AR>
__device__ __forceinline__ void fwd_pass_body(u64 (&x)[16], u64 *sm, const PassTw<LM, ROWS, STG> &tw, int t, int w, u64 q,
                                              const ModF &f) {
    typedef PassGeom<LM, ROWS> G_;
    constexpr int T = G_::T;
#pragma unroll
    for (int s = 8; s >= 1; s >>= 1) {
#pragma unroll
        for (int k = 0; k < 16; k++)
            if (!(k & s)) bf_fwd_ar<AR>(x[k], x[k + s], tw.a(s, k / (2 * s)), q, f);
    }
#pragma unroll
    for (int k = 0; k < 16; k++) sm[G_::sidx(t + T * k, w)] = x[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; k++) x[k] = sm[G_::sidx(16 * t + k, w)];
#pragma unroll
    for (int sp = T / 2; sp >= 1; sp >>= 1) {
#pragma unroll
        for (int k = 0; k < 16; k++)
            if (!(k & sp)) bf_fwd_ar<AR>(x[k], x[k + sp], tw.b(sp, k / (2 * sp)), q, f);
    }
}

// The stages and the stores of one tile whose words are in x: the plain
// residues (or, after the column pass, the lazy values) to p, or the fused
// epilogue's values.
template <int LM, int LS, bool ROWS, bool STG, int AR, bool SUBSC>
__device__ __forceinline__ void fwd_tile(u64 (&x)[16], u64 *sm, const PassTw<LM, ROWS, STG> &tw, int t, int w, u64 *p,
                                         bool on, long row, long seq, int N, u64 q, u64 wone, const ModF &f,
                                         const SubScale &ep) {
    typedef PassGeom<LM, ROWS> G_;
    constexpr int M = G_::M, T = G_::T;
    fwd_pass_body<LM, ROWS, STG, AR>(x, sm, tw, t, w, q, f);
    if (!ROWS) {
        // the store addresses are formed again here from an opaque copy of
        // the base, so that the 16 strided load addresses of the columns are
        // not kept live through the butterflies
        u64 *ps = p + ((16L * t) << LS);
        asm volatile("" : "+l"(ps));
#pragma unroll
        for (int k = 0; k < 16; k++) ps[k << LS] = x[k];
        return;
    }
    // back to layout A: a thread rewrites the words that it read, so only the
    // reads below wait for the others
#pragma unroll
    for (int k = 0; k < 16; k++) sm[G_::sidx(16 * t + k, w)] = x[k];
    __syncthreads();
    if (!on) return;
    if (ROWS && SUBSC) {
        const u32 arow = ep.row0 + (u32)row;
        const u32 it = arow / (u32)ep.rows_per_item;
        const int r = (int)(arow - it * (u32)ep.rows_per_item);
        const long off = (long)r * N + seq * M;
        const u64 *up = ep.u + it * ep.us + off;
        u64 *op = (ep.n_out ? ep.outs[it >> 1] + (it & 1) * ep.os : ep.out + it * ep.os) + off;
        // every operand before the first store: a load may not pass a store
        // that could alias it, so interleaved they would be 16 memory latencies
#pragma unroll
        for (int k = 0; k < 16; k++) x[k] = up[t + T * k];
#pragma unroll
        for (int k = 0; k < 16; k++) x[k] = subscale_value<AR>(ep, r, x[k], sm[G_::sidx(t + T * k, w)], q, wone, f);
        if (ep.add) {
            const u64 *ap = ep.add + it * ep.as + off;
            u64 y[16];
#pragma unroll
            for (int k = 0; k < 16; k++) y[k] = ap[t + T * k];
#pragma unroll
            for (int k = 0; k < 16; k++) x[k] = addmod(x[k], y[k], q);
        }
#pragma unroll
        for (int k = 0; k < 16; k++) op[t + T * k] = x[k];
        return;
    }
#pragma unroll
    for (int k = 0; k < 16; k++) p[t + T * k] = fwd_residue<AR>(sm[G_::sidx(t + T * k, w)], q, wone, f);
}

// Which rows and sequences a CTA transforms.
//
// Columns: blockIdx.y is the row; the prime's few twiddles are staged in
// shared memory while the words are on their way (each stage would wait for
// them otherwise).  Rows: the twiddles of a row sequence are
// twice its data and are read by nobody else in the limb, so a CTA takes the
// same sequences of `items` limbs of one prime (rows r, r + n, ... of the
// launch's row map) and stages their twiddles, one contiguous block, in the
// same way (STG).  blockIdx.y = prime + n * (group of items).
template <int LM, bool ROWS>
struct PassMap {
    typedef PassGeom<LM, ROWS> G_;
    int t, w;         // thread of its sequence, the sequence's slot in the CTA
    long row, seq;
    bool on;          // a row of the launch that is not skipped
    int pidx;         // the row's prime (uniform over the CTA)
    __device__ __forceinline__ PassMap(const RowMap &rm, long nr, int items, const RowSkip &skip) {
        if (ROWS) {
            const int wi = G_::W / items;   // sequences per item
            w = threadIdx.x / G_::T, t = threadIdx.x % G_::T;
            const int it = w / wi;
            const u32 n = (u32)rm.n, g = blockIdx.y / n, k = blockIdx.y - g * n;
            const u32 r0 = k + n * (g * (u32)items), r = r0 + n * (u32)it;
            seq = (long)blockIdx.x * wi + (w - it * wi);
            on = r < (u32)nr && !skip.skip(r);
            // threads without a row read (and drop) the first item's words:
            // only this CTA writes them, and after its barrier
            row = on ? r : r0;
            pidx = rm.at32(k);
        } else {
            t = threadIdx.x / G_::W, w = threadIdx.x % G_::W;
            row = blockIdx.y;
            seq = (long)blockIdx.x * G_::W + w;
            on = !skip.skip(blockIdx.y);
            pidx = rm.at32(blockIdx.y);
        }
    }
    // grid of nr rows of N words: (x, y)
    static dim3 grid(int N, int n, long nr, int items) {
        const unsigned tiles = (unsigned)((N >> LM) / (ROWS ? G_::W / items : G_::W));
        const long y = ROWS ? n * ((nr + (long)n * items - 1) / ((long)n * items)) : nr;
        return dim3(tiles, (unsigned)y);
    }
};

// Limbs of one prime that a row-pass CTA takes together: the most (4, 2 or
// 1) that leave at most a fifth of the threads without a row.
static int pass_items(int n, long nr) {
    const long per = (nr + n - 1) / n;
    for (int i : {4, 2})
        if (((per + i - 1) / i) * i * 5 <= per * 6) return i;
    return 1;
}

// LS: log2 of the columns' stride (words).
// Copies the twiddles of the CTA's W / items row sequences (columns: the M of
// the prime) to dst.
template <int LM, bool ROWS>
__device__ __forceinline__ void stage_twiddles(ulonglong2 *dst, const ulonglong2 *tab, int items) {
    typedef PassGeom<LM, ROWS> G_;
    const int n = ROWS ? G_::W / items * G_::M : G_::M;
    const ulonglong2 *src = ROWS ? tab + 256 + (long)blockIdx.x * n : tab;
    for (int i = threadIdx.x; i < n; i += 256) bc_copy16(bc_smem(dst + i), src + i);
    bc_commit();
}
__device__ __forceinline__ void staged_wait() { bc_wait_groups<0>(); }

template <int LM, int LS, bool ROWS, bool STG, int MINB, bool SUBSC>
__global__ void __launch_bounds__(256, MINB) k_ntt_fwd_fast(u64 *data, RowMap rm, long nr, int items,
                                                            const ModQ *mods, const ModF *modf,
                                                            const ulonglong2 *tw2, int logN, RowSkip skip,
                                                            SubScale ep) {
    typedef PassGeom<LM, ROWS> G_;
    constexpr int M = G_::M, T = G_::T;
    extern __shared__ __align__(16) u64 sm[];
    ulonglong2 *stg = (ulonglong2 *)(sm + G_::SM);
    const int N = 1 << logN;
    pdl_trigger();
    const PassMap<LM, ROWS> pm(rm, nr, items, skip);
    // uniform over the CTA.  Columns: a CTA of a skipped row waits all the same, or
    // a launch of which every row is skipped (a sum's digits at a level of one
    // digit) would end before the kernels ahead of it, and later kernels wait for
    // this one only.  Rows: groups past the launch's end, never the first one, so
    // the grid waits without them (with a wait here too, the other registers of
    // the row pass made 2024 rows of N = 2^16 3 % slower: 1081 -> 1115 us).
    if (ROWS) {
        if (pm.row >= nr) return;
    } else if (!pm.on) {
        pdl_wait();
        return;
    }
    const int t = pm.t, w = pm.w, pidx = pm.pidx;
    const u64 q = mods[pidx].q;
    const ModF f = modf[pidx];
    u64 *p = data + pm.row * (long)N + (ROWS ? pm.seq * M : pm.seq);
    const ulonglong2 *tab = tw2 + (long)pidx * (N + 256);
    if (STG) stage_twiddles<LM, ROWS>(stg, tab, items);
    const PassTw<LM, ROWS, STG> tw{
        STG ? stg + (ROWS ? (w % (G_::W / items)) * M : 0) : ROWS ? tab + 256 + pm.seq * M : tab, t};
    pdl_wait();
    if (ROWS && SUBSC && pm.on && threadIdx.x % (256 / items) == 0) {
        // the epilogue's operands (this item's sequences of u, and of the
        // addend) are contiguous: have the copy engine bring them into L2
        // while the butterflies run, so the epilogue does not wait on DRAM
        const u32 arow = ep.row0 + (u32)pm.row, it = arow / (u32)ep.rows_per_item;
        const long off = (long)(arow - it * (u32)ep.rows_per_item) * N + pm.seq * M;
        const u32 bytes = (u32)(G_::W / items) * M * 8;
        bc_prefetch_l2(ep.u + it * ep.us + off, bytes);
        if (ep.add) bc_prefetch_l2(ep.add + it * ep.as + off, bytes);
    }
    u64 x[16];
#pragma unroll
    for (int k = 0; k < 16; k++) {
        if (ROWS) x[k] = p[t + T * k];
        else x[k] = p[(long)(t + T * k) << LS];
    }
    if (STG) {
        staged_wait();
        __syncthreads();
    }
    const u64 wone = mods[pidx].wone;
    const int ar = ntt_arith(q, f);
#define FWD_TILE(AR) \
    fwd_tile<LM, LS, ROWS, STG, AR, SUBSC>(x, sm, tw, t, w, p, pm.on, pm.row, pm.seq, N, q, wone, f, ep)
    if (ar == AR_FQ) FWD_TILE(AR_FQ);
    else if (ar == AR_LAZY) FWD_TILE(AR_LAZY);
    else FWD_TILE(AR_RED);
#undef FWD_TILE
}

// One block of inverse stages on the 16 words of a thread: butterflies of
// pair distance S0 .. S1 (doubling), the twiddle of pair j at distance s being
// tw(s, j).
//
// Float-quotient limbs: sums are not reduced within a block.  From |x| <= q at
// most three sums in a row meet a product, |x - y| <= 16 q, and after the
// block the words whose last butterfly was a sum (k & S1 == 0) are reduced, so
// that every word enters the next block below q again.
template <int AR, int S0, int S1, class Tw>
__device__ __forceinline__ void inv_stages(u64 (&x)[16], u64 q, const ModF &f, Tw tw) {
#pragma unroll
    for (int s = S0; s <= S1; s <<= 1) {
#pragma unroll
        for (int k = 0; k < 16; k++)
            if (!(k & s)) {
                const ulonglong2 wv = tw(s, k / (2 * s));
                if constexpr (AR == AR_FQ) {
                    const u64 a = x[k], d = a - x[k + s];
                    x[k] = a + x[k + s];
                    x[k + s] = fq_mul(d, wv, f);
                } else {
                    bf_inv4(x[k], x[k + s], wv.x, wv.y, q);
                }
            }
    }
}

// The stages and stores of one tile whose words are in x in layout B.
template <int LM, int LS, bool ROWS, bool STG, int AR>
__device__ __forceinline__ void inv_tile(u64 (&x)[16], u64 *sm, const PassTw<LM, ROWS, STG> &tw, int t, int w, u64 *p,
                                         bool on, u64 q, const ModF &f, const u64 *ninv,
                                         const ulonglong2 *ninvf) {
    typedef PassGeom<LM, ROWS> G_;
    constexpr int T = G_::T;
    inv_stages<AR, 1, T / 2>(x, q, f, [&](int sp, int j) { return tw.b(sp, j); });
    if constexpr (AR == AR_FQ) {
#pragma unroll
        for (int k = 0; k < 16; k++)
            if (!(k & (T / 2))) x[k] = fq_red(x[k], f);
    }
#pragma unroll
    for (int k = 0; k < 16; k++) sm[G_::sidx(16 * t + k, w)] = x[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; k++) x[k] = sm[G_::sidx(t + T * k, w)];
    auto ta = [&](int s, int j) { return tw.a(s, j); };
    if constexpr (!ROWS && AR == AR_FQ) {
        // the transform's last stage carries N^-1: its sums times N^-1, its
        // differences times N^-1 times the stage's twiddle
        inv_stages<AR, 1, 4>(x, q, f, ta);
        const ulonglong2 n0 = ninvf[0], n1 = ninvf[1];
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const u64 a = x[k], b = x[k + 8];
            x[k] = fq_pos(fq_mul(a + b, n0, f), q);
            x[k + 8] = fq_pos(fq_mul(a - b, n1, f), q);
        }
    } else {
        inv_stages<AR, 1, 8>(x, q, f, ta);
        if constexpr (AR == AR_FQ) {
#pragma unroll
            for (int k = 0; k < 8; k++) x[k] = fq_red(x[k], f);
        } else if constexpr (!ROWS) {
            const u64 ni = ninv[0], nip = ninv[1];
#pragma unroll
            for (int k = 0; k < 16; k++) x[k] = shoup(x[k], ni, nip, q);
        }
    }
    if (!on) return;
    u64 *ps = ROWS ? p + t : p + ((long)t << LS);
    if (!ROWS) asm volatile("" : "+l"(ps));   // as in fwd_tile
#pragma unroll
    for (int k = 0; k < 16; k++) ps[ROWS ? T * k : (T * k) << LS] = x[k];
}

template <int LM, int LS, bool ROWS, bool STG, int MINB>
__global__ void __launch_bounds__(256, MINB) k_ntt_inv_fast(u64 *data, RowMap rm, long nr, int items, NttSrc src,
                                                            const ModQ *mods, const ModF *modf,
                                                            const ulonglong2 *tw2, const u64 *ninv,
                                                            const ulonglong2 *ninvf, int logN) {
    typedef PassGeom<LM, ROWS> G_;
    constexpr int M = G_::M, T = G_::T;
    extern __shared__ __align__(16) u64 sm[];
    ulonglong2 *stg = (ulonglong2 *)(sm + G_::SM);
    const int N = 1 << logN;
    pdl_trigger();
    const PassMap<LM, ROWS> pm(rm, nr, items, RowSkip());
    if (ROWS && pm.row >= nr) return;   // a group past the launch's end, as above
    const int t = pm.t, w = pm.w, pidx = pm.pidx;
    const u64 q = mods[pidx].q;
    const ModF f = modf[pidx];
    u64 *p = data + pm.row * (long)N + (ROWS ? pm.seq * M : pm.seq);
    const ulonglong2 *tab = tw2 + (long)pidx * (N + 256);
    if (STG) stage_twiddles<LM, ROWS>(stg, tab, items);
    const PassTw<LM, ROWS, STG> tw{
        STG ? stg + (ROWS ? (w % (G_::W / items)) * M : 0) : ROWS ? tab + 256 + pm.seq * M : tab, t};
    u64 x[16];
    pdl_wait();
    if (ROWS) {
        const u64 *in = p;
        if (src.src) {
            const u32 r = src.row0 + (u32)pm.row, it = r / (u32)src.rows_per_item;
            in = src.src + it * src.stride + (long)(r - it * src.rows_per_item) * N + pm.seq * M;
        }
#pragma unroll
        for (int k = 0; k < 16; k++) sm[G_::sidx(t + T * k, w)] = in[t + T * k];
        if (STG) staged_wait();
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 16; k++) x[k] = sm[G_::sidx(16 * t + k, w)];
    } else {
#pragma unroll
        for (int k = 0; k < 16; k++) x[k] = p[(16L * t + k) << LS];
        if (STG) {
            staged_wait();
            __syncthreads();
        }
    }
    if (f.on) inv_tile<LM, LS, ROWS, STG, AR_FQ>(x, sm, tw, t, w, p, pm.on, q, f, ninv + 2 * pidx, ninvf + 2 * pidx);
    else inv_tile<LM, LS, ROWS, STG, AR_LAZY>(x, sm, tw, t, w, p, pm.on, q, f, ninv + 2 * pidx, ninvf + 2 * pidx);
}

// The build of a launch: 2, 3 or 4 CTAs per SM as pinned or tuned on a large
// launch (2, 3, 5), but the one with the most registers where the whole grid
// fits the GPU at once and a CTA's own latency is what counts.
static int pass_build(const Ctx *ctx, int minb, dim3 grid) {
    return !ctx->ntt_pinned && (long)grid.x * grid.y <= 2L * ctx->nsm ? 2 : minb;
}
// Whether a row pass stages its twiddles: 64 KB for one item per CTA leave 2
// CTAs per SM, which only a small grid does not miss.
static bool pass_staged(const Ctx *ctx, int items, dim3 grid) {
    return items > 1 || (long)grid.x * grid.y <= 2L * ctx->nsm;
}

// One launch; a kernel's shared-memory limit is raised once per device (the
// attribute is per kernel instantiation: KERN is part of this function's type).
template <auto KERN, class... A>
static void pass_launch(const Ctx *ctx, dim3 grid, size_t smem, cudaStream_t st, A... args) {
    static std::atomic<bool> raised[64];
    if (smem > 48 * 1024 && !raised[ctx->device & 63].load(std::memory_order_acquire)) {
        cudaFuncSetAttribute(KERN, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
        raised[ctx->device & 63].store(true, std::memory_order_release);
    }
    launch_pdl(KERN, grid, 256, smem, st, args...);
}

template <int LM, int LS, bool ROWS, bool STG, bool SUB>
static void fwd_pass_launch(Ctx *ctx, u64 *d, long nr, const RowMap &m, cudaStream_t st, const RowSkip &sk,
                            const SubScale &e, int items, dim3 grid) {
    typedef PassGeom<LM, ROWS> G_;
    const size_t smem = G_::SM * 8 + (STG ? (ROWS ? G_::W / items : 1) * G_::M * 16 : 0);
    const int minb = pass_build(ctx, ctx->ntt_minb, grid);
#define FWD_LAUNCH(MINB)                                                                                     \
    pass_launch<k_ntt_fwd_fast<LM, LS, ROWS, STG, MINB, SUB>>(ctx, grid, smem, st, d, m, nr, items,            \
                (const ModQ *)ctx->d_mod, (const ModF *)ctx->d_modf, (const ulonglong2 *)ctx->d_psi2, ctx->logN, sk, e)
    if (minb == 3) FWD_LAUNCH(3);
    else if (minb == 5) FWD_LAUNCH(4);
    else FWD_LAUNCH(2);
#undef FWD_LAUNCH
}

template <int LM, int LS, bool ROWS>
static void fwd_pass(Ctx *ctx, u64 *d, long nr, const RowMap &m, cudaStream_t st, const RowSkip &sk,
                     const SubScale *ep = nullptr) {
    const SubScale e = ep ? *ep : SubScale();
    const int items = ROWS ? pass_items(m.n, nr) : 1;
    const dim3 grid = PassMap<LM, ROWS>::grid(ctx->N, m.n, nr, items);
    if constexpr (ROWS) {
        if (pass_staged(ctx, items, grid)) {
            if (ep) fwd_pass_launch<LM, LS, true, true, true>(ctx, d, nr, m, st, sk, e, items, grid);
            else fwd_pass_launch<LM, LS, true, true, false>(ctx, d, nr, m, st, sk, e, items, grid);
        } else {
            if (ep) fwd_pass_launch<LM, LS, true, false, true>(ctx, d, nr, m, st, sk, e, items, grid);
            else fwd_pass_launch<LM, LS, true, false, false>(ctx, d, nr, m, st, sk, e, items, grid);
        }
    } else {
        // staged columns: 17.5 -> 16.7 us for the two passes of 4 rows, but
        // 566 -> 584 us for 1024 rows of N = 2^16, whose CTAs find the
        // prime's 4 KB in L1
        if (pass_staged(ctx, 1, grid)) fwd_pass_launch<LM, LS, false, true, false>(ctx, d, nr, m, st, sk, e, items, grid);
        else fwd_pass_launch<LM, LS, false, false, false>(ctx, d, nr, m, st, sk, e, items, grid);
    }
}

template <int LM, int LS, bool ROWS, bool STG>
static void inv_pass_launch(Ctx *ctx, u64 *d, long nr, const RowMap &m, cudaStream_t st, int items, dim3 grid,
                            const NttSrc &src) {
    typedef PassGeom<LM, ROWS> G_;
    const size_t smem = G_::SM * 8 + (STG ? (ROWS ? G_::W / items : 1) * G_::M * 16 : 0);
    const int minb = pass_build(ctx, ctx->ntt_minb_inv, grid);
#define INV_LAUNCH(MINB)                                                                                     \
    pass_launch<k_ntt_inv_fast<LM, LS, ROWS, STG, MINB>>(ctx, grid, smem, st, d, m, nr, items, src,            \
                (const ModQ *)ctx->d_mod, (const ModF *)ctx->d_modf, (const ulonglong2 *)ctx->d_ipsi2,       \
                (const u64 *)ctx->d_ninv, (const ulonglong2 *)ctx->d_ninvf, ctx->logN)
    if (minb == 3) INV_LAUNCH(3);
    else if (minb == 5) INV_LAUNCH(4);
    else INV_LAUNCH(2);
#undef INV_LAUNCH
}

template <int LM, int LS, bool ROWS>
static void inv_pass(Ctx *ctx, u64 *d, long nr, const RowMap &m, cudaStream_t st, const NttSrc &src = NttSrc()) {
    const int items = ROWS ? pass_items(m.n, nr) : 1;
    const dim3 grid = PassMap<LM, ROWS>::grid(ctx->N, m.n, nr, items);
    if constexpr (ROWS) {
        if (pass_staged(ctx, items, grid)) inv_pass_launch<LM, LS, true, true>(ctx, d, nr, m, st, items, grid, src);
        else inv_pass_launch<LM, LS, true, false>(ctx, d, nr, m, st, items, grid, src);
    } else {
        inv_pass_launch<LM, LS, false, true>(ctx, d, nr, m, st, items, grid, src);
    }
}

// ------------------------------------------------------ integer roofline
// Peak rate of the forward butterfly that the NTT runs on the 40-bit limbs
// (one float-quotient product and two additions) with operands in registers:
// 16 independent chains per thread, `iters` rounds, every SM filled.  The
// values leave the product's range after a few rounds; only the instruction
// stream matters.  The result is the denominator of the NTT's "alu" roofline.
__global__ void __launch_bounds__(256, 3) k_bfly_peak(u64 *sink, int iters, const ModF f, ulonglong2 tw) {
    u64 x[16];
#pragma unroll
    for (int k = 0; k < 16; k++) x[k] = threadIdx.x * 16 + k;
    tw.x += threadIdx.x;   // per-thread operands, as in the transform
    for (int it = 0; it < iters; it++) {
#pragma unroll
        for (int k = 0; k < 16; k += 2) bf_fwd_ar<AR_FQ>(x[k], x[k + 1], tw, 0, f);
#pragma unroll
        for (int k = 0; k < 16; k += 4) {
            bf_fwd_ar<AR_FQ>(x[k], x[k + 2], tw, 0, f);
            bf_fwd_ar<AR_FQ>(x[k + 1], x[k + 3], tw, 0, f);
        }
    }
    u64 acc = 0;
#pragma unroll
    for (int k = 0; k < 16; k++) acc ^= x[k];
    if (acc == 0x1234567ull) sink[0] = acc;  // keeps the work alive
}

double bfly_peak(int iters) {
    const u64 q = 1099510054913ull;  // a 40-bit prime = 1 mod 2^17
    const u64 w = 123456789012345ull % q;
    const ModF f = h_modf(q);
    const ulonglong2 tw = h_fq(w, q);
    int nsm = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    u64 *sink;
    cudaMalloc(&sink, 8);
    const int blocks = nsm * 8, threads = 256;
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    k_bfly_peak<<<blocks, threads>>>(sink, 16, f, tw);  // warm-up
    cudaEventRecord(a);
    k_bfly_peak<<<blocks, threads>>>(sink, iters, f, tw);
    cudaEventRecord(b);
    cudaEventSynchronize(b);
    float ms = 0;
    cudaEventElapsedTime(&ms, a, b);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    cudaFree(sink);
    double bfly = (double)blocks * threads * iters * 16.0;  // 8 + 8 butterflies per round
    return bfly / (ms * 1e-3);
}

// ----------------------------------------------------------------- launch
static void split(int logN, int &logN1, int &C, int &R) {
    logN1 = logN / 2;
    int N1 = 1 << logN1, N2 = 1 << (logN - logN1);
    C = 2048 / N1;
    if (C < 1) C = 1;
    if (C > N2) C = N2;
    R = 2048 / N2;
    if (R < 1) R = 1;
    if (R > N1) R = N1;
}

// Both passes over nr rows (at most 65535) of N = 2^14 .. 2^16: columns of
// 128 or 256 words first, then rows.
static void fwd_both(Ctx *ctx, u64 *d, long nr, const RowMap &m, cudaStream_t st, const RowSkip &sk,
                     const SubScale *ep) {
    if (ctx->logN == 16) fwd_pass<8, 8, false>(ctx, d, nr, m, st, sk);
    else if (ctx->logN == 15) fwd_pass<7, 8, false>(ctx, d, nr, m, st, sk);
    else fwd_pass<7, 7, false>(ctx, d, nr, m, st, sk);
    if (ctx->logN >= 15) fwd_pass<8, 0, true>(ctx, d, nr, m, st, sk, ep);
    else fwd_pass<7, 0, true>(ctx, d, nr, m, st, sk, ep);
}
static void inv_both(Ctx *ctx, u64 *d, long nr, const RowMap &m, cudaStream_t st, const NttSrc &src = NttSrc()) {
    if (ctx->logN >= 15) inv_pass<8, 0, true>(ctx, d, nr, m, st, src);
    else inv_pass<7, 0, true>(ctx, d, nr, m, st, src);
    if (ctx->logN == 16) inv_pass<8, 8, false>(ctx, d, nr, m, st);
    else if (ctx->logN == 15) inv_pass<7, 8, false>(ctx, d, nr, m, st);
    else inv_pass<7, 7, false>(ctx, d, nr, m, st);
}

// Picks the CTAs per SM (2, 3 or 4) of the register-blocked passes, forward
// and inverse separately: each variant transforms 1024 rows over the
// context's whole chain (the 40-bit limbs run the non-reducing butterflies,
// as in Decompose), 3 repetitions, fastest kept.
static void tune_ntt(Ctx *ctx, cudaStream_t st) {
    ctx->ntt_tuned = true;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaStreamIsCapturing(st, &cap);
    if (cap != cudaStreamCaptureStatusNone) {
        ctx->ntt_tuned = false;
        return;
    }
    const long R = 1024;
    Buf scratch(&ctx->pool, (size_t)R * ctx->N);
    // any words do for timing; 0x15.. keeps them below the 60-bit primes
    cudaMemsetAsync(scratch.p, 0x15, (size_t)R * ctx->N * 8, st);
    RowMap m = ctx->map_qp(ctx->L);
    RowSkip none;
    cudaEvent_t a = ctx->ev_get(), b = ctx->ev_get();
    for (int dir = 0; dir < 2; dir++) {
        float best = 1e30f;
        int pick = 2;
        for (int minb : {2, 3, 5}) {
            (dir == 0 ? ctx->ntt_minb : ctx->ntt_minb_inv) = minb;
            float t = 1e30f;
            for (int rep = 0; rep < 3; rep++) {
                cudaEventRecord(a, st);
                if (dir == 0) fwd_both(ctx, scratch.p, R, m, st, none, nullptr);
                else inv_both(ctx, scratch.p, R, m, st);
                cudaEventRecord(b, st);
                cudaEventSynchronize(b);
                float ms = 0;
                cudaEventElapsedTime(&ms, a, b);
                t = std::min(t, ms);
                ctx->n_launch += 2;
            }
            char line[112];
            snprintf(line, sizeof line, "ntt %s logN %d rows %ld ctas_per_sm %d ms %.4f\n", dir ? "inverse" : "forward",
                     ctx->logN, R, minb == 5 ? 4 : minb, t);
            ctx->tune_log += line;
            if (t < best) best = t, pick = minb;
        }
        (dir == 0 ? ctx->ntt_minb : ctx->ntt_minb_inv) = pick;
        // then the rows per launch pair: all, or chunks of 96 or 48 MiB
        // whose pass-0 output pass 1 still finds in L2
        int &chunk = dir == 0 ? ctx->ntt_chunk : ctx->ntt_chunk_inv;
        int cpick = 0;
        for (long mb : {0L, 96L, 48L}) {
            const int c = mb ? (int)std::max(1L, (mb << 20) / (8L * ctx->N)) : 0;
            if (c >= R) continue;
            chunk = c;
            float t = 1e30f;
            for (int rep = 0; rep < 3; rep++) {
                cudaEventRecord(a, st);
                const long step = c ? c : R;
                for (long r0 = 0; r0 < R; r0 += step) {
                    const long nr = std::min(step, R - r0);
                    u64 *d = scratch.p + r0 * (long)ctx->N;
                    RowMap mm = m.shifted(r0);
                    if (dir == 0) fwd_both(ctx, d, nr, mm, st, none, nullptr);
                    else inv_both(ctx, d, nr, mm, st);
                }
                cudaEventRecord(b, st);
                cudaEventSynchronize(b);
                float ms = 0;
                cudaEventElapsedTime(&ms, a, b);
                t = std::min(t, ms);
            }
            char line[112];
            snprintf(line, sizeof line, "ntt %s logN %d rows %ld rows_per_launch %d ms %.4f\n",
                     dir ? "inverse" : "forward", ctx->logN, R, c ? c : (int)R, t);
            ctx->tune_log += line;
            if (mb == 0 || t < best) best = t, cpick = c;
        }
        chunk = cpick;
    }
    ctx->ev_free.push_back(a);
    ctx->ev_free.push_back(b);
}

void ntt_fwd(Ctx *ctx, u64 *data, long rows, const RowMap &rm, cudaStream_t st, const RowSkip *skip) {
    if (rows <= 0) return;
    if (ctx->autotune && !ctx->ntt_tuned && ctx->logN >= 14 && ctx->logN <= 16) tune_ntt(ctx, st);
    int logN = ctx->logN, logN1, C, R;
    split(logN, logN1, C, R);
    int N1 = 1 << logN1, N2 = 1 << (logN - logN1);
    const long chunk = ctx->ntt_chunk > 0 && ctx->ntt_chunk < 65535 ? ctx->ntt_chunk : 65535;
    for (long r0 = 0; r0 < rows; r0 += chunk) {
        long nr = rows - r0 < chunk ? rows - r0 : chunk;
        u64 *d = data + r0 * (long)ctx->N;
        RowMap m = rm.shifted(r0);
        ctx->n_launch += 2;
        cudaEvent_t e0;
        ctx->trace_begin(1, e0);
        if (logN >= 14 && logN <= 16) {
            RowSkip sk;
            long done = nr;
            if (skip) {
                sk = *skip;
                sk.row0 = (unsigned)(r0 % ((long)sk.ndig * sk.rows_per_digit));
                done = 0;
                for (long r = 0; r < nr; r++) done += !sk.skip((unsigned)r);
            }
            fwd_both(ctx, d, nr, m, st, sk, nullptr);
            // algorithmic bytes: every transformed word read and written once
            // (the two passes move twice that)
            ctx->trace_end(1, e0, 2.0 * done * ctx->N * 8.0);
            continue;
        }
        if (skip) throw std::logic_error("row skipping needs the register-blocked NTT (logN 14..16)");
        k_ntt_fwd_p1<<<dim3(N2 / C, (unsigned)nr), 256, N1 * C * 8, st>>>(d, m, ctx->d_mod, ctx->d_psi,
                                                                       ctx->d_psip, logN, logN1, C);
        k_ntt_fwd_p2<<<dim3(N1 / R, (unsigned)nr), 256, R * N2 * 8, st>>>(d, m, ctx->d_mod, ctx->d_psi,
                                                                       ctx->d_psip, logN, logN1, R);
    }
}

void ntt_fwd_subscale(Ctx *ctx, u64 *data, long rows, const RowMap &rm, cudaStream_t st, const SubScale &ep) {
    if (rows <= 0) return;
    if (ctx->autotune && !ctx->ntt_tuned && ctx->logN >= 14 && ctx->logN <= 16) tune_ntt(ctx, st);
    int logN = ctx->logN, logN1, C, R;
    split(logN, logN1, C, R);
    if (logN < 14 || logN > 16) throw std::logic_error("the fused NTT epilogue needs the register-blocked NTT");
    const long chunk = ctx->ntt_chunk > 0 && ctx->ntt_chunk < 65535 && !ep.n_out ? ctx->ntt_chunk : 65535;
    for (long r0 = 0; r0 < rows; r0 += chunk) {
        long nr = rows - r0 < chunk ? rows - r0 : chunk;
        u64 *d = data + r0 * (long)ctx->N;
        RowMap m = rm.shifted(r0);
        // the chunk's rows counted from the item it starts in
        SubScale e = ep;
        const long i0 = r0 / ep.rows_per_item;
        if (ep.n_out && r0) throw std::logic_error("separate outputs take one launch");
        e.u += i0 * ep.us, e.out += i0 * ep.os;
        if (e.add) e.add += i0 * ep.as;
        e.row0 = (unsigned)(r0 - i0 * ep.rows_per_item);
        ctx->n_launch += 2;
        cudaEvent_t e0;
        ctx->trace_begin(1, e0);
        RowSkip none;
        fwd_both(ctx, d, nr, m, st, none, &e);
        // algorithmic bytes of the transform: every word read and written once
        // (the fused epilogue's read of u is not counted, so butterflies per
        // traced byte stay those of a plain transform)
        ctx->trace_end(1, e0, 2.0 * nr * ctx->N * 8.0);
    }
}

void ntt_inv(Ctx *ctx, u64 *data, long rows, const RowMap &rm, cudaStream_t st, const NttSrc &src) {
    if (rows <= 0) return;
    if (src.src && (ctx->logN < 14 || ctx->logN > 16)) {   // the shared-memory passes work in place
        launch_copy_rows(data, (long)src.rows_per_item * ctx->N, src.src, src.stride, (int)(rows / src.rows_per_item),
                         (long)src.rows_per_item * ctx->N, st);
        ntt_inv(ctx, data, rows, rm, st);
        return;
    }
    if (ctx->autotune && !ctx->ntt_tuned && ctx->logN >= 14 && ctx->logN <= 16) tune_ntt(ctx, st);
    int logN = ctx->logN, logN1, C, R;
    split(logN, logN1, C, R);
    int N1 = 1 << logN1, N2 = 1 << (logN - logN1);
    const long chunk = ctx->ntt_chunk_inv > 0 && ctx->ntt_chunk_inv < 65535 ? ctx->ntt_chunk_inv : 65535;
    for (long r0 = 0; r0 < rows; r0 += chunk) {
        long nr = rows - r0 < chunk ? rows - r0 : chunk;
        u64 *d = data + r0 * (long)ctx->N;
        RowMap m = rm.shifted(r0);
        ctx->n_launch += 2;
        cudaEvent_t e0;
        ctx->trace_begin(2, e0);
        if (logN >= 14 && logN <= 16) {
            // a chunk starts at row r0: the item it lies in, and its row there
            NttSrc s = src;
            if (s.src) {
                const long it = r0 / s.rows_per_item;
                s.src += it * s.stride, s.row0 = (unsigned)(r0 - it * s.rows_per_item);
            }
            inv_both(ctx, d, nr, m, st, s);
            ctx->trace_end(2, e0, 2.0 * nr * ctx->N * 8.0);
            continue;
        }
        k_ntt_inv_p2<<<dim3(N1 / R, (unsigned)nr), 256, R * N2 * 8, st>>>(d, m, ctx->d_mod, ctx->d_ipsi,
                                                                       ctx->d_ipsip, logN, logN1, R);
        k_ntt_inv_p1<<<dim3(N2 / C, (unsigned)nr), 256, N1 * C * 8, st>>>(d, m, ctx->d_mod, ctx->d_ipsi,
                                                                       ctx->d_ipsip, ctx->d_ninv, logN,
                                                                       logN1, C);
    }
}

}  // namespace he

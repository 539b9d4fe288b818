// relin.cu -- the sum of relinearised products  sum_k Mult(A^(k), B^(k)) of a
// matrix product (Sec. 4.3 DMatrixMult; App. A Mult, KeySwitch), for runs of k.
//
// Every term is relinearised by itself, KeySwitch(d2_k, rlk) = ModDown(sum_d
// digit_{k,d} rlk_d), and the terms are added mod q.  What the paper rounds per
// term are integers: the conversions' sources y.  Everything between them is
// linear mod q, so the residues of the sum are the same when the linear parts
// run once on summed integers:
//   * Decompose's extended rows are sum_i y_{k,i} w_{i,r} mod r: on the rows of Q
//     they only enter sum_k, so the integers y_{k,i} are summed over k and
//     converted and transformed once.  The P rows are needed term by term.
//   * ModDown's input on the rows of Q only enters sum_k; its P rows give, term
//     by term, the integers y_{k,j} and the overflow count e_k (exact), which
//     are summed and converted once.
// Per term this leaves the inverse NTT of d2_k, ndig alpha rows of forward
// NTT, the inner product and 2 alpha rows of inverse NTT on the P rows, in
// place of ndig (l + 1 + alpha) - (l + 1) + 2 (l + 1) rows of forward NTT and the
// inner product on every row: 20 instead of 229 rows at level 18 with alpha = 2.
// The integer sums are kept as two words (sums of low and of high 32 bits,
// below 2^40 for up to kRelinTerms terms; n <= 181 at the ring degrees of this path).
#include "eval.h"
#include "kernels.cuh"

namespace he {

// ------------------------------------------------------------ tensor of a run
// For products p = A[ia[p]] B[ib[p]] of the terms kk < K: d01[p] (+)= sum_kk (d0,
// d1), D2[p] (+)= sum_kk d2, and d2[kk][p] unless null.  a: [K][nA] ciphertexts
// of `limbs` limbs; b: [K][nB] ciphertexts at stride bs, b's polynomials bp words
// apart.  The products of a 40-bit limb take one float quotient each, with
// 1/q of the second factor formed on the fly (43 -> 14 multiply slots).
constexpr int kPairs = 64;
struct PairIdx {
    short a[kPairs], b[kPairs];
};

template <bool D2K>
__global__ void __launch_bounds__(256) k_tensor_run(u64 *d01, u64 *D2, u64 *d2, const u64 *a, const u64 *b, int K,
                                                    int P, int p0, int nA, int nB, int limbs, int logN, long bs,
                                                    long bp, const __grid_constant__ PairIdx ix, const ModQ *mods,
                                                    const ModF *modf, int accumulate) {
    pdl_trigger();
    pdl_wait();
    const long N = 1L << logN;
    const int x = 2 * (blockIdx.x * 256 + threadIdx.x);   // 256 | N / 2
    const int r = blockIdx.y, p = p0 + blockIdx.z;
    const ModQ m = mods[r];
    const ModF f = modf[r];
    const long as = 2L * limbs * N, ro = (long)r * N + x;
    const u64 *ap = a + (long)ix.a[blockIdx.z] * as + ro, *bq = b + (long)ix.b[blockIdx.z] * bs + ro;
    u64 s0[2] = {0, 0}, s1[2] = {0, 0}, s2[2] = {0, 0};
    if (f.on) {   // uniform over the CTA
        const float c = f.qi * 1.4901161193847656e-08f;   // 2^6 / q from 2^32 / q
        for (int k = 0; k < K; k++) {
            const ulonglong2 a0 = *(const ulonglong2 *)(ap + (long)k * nA * as);
            const ulonglong2 a1 = *(const ulonglong2 *)(ap + (long)k * nA * as + limbs * N);
            const ulonglong2 b0 = *(const ulonglong2 *)(bq + (long)k * nB * bs);
            const ulonglong2 b1 = *(const ulonglong2 *)(bq + (long)k * nB * bs + bp);
            u64 o[2];
#pragma unroll
            for (int j = 0; j < 2; j++) {
                const u64 u0 = j ? a0.y : a0.x, u1 = j ? a1.y : a1.x;
                const ulonglong2 v0 = fq_svar(j ? b0.y : b0.x, c), v1 = fq_svar(j ? b1.y : b1.x, c);
                // each product below q in magnitude: 16 terms stay below 17 q
                if (k && !(k & 7)) s0[j] = fq_red(s0[j], f), s1[j] = fq_red(s1[j], f), s2[j] = fq_red(s2[j], f);
                s0[j] += fq_mul(u0, v0, f);
                s1[j] += fq_mul(u0, v1, f) + fq_mul(u1, v0, f);
                const u64 t = fq_mul(u1, v1, f);
                s2[j] += t;
                if (D2K) o[j] = fq_pos(t, m.q);
            }
            if (D2K) *(ulonglong2 *)(d2 + ((long)k * P + p) * limbs * N + ro) = make_ulonglong2(o[0], o[1]);
        }
#pragma unroll
        for (int j = 0; j < 2; j++) {
            s0[j] = fq_pos(fq_red(s0[j], f), m.q);
            s1[j] = fq_pos(fq_red(s1[j], f), m.q);
            s2[j] = fq_pos(fq_red(s2[j], f), m.q);
        }
    } else {
        for (int k = 0; k < K; k++) {
            const ulonglong2 a0 = *(const ulonglong2 *)(ap + (long)k * nA * as);
            const ulonglong2 a1 = *(const ulonglong2 *)(ap + (long)k * nA * as + limbs * N);
            const ulonglong2 b0 = *(const ulonglong2 *)(bq + (long)k * nB * bs);
            const ulonglong2 b1 = *(const ulonglong2 *)(bq + (long)k * nB * bs + bp);
            u64 o[2];
#pragma unroll
            for (int j = 0; j < 2; j++) {
                const u64 u0 = j ? a0.y : a0.x, u1 = j ? a1.y : a1.x, v0 = j ? b0.y : b0.x, v1 = j ? b1.y : b1.x;
                s0[j] = addmod(s0[j], mulmod(u0, v0, m), m.q);
                s1[j] = addmod(s1[j], addmod(mulmod(u0, v1, m), mulmod(u1, v0, m), m.q), m.q);
                o[j] = mulmod(u1, v1, m);
                s2[j] = addmod(s2[j], o[j], m.q);
            }
            if (D2K) *(ulonglong2 *)(d2 + ((long)k * P + p) * limbs * N + ro) = make_ulonglong2(o[0], o[1]);
        }
    }
    u64 *o0 = d01 + (long)p * as + ro, *o1 = o0 + limbs * N, *o2 = D2 + (long)p * limbs * N + ro;
    if (accumulate) {
        const ulonglong2 v0 = *(ulonglong2 *)o0, v1 = *(ulonglong2 *)o1, v2 = *(ulonglong2 *)o2;
        s0[0] = addmod(s0[0], v0.x, m.q), s0[1] = addmod(s0[1], v0.y, m.q);
        s1[0] = addmod(s1[0], v1.x, m.q), s1[1] = addmod(s1[1], v1.y, m.q);
        s2[0] = addmod(s2[0], v2.x, m.q), s2[1] = addmod(s2[1], v2.y, m.q);
    }
    *(ulonglong2 *)o0 = make_ulonglong2(s0[0], s0[1]);
    *(ulonglong2 *)o1 = make_ulonglong2(s1[0], s1[1]);
    *(ulonglong2 *)o2 = make_ulonglong2(s2[0], s2[1]);
}

void launch_tensor_run(Ctx *c, u64 *d01, u64 *D2, u64 *d2, const u64 *a, const u64 *b, int K, int P, int nA, int nB,
                       const int *ia, const int *ib, int limbs, long bs, long bp, bool accumulate) {
    for (int p0 = 0; p0 < P; p0 += kPairs) {
        const int n = std::min(kPairs, P - p0);
        PairIdx ix;
        for (int i = 0; i < n; i++) ix.a[i] = (short)ia[p0 + i], ix.b[i] = (short)ib[p0 + i];
        const dim3 grid((unsigned)(c->N / 512), (unsigned)limbs, (unsigned)n);
        c->n_launch++;
        if (d2)
            launch_pdl(k_tensor_run<true>, dim3(grid), 256, 0, c->stream, d01, D2, d2, a, b, K, P, p0, nA, nB, limbs, c->logN, bs, bp,
                                                            ix, c->d_mod, c->d_modf, accumulate);
        else
            launch_pdl(k_tensor_run<false>, dim3(grid), 256, 0, c->stream, d01, D2, d2, a, b, K, P, p0, nA, nB, limbs, c->logN, bs,
                                                             bp, ix, c->d_mod, c->d_modf, accumulate);
    }
}

// Tensors of separate ciphertexts: d01 [n][2][limbs][N], d2 [n][limbs][N] of
// a[i] b[i], each given by its first polynomial and the distance of its second.
struct MultPtrs {
    const u64 *a[kMultMany], *b[kMultMany];
    long as[kMultMany], bs[kMultMany];
};
__global__ void __launch_bounds__(256) k_tensor_ptrs(u64 *d01, u64 *d2, const __grid_constant__ MultPtrs mp, int limbs,
                                                     int logN, const ModQ *mods, const ModF *modf) {
    pdl_trigger();
    pdl_wait();
    const long N = 1L << logN;
    const int r = blockIdx.y, i = blockIdx.z;
    const long ro = (long)r * N + blockIdx.x * 256 + threadIdx.x;   // 256 | N
    const ModQ m = mods[r];
    const ModF f = modf[r];
    const u64 a0 = mp.a[i][ro], a1 = mp.a[i][ro + mp.as[i]], b0 = mp.b[i][ro], b1 = mp.b[i][ro + mp.bs[i]];
    u64 o0, o1, o2;
    if (f.on) {   // uniform over the CTA
        const float c = f.qi * 1.4901161193847656e-08f;   // 2^6 / q
        const ulonglong2 v0 = fq_svar(b0, c), v1 = fq_svar(b1, c);
        o0 = fq_pos(fq_mul(a0, v0, f), m.q);
        o1 = fq_pos(fq_red(fq_mul(a0, v1, f) + fq_mul(a1, v0, f), f), m.q);
        o2 = fq_pos(fq_mul(a1, v1, f), m.q);
    } else {
        o0 = mulmod(a0, b0, m);
        o1 = addmod(mulmod(a0, b1, m), mulmod(a1, b0, m), m.q);
        o2 = mulmod(a1, b1, m);
    }
    d01[((long)i * 2 * limbs) * N + ro] = o0;
    d01[((long)i * 2 * limbs + limbs) * N + ro] = o1;
    d2[(long)i * limbs * N + ro] = o2;
}

// out[i] [2][level][N] = Rescale(Mult(a[i], b[i])) at level `level` for n <= kMultMany
// pairs of ciphertexts at levels >= level: the words of mult_relin and rescale,
// with (d0, d1) lifted into the key switch's Q_l P sum (ModDown(u + P d) = d +
// ModDown(u)) so that one ModDown + rescale ends both.
void mult_rescale_many(Ctx *c, const u64 *const *a, const int *a_level, const u64 *const *b, const int *b_level, int n,
                       int level, u64 *const *out) {
    if (!c->rlk) throw HeError(HE_ERR_KEY_MISSING, "relinearisation key missing");
    const int nq = level + 1, rows = c->qp_rows(level);
    const size_t N = c->N;
    Buf d01(&c->pool, n * 2 * nq * N), d2(&c->pool, n * nq * N), dg(&c->pool, (size_t)n * c->ndig(level) * rows * N),
        u(&c->pool, n * 2 * rows * N);
    MultPtrs mp = {};
    for (int i = 0; i < n; i++) {
        mp.a[i] = a[i], mp.as[i] = (long)(a_level[i] + 1) * N;
        mp.b[i] = b[i], mp.bs[i] = (long)(b_level[i] + 1) * N;
    }
    c->n_launch++;
    launch_pdl(k_tensor_ptrs, dim3((unsigned)(N / 256), (unsigned)nq, (unsigned)n), 256, 0, c->stream, d01.p, d2.p, mp, nq,
               c->logN, c->d_mod, c->d_modf);
    modup(c, d2.p, (long)(nq * N), n, level, dg.p);
    launch_multsum(c, u.p, dg.p, c->rlk, 1u, n, level, nullptr, 0, c->stream);
    c->n_ms += n;
    launch_add_lifted(c, u.p, d01.p, n, level, c->stream);
    moddown_rescale(c, u.p, n, level, nullptr, out);
    c->n_md += n;
}

// ------------------------------------------------------- per-term conversions
// Decompose's integers of a run: d2 [K][P][nq][N] (coefficient form) -> SY
// [P][2][nq][N] (+)= sum_kk (low, high words of y_{kk,i}), and the P rows of the
// digits digP [K][P][ndig][A][N].  blockIdx.y is the digit.
template <int A>
__global__ void __launch_bounds__(256) k_relin_up(const u64 *d2, u64 *SY, u64 *digP, int K, int P, int level, int ndig,
                                                  int logN, int Lp1, const ModQ *mods, const ShoupPair *up_inv,
                                                  const ShoupPair *up_mod, int accumulate) {
    pdl_trigger();
    pdl_wait();
    const int nq = level + 1, rows = nq + A, d = blockIdx.y, i0 = d * A, ns = min(A, nq - i0);
    const long N = 1L << logN;
    ShoupPair inv[A], wp[A][A];   // wp[s][j]: (Q_d / q_s) mod p_j
    u64 qs[A], pj[A], p1[A];
#pragma unroll
    for (int s = 0; s < A; s++) {
        if (s < ns) inv[s] = up_inv[d * A + s], qs[s] = mods[i0 + s].q;
        pj[s] = mods[Lp1 + s].q, p1[s] = mods[Lp1 + s].wone;
#pragma unroll
        for (int j = 0; j < A; j++)
            if (s < ns) wp[s][j] = up_mod[((long)d * A + s) * rows + nq + j];
    }
    const long units = (long)P << logN;
    for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < units; idx += (long)gridDim.x * blockDim.x) {
        const int p = (int)(idx >> logN), x = (int)(idx & (N - 1));
        u64 lo[A], hi[A];
#pragma unroll
        for (int s = 0; s < A; s++) {
            lo[s] = hi[s] = 0;
            if (accumulate && s < ns) {
                lo[s] = SY[(((long)p * 2) * nq + i0 + s) * N + x];
                hi[s] = SY[(((long)p * 2 + 1) * nq + i0 + s) * N + x];
            }
        }
        for (int k = 0; k < K; k++) {
            const long it = (long)k * P + p;
            u64 y[A], acc[A];
#pragma unroll
            for (int j = 0; j < A; j++) acc[j] = 0;
#pragma unroll
            for (int s = 0; s < A; s++)
                if (s < ns) {
                    y[s] = shoup(d2[(it * nq + i0 + s) * N + x], inv[s].w, inv[s].wp, qs[s]);
                    lo[s] += (u32)y[s];
                    hi[s] += y[s] >> 32;
#pragma unroll
                    for (int j = 0; j < A; j++) acc[j] += shoup_lazy(y[s], wp[s][j].w, wp[s][j].wp, pj[j]);
                }
            u64 *o = digP + ((it * ndig + d) * A) * N + x;
#pragma unroll
            for (int j = 0; j < A; j++) o[j * N] = reduce_any(acc[j], pj[j], p1[j]);   // < 2 A p <= 8 p < 2^64
        }
#pragma unroll
        for (int s = 0; s < A; s++)
            if (s < ns) {
                SY[(((long)p * 2) * nq + i0 + s) * N + x] = lo[s];
                SY[(((long)p * 2 + 1) * nq + i0 + s) * N + x] = hi[s];
            }
    }
}

// ModDown's integers of a run: uP [K][P][2][A][N] (coefficient form) -> YP
// [P][2][2 A + 1][N] (+)= sum_kk (low words of y_j, high words of y_j, e).
template <int A>
__global__ void __launch_bounds__(256) k_relin_down(const u64 *uP, u64 *YP, int K, int P, int logN,
                                                    const __grid_constant__ MdExact k, int accumulate) {
    pdl_trigger();
    pdl_wait();
    const long N = 1L << logN;
    const long idx = (long)blockIdx.x * 256 + threadIdx.x;   // (p, poly, x): 256 | N
    const long pp = idx >> logN;
    const int x = (int)(idx & (N - 1));
    if (pp >= 2L * P) return;
    u64 *o = YP + pp * (2 * A + 1) * N + x;
    u64 s[2 * A + 1];
#pragma unroll
    for (int i = 0; i < 2 * A + 1; i++) s[i] = accumulate ? o[i * N] : 0;
    for (int t = 0; t < K; t++) {
        u64 y[A];
#pragma unroll
        for (int j = 0; j < A; j++) {
            const u64 v = uP[(((long)t * 2 * P + pp) * A + j) * N + x];
            y[j] = shoup(addmod(v, k.hp[j], k.p[j]), k.pinv[j].w, k.pinv[j].wp, k.p[j]);
            s[j] += (u32)y[j];
            s[A + j] += y[j] >> 32;
        }
        s[2 * A] += (u64)md_overflow<A>(y, k);
    }
#pragma unroll
    for (int i = 0; i < 2 * A + 1; i++) o[i * N] = s[i];
}

// ------------------------------------------------------ conversions of the sums
// A linear map of `words` integers y_w (each below 2^40) onto the rows of Q:
// sum_w y_w W[w][r] mod q_r, plus Kc W[words][r] (0: none).  Used for the Q rows of
// the summed digits (the low and high words of a digit's y; own rows copied)
// and for the summed ModDown.  Of kRelinTerms = 256 terms with A <= 4 sources the
// low words' sums are below 2^40, the high words' below 2^36 (y < 2^60), the
// counts below 2^10: against |W| <= q/2 all of them stay below 2^41.2 q, within
// FqDot's bound although there are up to ten.
struct LinRows {
    int words;
    const ulonglong2 *Wf;   // [words (+1)][nt]: factors of fq_mul
    const ShoupPair *Ws;    // the same as Shoup pairs
    int nt;              // row stride of the tables
    u32 Kc;
};
__device__ __forceinline__ u64 lin_row(const LinRows &L, const u64 *y, int r, u64 q, u64 wone, const ModF &f) {
    if (f.on) {
        FqDot t(0, f);
#pragma unroll
        for (int w = 0; w < 10; w++)
            if (w < L.words) t.narrow(y[w], L.Wf[w * L.nt + r]);
        if (L.Kc) t.narrow(L.Kc, L.Wf[L.words * L.nt + r]);
        return t.get(q, f);
    }
    u64 acc = 0;   // each lazy product below 2 q: reduced every 4 of them (q < 2^60)
#pragma unroll
    for (int w = 0; w < 10; w++)
        if (w < L.words) {
            const ShoupPair s = L.Ws[w * L.nt + r];
            acc += shoup_lazy(y[w], s.w, s.wp, q);
            if ((w & 3) == 3) acc = reduce_any(acc, q, wone);
        }
    if (L.Kc) {
        const ShoupPair s = L.Ws[L.words * L.nt + r];
        acc += shoup_lazy(L.Kc, s.w, s.wp, q);
    }
    return reduce_any(acc, q, wone);
}

// Q rows of the summed digits: dig [P][ndig][nq][N]; own rows from D2 [P][nq][N].
// Table rows of digit d: [d][2 A][nq].
template <int A>
__global__ void __launch_bounds__(256) k_relin_up_fin(u64 *dig, const u64 *SY, const u64 *D2, int P, int level,
                                                      int ndig, int logN, const ulonglong2 *Wf, const ShoupPair *Ws,
                                                      const ModQ *mods, const ModF *modf) {
    pdl_trigger();
    pdl_wait();
    const int nq = level + 1, d = blockIdx.y, i0 = d * A, ns = min(A, nq - i0);
    const long N = 1L << logN, units = (long)P << logN;
    LinRows L = {};
    L.words = 2 * ns, L.nt = nq;
    L.Wf = Wf + (long)d * 2 * A * nq, L.Ws = Ws + (long)d * 2 * A * nq;
    for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < units; idx += (long)gridDim.x * blockDim.x) {
        const int p = (int)(idx >> logN), x = (int)(idx & (N - 1));
        u64 y[10];
#pragma unroll
        for (int s = 0; s < A; s++)
            if (s < ns) {
                y[2 * s] = SY[(((long)p * 2) * nq + i0 + s) * N + x];
                y[2 * s + 1] = SY[(((long)p * 2 + 1) * nq + i0 + s) * N + x];
            }
        u64 *o = dig + ((long)p * ndig + d) * nq * N + x;
        for (int r = 0; r < nq; r++) {
            const bool own = r >= i0 && r < i0 + ns;   // uniform over the CTA
            o[r * N] = own ? D2[((long)p * nq + r) * N + x] : lin_row(L, y, r, mods[r].q, mods[r].wone, modf[r]);
        }
    }
}

// conv [items][nq][N] of the summed ModDown, items = 2 P; K terms.
template <int A>
__global__ void __launch_bounds__(256) k_relin_down_fin(u64 *conv, const u64 *YP, int items, int K, int level, int logN,
                                                        int nt, const ulonglong2 *Wf, const ShoupPair *Ws,
                                                        const ModQ *mods, const ModF *modf) {
    pdl_trigger();
    pdl_wait();
    const int nq = level + 1;
    const long N = 1L << logN, units = (long)items << logN;
    LinRows L = {};
    L.words = 2 * A + 1, L.nt = nt, L.Wf = Wf, L.Ws = Ws, L.Kc = (u32)K;
    for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < units; idx += (long)gridDim.x * blockDim.x) {
        const int it = (int)(idx >> logN), x = (int)(idx & (N - 1));
        u64 y[10];
#pragma unroll
        for (int w = 0; w < 2 * A + 1; w++) y[w] = YP[((long)it * (2 * A + 1) + w) * N + x];
        u64 *o = conv + (long)it * nq * N + x;
        for (int r = 0; r < nq; r++) o[r * N] = lin_row(L, y, r, mods[r].q, mods[r].wone, modf[r]);
    }
}

template <int A>
static void run_a(Ctx *c, RelinSum &S, u64 *d2, int K) {
    const int nq = S.level + 1, nd = c->ndig(S.level), P = S.P;
    const long N = c->N;
    const LevelConsts &lc = c->lc(S.level);
    const bool acc = S.terms > 0;
    // d2 to coefficients, in place
    ntt_inv(c, d2, (long)K * P * nq, c->map_q(S.level), c->stream);
    Buf digP(&c->pool, (size_t)K * P * nd * A * N), uP(&c->pool, (size_t)K * P * 2 * A * N);
    const unsigned gx = (unsigned)std::min<long>((long)P * N / 256, std::max(1L, (long)c->nsm * 8 / nd));
    c->n_launch++;
    cudaEvent_t e0;
    c->trace_begin(3, e0);
    launch_pdl(k_relin_up<A>, dim3(gx, nd), 256, 0, c->stream, d2, S.SY.p, digP.p, K, P, S.level, nd, c->logN, c->L + 1, c->d_mod,
                                                       lc.d_up_inv, lc.d_up_mod, acc);
    c->trace_end(3, e0, 8.0 * N * P * (K * (nq + (double)nd * A) + (acc ? 4.0 : 2.0) * nq));
    ntt_fwd(c, digP.p, (long)K * P * nd * A, c->map_p(), c->stream);
    c->trace_begin(0, e0);
    launch_relin_ms(c, uP.p, digP.p, K * P, nd, c->stream);
    c->trace_end(0, e0, 8.0 * N * A * (2.0 * nd + (double)K * P * (nd + 2)), (double)K * P * nd * A * N * 2.0);
    ntt_inv(c, uP.p, (long)K * P * 2 * A, c->map_p(), c->stream);
    c->n_launch++;
    c->trace_begin(4, e0);
    launch_pdl(k_relin_down<A>, dim3((unsigned)(2L * P * N / 256)), 256, 0, c->stream, uP.p, S.YP.p, K, P, c->logN, c->md_exact, acc);
    c->trace_end(4, e0, 8.0 * N * 2 * P * (K * A + (acc ? 2.0 : 1.0) * (2 * A + 1)));
    S.terms += K;
}

template <int A>
static void finish_a(Ctx *c, RelinSum &S, const u64 *D2, u64 *out) {
    const int nq = S.level + 1, nd = c->ndig(S.level), P = S.P;
    const long N = c->N;
    const LevelConsts &lc = c->lc(S.level);
    Buf dig(&c->pool, (size_t)P * nd * nq * N), u(&c->pool, (size_t)P * 2 * nq * N), conv(&c->pool, (size_t)P * 2 * nq * N);
    const unsigned gx = (unsigned)std::min<long>((long)P * N / 256, std::max(1L, (long)c->nsm * 8 / nd));
    c->n_launch++;
    cudaEvent_t e0;
    c->trace_begin(3, e0);
    launch_pdl(k_relin_up_fin<A>, dim3(gx, nd), 256, 0, c->stream, dig.p, S.SY.p, D2, P, S.level, nd, c->logN, lc.d_su_f,
                                                           lc.d_su_s, c->d_mod, c->d_modf);
    c->trace_end(3, e0, 8.0 * N * P * (3.0 * nq + (double)nd * nq));
    RowSkip sk;
    sk.rows_per_digit = nq, sk.ndig = nd, sk.alpha = A, sk.nq = nq;
    ntt_fwd(c, dig.p, (long)P * nd * nq, c->map_q(S.level), c->stream, &sk);
    launch_multsum_q(c, u.p, dig.p, c->rlk, P, S.level, c->stream);
    c->n_launch++;
    c->trace_begin(4, e0);
    launch_pdl(k_relin_down_fin<A>, dim3((unsigned)std::min<long>(2L * P * N / 256, (long)c->nsm * 8)), 256, 0, c->stream, 
        conv.p, S.YP.p, 2 * P, S.terms, S.level, c->logN, c->L + 1, c->d_sd_f, c->d_sd_s, c->d_mod, c->d_modf);
    c->trace_end(4, e0, 8.0 * N * 2 * P * (2 * A + 1 + nq));
    SubScale ep;
    ep.u = u.p, ep.us = (long)nq * N, ep.out = out, ep.os = (long)nq * N, ep.w = c->d_dn_Pinv, ep.wf = c->d_dn_Pinvf;
    ep.rows_per_item = nq, ep.add = out, ep.as = (long)nq * N;
    ntt_fwd_subscale(c, conv.p, 2L * P * nq, c->map_q(S.level), c->stream, ep);
}

RelinSum::RelinSum(Ctx *c, int P_, int level_)
    : P(P_), level(level_), SY(&c->pool, (size_t)P_ * 2 * (level_ + 1) * c->N),
      YP(&c->pool, (size_t)P_ * 2 * (2 * c->alpha + 1) * c->N) {}

// Terms d2 [K][P][level + 1][N] (NTT domain; overwritten).
void relin_sum_run(Ctx *c, RelinSum &S, u64 *d2, int K) {
    if (S.terms + K > kRelinTerms) throw HeError(HE_ERR_ARG, "too many terms in a summed relinearisation");
    switch (c->alpha) {
    case 1: run_a<1>(c, S, d2, K); break;
    case 2: run_a<2>(c, S, d2, K); break;
    case 3: run_a<3>(c, S, d2, K); break;
    default: run_a<4>(c, S, d2, K); break;
    }
    c->n_dp += (long long)K * S.P;
    c->n_ms += (long long)K * S.P;
    c->n_md += (long long)K * S.P;
}

// out [P][2][level + 1][N] += the summed key switch; D2: sum of the terms' d2.
void relin_sum_finish(Ctx *c, RelinSum &S, const u64 *D2, u64 *out) {
    switch (c->alpha) {
    case 1: finish_a<1>(c, S, D2, out); break;
    case 2: finish_a<2>(c, S, D2, out); break;
    case 3: finish_a<3>(c, S, D2, out); break;
    default: finish_a<4>(c, S, D2, out); break;
    }
}

}  // namespace he

// kernels.cu -- element-wise, sampling, encoding and key-switching kernels.
//
// Layouts: a polynomial is [limbs][N] u64 (limb-major, coalesced along N);
// a ciphertext is [2][level+1][N]; an extended polynomial over Q_l P has
// rows q_0..q_l then p_0..p_{alpha-1}; a batch of B items is contiguous.
#include <cmath>

#include <cstdio>
#include <set>
#include <stdexcept>

#include "bulkcopy.cuh"
#include "he_internal.h"
#include "kernels.cuh"

namespace he {

static inline unsigned nblk(long n, int t) { return (unsigned)((n + t - 1) / t); }

// --------------------------------------------------------------- Philox
// Philox4x32-10 (Salmon et al., SC'11): ten rounds of two 32x32->64 products
// (multipliers 0xD2511F53, 0xCD9E8D57) with the key bumped by the Weyl
// constants 0x9E3779B9, 0xBB67AE85 between rounds.
__device__ __forceinline__ void philox4x32_10(u32 c[4], u32 k0, u32 k1) {
#pragma unroll
    for (int r = 0; r < 10; r++) {
        if (r) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
        u32 lo0 = 0xD2511F53u * c[0], hi0 = __umulhi(0xD2511F53u, c[0]);
        u32 lo1 = 0xCD9E8D57u * c[2], hi1 = __umulhi(0xCD9E8D57u, c[2]);
        u32 n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
        c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
    }
}

// uniform residue of limb (global prime index) j at coefficient i:
// block (i, j, obj, tag) read as hi64:lo64 = (w3 w2):(w1 w0), reduced mod q.
__global__ void k_sample_uniform(u64 *out, long rows, int N, RowMap rm, const ModQ *mods, u32 obj, u32 tag,
                                 u32 k0, u32 k1) {
    long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= rows * N) return;
    long row = idx / N;
    int i = (int)(idx - row * N);
    int pidx = rm.at(row);
    u32 c[4] = {(u32)i, (u32)pidx, obj, tag};
    philox4x32_10(c, k0, k1);
    u64 lo = (u64)c[0] | ((u64)c[1] << 32);
    u64 hi = (u64)c[2] | ((u64)c[3] << 32);
    out[idx] = mod128(hi, lo, mods[pidx]);
}

struct GaussT {
    u64 T[20];
};

// kind 0: ternary from w0 mod 3 -> {0, 1, -1}; kind 1: discrete Gaussian by
// inversion of the cumulative table T on r = (w1:w0) >> 1, sign = w2 bit 0.
__global__ void k_sample_small(i64 *out, int N, int kind, GaussT gt, u32 obj, u32 tag, u32 k0, u32 k1) {
    pdl_trigger();
    pdl_wait();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    u32 c[4] = {(u32)i, 0u, obj, tag};
    philox4x32_10(c, k0, k1);
    if (kind == 0) {
        u32 r = c[0] % 3u;
        out[i] = r == 0 ? 0 : (r == 1 ? 1 : -1);
    } else {
        u64 r = (((u64)c[1] << 32) | (u64)c[0]) >> 1;
        int k = 0;
        while (k < 19 && r >= gt.T[k]) k++;
        i64 x = k;
        if (x != 0 && (c[2] & 1u)) x = -x;
        out[i] = x;
    }
}

__global__ void k_small_to_rns(const i64 *x, u64 *out, long rows, int N, RowMap rm, const ModQ *mods) {
    pdl_trigger();
    pdl_wait();
    long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= rows * N) return;
    long row = idx / N;
    int i = (int)(idx - row * N);
    out[idx] = from_signed(x[i], mods[rm.at(row)].q);
}

void launch_sample_uniform(Ctx *c, u64 *out, int rows, const RowMap &rm, const int *, uint32_t obj,
                           uint32_t tag, cudaStream_t st) {
    long n = (long)rows * c->N;
    c->n_launch++;
    k_sample_uniform<<<nblk(n, 256), 256, 0, st>>>(out, rows, c->N, rm, c->d_mod, obj, tag, (u32)c->seed,
                                                   (u32)(c->seed >> 32));
}

void launch_sample_small(Ctx *c, i64 *out, int kind, uint32_t obj, uint32_t tag, cudaStream_t st) {
    GaussT gt;
    for (int k = 0; k < 20; k++) gt.T[k] = c->gauss_T[k];
    c->n_launch++;
    launch_pdl(k_sample_small, dim3(nblk(c->N, 256)), 256, 0, st, out, c->N, kind, gt, obj, tag, (u32)c->seed,
                                                   (u32)(c->seed >> 32));
}

void launch_small_to_rns(Ctx *c, const i64 *x, u64 *out, int rows, const RowMap &rm, cudaStream_t st) {
    long n = (long)rows * c->N;
    c->n_launch++;
    launch_pdl(k_small_to_rns, dim3(nblk(n, 256)), 256, 0, st, x, out, rows, c->N, rm, c->d_mod);
}

// ------------------------------------------------------ encode / decode
// Inverse canonical embedding (App. A Encode) evaluated in a fixed order so
// that the integer plaintext is reproducible: slot j goes to position
// t = (5^j mod 2N - 1)/4, bit-reversal, radix-2 DIT passes with roots
// conj(zeta^(4 k S/len)), twist by conj(zeta^i), scale by `scale`/S, round
// half away from zero.  Explicit _rn intrinsics: no contraction into FMA.
__device__ __forceinline__ int brev_bits(int x, int bits) { return (int)(__brev((unsigned)x) >> (32 - bits)); }

__global__ void k_enc_permute(const double *zr, const double *zi, double *xr, double *xi, const int *slot_t,
                              int S, int logS) {
    pdl_trigger();
    pdl_wait();
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= S) return;
    int t = brev_bits(slot_t[j], logS);
    xr[t] = zr[j];
    xi[t] = zi[j];
}

__global__ void k_dft_pass(double *xr, double *xi, const double *zeta, int S, int len, int sign) {
    pdl_trigger();
    pdl_wait();
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    int half = len >> 1;
    if (e >= S / 2) return;
    int s = (e / half) * len, k = e % half;
    int ex = k * (4 * (S / len));
    double wr = zeta[2 * ex], wi = zeta[2 * ex + 1];
    if (sign < 0) wi = -wi;
    double br = xr[s + k + half], bi = xi[s + k + half];
    double tr = __dsub_rn(__dmul_rn(br, wr), __dmul_rn(bi, wi));
    double ti = __dadd_rn(__dmul_rn(br, wi), __dmul_rn(bi, wr));
    double ar = xr[s + k], ai = xi[s + k];
    xr[s + k] = __dadd_rn(ar, tr);
    xi[s + k] = __dadd_rn(ai, ti);
    xr[s + k + half] = __dsub_rn(ar, tr);
    xi[s + k + half] = __dsub_rn(ai, ti);
}

__global__ void k_enc_final(const double *xr, const double *xi, const double *zeta, double f, i64 *m, int S) {
    pdl_trigger();
    pdl_wait();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= S) return;
    double wr = zeta[2 * i], wi = -zeta[2 * i + 1];
    double yr = __dsub_rn(__dmul_rn(xr[i], wr), __dmul_rn(xi[i], wi));
    double yi = __dadd_rn(__dmul_rn(xr[i], wi), __dmul_rn(xi[i], wr));
    m[i] = (i64)round(__dmul_rn(yr, f));
    m[i + S] = (i64)round(__dmul_rn(yi, f));
}

// Decode (App. A): x_i = u_i zeta^i with u_i = (m_i + I m_{i+S}) / scale,
// length-S DFT with exponent +1, slot j = x[t(j)].
__global__ void k_dec_twist(const double *coef, double scale, const double *zeta, double *xr, double *xi, int S,
                            int logS) {
    pdl_trigger();
    pdl_wait();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= S) return;
    double ur = coef[i] / scale, ui = coef[i + S] / scale;
    double wr = zeta[2 * i], wi = zeta[2 * i + 1];
    int t = brev_bits(i, logS);
    xr[t] = ur * wr - ui * wi;
    xi[t] = ur * wi + ui * wr;
}

__global__ void k_dec_gather(const double *xr, const double *xi, const int *slot_t, double *zr, double *zi, int S) {
    pdl_trigger();
    pdl_wait();
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= S) return;
    zr[j] = xr[slot_t[j]];
    zi[j] = xi[slot_t[j]];
}

void launch_encode(Ctx *c, const double *zre, const double *zim, double scale, i64 *m_out, cudaStream_t st) {
    int S = c->S, logS = c->logN - 1;
    Buf tmp(&c->pool, (size_t)S), tmp2(&c->pool, (size_t)S);  // S doubles each
    double *xr = (double *)tmp.p, *xi = (double *)tmp2.p;
    c->n_launch++;
    launch_pdl(k_enc_permute, dim3(nblk(S, 256)), 256, 0, st, zre, zim, xr, xi, c->d_slot_t, S, logS);
    for (int len = 2; len <= S; len <<= 1) {
        c->n_launch++;
        launch_pdl(k_dft_pass, dim3(nblk(S / 2, 256)), 256, 0, st, xr, xi, c->d_zeta, S, len, -1);
    }
    double f = scale / (double)S;
    c->n_launch++;
    launch_pdl(k_enc_final, dim3(nblk(S, 256)), 256, 0, st, xr, xi, c->d_zeta, f, m_out, S);
}

void launch_decode(Ctx *c, const double *coef, double scale, double *zre, double *zim, cudaStream_t st) {
    int S = c->S, logS = c->logN - 1;
    Buf tmp(&c->pool, (size_t)S);
    Buf tmp2(&c->pool, (size_t)S);
    double *xr = (double *)tmp.p, *xi = (double *)tmp2.p;
    c->n_launch++;
    launch_pdl(k_dec_twist, dim3(nblk(S, 256)), 256, 0, st, coef, scale, c->d_zeta, xr, xi, S, logS);
    for (int len = 2; len <= S; len <<= 1) {
        c->n_launch++;
        launch_pdl(k_dft_pass, dim3(nblk(S / 2, 256)), 256, 0, st, xr, xi, c->d_zeta, S, len, +1);
    }
    c->n_launch++;
    launch_pdl(k_dec_gather, dim3(nblk(S, 256)), 256, 0, st, xr, xi, c->d_slot_t, zre, zim, S);
}

// ----------------------------------------------------------- elementwise
#define EW_PROLOGUE                                                   \
    long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;           \
    if (idx >= rows * (long)N) return;                                \
    long row = idx / N;                                               \
    const ModQ &m = mods[rm.at(row)];                           \
    (void)m;

__global__ void k_add(u64 *o, const u64 *a, const u64 *b, long rows, int N, RowMap rm, const ModQ *mods) {
    pdl_trigger();
    pdl_wait();
    EW_PROLOGUE
    o[idx] = addmod(a[idx], b[idx], m.q);
}
__global__ void k_sub(u64 *o, const u64 *a, const u64 *b, long rows, int N, RowMap rm, const ModQ *mods) {
    pdl_trigger();
    pdl_wait();
    EW_PROLOGUE
    o[idx] = submod(a[idx], b[idx], m.q);
}
__global__ void k_neg(u64 *o, const u64 *a, long rows, int N, RowMap rm, const ModQ *mods) {
    pdl_trigger();
    pdl_wait();
    EW_PROLOGUE
    u64 v = a[idx];
    o[idx] = v ? m.q - v : 0;
}
__global__ void k_mul(u64 *o, const u64 *a, const u64 *b, long rows, int N, RowMap rm, const ModQ *mods) {
    pdl_trigger();
    pdl_wait();
    EW_PROLOGUE
    o[idx] = mulmod(a[idx], b[idx], m);
}
__global__ void k_mulM(u64 *o, const u64 *a, const u64 *bM, long rows, int N, RowMap rm, const ModQ *mods) {
    pdl_trigger();
    pdl_wait();
    EW_PROLOGUE
    o[idx] = mulmont(a[idx], bM[idx], m);
}
__global__ void k_to_mont(u64 *o, const u64 *a, long rows, int N, RowMap rm, const ModQ *mods) {
    pdl_trigger();
    pdl_wait();
    EW_PROLOGUE
    o[idx] = mulmont(a[idx], m.r2, m);  // a R^2 R^-1 = a R
}
__global__ void k_from_mont(u64 *o, const u64 *a, long rows, int N, RowMap rm, const ModQ *mods) {
    pdl_trigger();
    pdl_wait();
    EW_PROLOGUE
    o[idx] = redc(a[idx], 0, m);
}

#define EW_LAUNCH(kern, ...)                                                         \
    do {                                                                             \
        long n__ = rows * (long)c->N;                                                \
        if (n__ > 0) c->n_launch++, launch_pdl(kern, dim3(nblk(n__, 256)), 256, 0, st, __VA_ARGS__, rows, c->N, rm, c->d_mod); \
    } while (0)

void launch_add(Ctx *c, u64 *out, const u64 *a, const u64 *b, long rows, const RowMap &rm, cudaStream_t st) {
    EW_LAUNCH(k_add, out, a, b);
}
void launch_sub(Ctx *c, u64 *out, const u64 *a, const u64 *b, long rows, const RowMap &rm, cudaStream_t st) {
    EW_LAUNCH(k_sub, out, a, b);
}
void launch_neg(Ctx *c, u64 *out, const u64 *a, long rows, const RowMap &rm, cudaStream_t st) {
    EW_LAUNCH(k_neg, out, a);
}
void launch_mul(Ctx *c, u64 *out, const u64 *a, const u64 *b, long rows, const RowMap &rm, cudaStream_t st) {
    EW_LAUNCH(k_mul, out, a, b);
}
void launch_mulM(Ctx *c, u64 *out, const u64 *a, const u64 *bM, long rows, const RowMap &rm, cudaStream_t st) {
    EW_LAUNCH(k_mulM, out, a, bM);
}
void launch_to_mont(Ctx *c, u64 *out, const u64 *a, long rows, const RowMap &rm, cudaStream_t st) {
    EW_LAUNCH(k_to_mont, out, a);
}
void launch_from_mont(Ctx *c, u64 *out, const u64 *a, long rows, const RowMap &rm, cudaStream_t st) {
    EW_LAUNCH(k_from_mont, out, a);
}

// out[row] = a[row] * w[row % rows_per_item] (Shoup constant per row)
__global__ void k_mulconst_rows(u64 *o, const u64 *a, const ShoupPair *w, int rpi, long rows, int N, RowMap rm,
                                const ModQ *mods) {
    EW_PROLOGUE
    ShoupPair s = w[row % rpi];
    o[idx] = shoup(a[idx], s.w, s.wp, m.q);
}
void launch_mulconst_rows(Ctx *c, u64 *out, const u64 *a, const ShoupPair *w, long rows, int rpi,
                          const RowMap &rm, cudaStream_t st) {
    long n = rows * (long)c->N;
    if (n > 0)
        c->n_launch++;
        k_mulconst_rows<<<nblk(n, 256), 256, 0, st>>>(out, a, w, rpi, rows, c->N, rm, c->d_mod);
}

// NTT-domain index of the automorphism X -> X^g: output slot x (evaluation
// point psi^(2 brv(x)+1)) reads input slot brv(((2 brv(x)+1) g mod 2N - 1)/2).
__device__ __forceinline__ int auto_index(int x, u32 g, int logN) {
    int N = 1 << logN;
    u32 e = 2u * (u32)brev_bits(x, logN) + 1u;
    u32 e2 = (u32)(((u64)e * g) & (u64)(2 * N - 1));
    return brev_bits((int)((e2 - 1) >> 1), logN);
}

__global__ void k_automorph(u64 *o, const u64 *in, long rows, int logN, u32 g) {
    int N = 1 << logN;
    long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= rows * (long)N) return;
    long row = idx / N;
    int x = (int)(idx - row * N);
    o[idx] = in[row * N + auto_index(x, g, logN)];
}
void launch_automorph(Ctx *c, u64 *out, const u64 *in, long rows, const RowMap &, uint32_t g, cudaStream_t st) {
    long n = rows * (long)c->N;
    c->n_launch++;
    if (n > 0) k_automorph<<<nblk(n, 256), 256, 0, st>>>(out, in, rows, c->logN, g);
}

// tensor product in the NTT domain: d0 = a0 b0, d1 = a0 b1 + a1 b0, d2 = a1 b1.
// a, b, d01: [B][2][limbs][N] (d01: d0, d1 of each item); d2: [B][limbs][N].
__global__ void k_tensor(u64 *d01, u64 *d2, const u64 *a, const u64 *b, int B, int limbs, int N, RowMap rm,
                         const ModQ *mods) {
    pdl_trigger();
    pdl_wait();
    long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    long per = (long)limbs * N;
    if (idx >= (long)B * per) return;
    int it = (int)(idx / per);
    long off = idx - (long)it * per;
    int limb = (int)(off / N);
    const ModQ &m = mods[rm.at(limb)];
    const u64 *pa = a + it * 2 * per, *pb = b + it * 2 * per;
    u64 a0 = pa[off], a1 = pa[per + off], b0 = pb[off], b1 = pb[per + off];
    U128 acc = {0, 0};
    mac128(acc, a0, b1);
    mac128(acc, a1, b0);
    u64 t1 = redc(acc.lo, acc.hi, m);
    u64 v0 = mulmod(a0, b0, m), v1 = redc(t1 * m.r2, mulhi64(t1, m.r2), m), v2 = mulmod(a1, b1, m);
    u64 *o = d01 + (long)it * 2 * per + off;
    o[0] = v0;
    o[per] = v1;
    d2[(long)it * per + off] = v2;
}
void launch_tensor(Ctx *c, u64 *d01, u64 *d2, const u64 *a, const u64 *b, int B, int limbs, const RowMap &rm,
                   cudaStream_t st) {
    long n = (long)B * limbs * c->N;
    c->n_launch++;
    launch_pdl(k_tensor, dim3(nblk(n, 256)), 256, 0, st, d01, d2, a, b, B, limbs, c->N, rm, c->d_mod);
}

// ------------------------------------------------------------- ModUp
// Decompose (Sec. 3.3): per digit d, y_i = [c_i (Q_d/q_i)^-1]_{q_i}; every
// target row r of Q_l P gets sum_i y_i (Q_d/q_i mod r) mod r, except the
// digit's own rows, which keep c_r.  In/out in coefficient form.
// coef: [B][l+1][N]; out: [B][ndig][l+1+alpha][N].
//
// blockIdx.y is the digit: a CTA stages that digit's conversion constants
// and row primes in shared memory once and walks (item, coefficient pair)
// with a grid stride.  Each thread converts two adjacent coefficients with
// 16-byte loads and stores.  Rows of 40-bit primes sum their products with one
// float quotient (FqDot); the others sum A lazy Shoup products (each in
// [0, 2r)) and reduce once.  Bound by the integer multiplies (FMA-heavy pipe).
static int sm_count(int dev) {
    static int n[64];
    dev &= 63;
    if (!n[dev]) cudaDeviceGetAttribute(&n[dev], cudaDevAttrMultiProcessorCount, dev);
    return n[dev] > 0 ? n[dev] : 1;
}

// C adjacent words, one 16-byte access for C = 2
template <int C>
struct Words {
    u64 w[C];
};
template <int C>
__device__ __forceinline__ Words<C> load_words(const u64 *p) {
    Words<C> r;
    if constexpr (C == 2) {
        const ulonglong2 v = *(const ulonglong2 *)p;
        r.w[0] = v.x, r.w[1] = v.y;
    } else {
        r.w[0] = *p;
    }
    return r;
}
template <int C>
__device__ __forceinline__ void store_words(u64 *p, const Words<C> &r) {
    if constexpr (C == 2) *(ulonglong2 *)p = make_ulonglong2(r.w[0], r.w[1]);
    else *p = r.w[0];
}

// A: special primes per digit; C: adjacent coefficients per thread (2 on
// launches that fill the GPU, 1 on small ones, where more threads hide more
// latency).  up_fq null: every row takes the Shoup products.
template <int A, int C>
__global__ void __launch_bounds__(256) k_modup_bconv(const u64 *coef, u64 *out, int B, int level, int ndig, int N,
                                                     RowMap qp, const ModQ *mods, const ModF *modf,
                                                     const ShoupPair *up_inv, const ShoupPair *up_mod,
                                                     const FqPair *up_fq, const u64 *own_ntt, long own_s) {
    pdl_trigger();
    if (!up_fq) pdl_wait();   // constants that the caller uploaded in the stream
    __shared__ ShoupPair s_mod[A * 64];   // [s][r], rows <= 64
    __shared__ FqPair s_fq[A * 64];
    __shared__ ModF s_f[64];
    __shared__ u64 s_q[64], s_w1[64];
    const int d = blockIdx.y;
    const int rows = level + 1 + A;
    const int i0 = d * A;
    const int ns = min(A, level + 1 - i0);
    for (int r = threadIdx.x; r < rows; r += blockDim.x) {
        const int p = r <= qp.lq ? r : qp.base_p + (r - qp.lq - 1);   // qp is unshifted
        s_q[r] = mods[p].q, s_w1[r] = mods[p].wone, s_f[r] = modf[p];
        if (!up_fq) s_f[r].on = 0;
    }
    for (int e = threadIdx.x; e < ns * rows; e += blockDim.x) {
        const int sd = e / rows, r = e - sd * rows;
        s_mod[e] = up_mod[((long)d * A + sd) * rows + r];
        if (up_fq) s_fq[e] = up_fq[((long)d * A + sd) * rows + r];
    }
    ShoupPair inv[A];
    u64 qs[A];
    bool narrow[A];   // uniform over the CTA
#pragma unroll
    for (int sd = 0; sd < A; sd++)
        if (sd < ns) inv[sd] = up_inv[d * A + sd], qs[sd] = mods[i0 + sd].q, narrow[sd] = qs[sd] < kNarrow;
    __syncthreads();
    pdl_wait();
    const int per = N / C;
    const long units = (long)B * per;
    for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < units; idx += (long)gridDim.x * blockDim.x) {
        const int b = (int)(idx / per);
        const int x = C * (int)(idx - (long)b * per);
        const u64 *cb = coef + (long)b * (level + 1) * N + x;
        u64 *ob = out + ((long)b * ndig + d) * rows * N + x;
        u64 y[C][A];
#pragma unroll
        for (int sd = 0; sd < A; sd++) {
#pragma unroll
            for (int c = 0; c < C; c++) y[c][sd] = 0;
            if (sd < ns) {
                const Words<C> v = load_words<C>(cb + (long)(i0 + sd) * N);
#pragma unroll
                for (int c = 0; c < C; c++) y[c][sd] = shoup(v.w[c], inv[sd].w, inv[sd].wp, qs[sd]);
            }
        }
        for (int r = 0; r < rows; r++) {
            Words<C> o;
            if (r >= i0 && r < i0 + ns) {   // uniform over the CTA
                o = load_words<C>(own_ntt ? own_ntt + (long)b * own_s + (long)r * N + x : cb + (long)r * N);
            } else if (s_f[r].on) {   // uniform over the CTA
                const ModF m = s_f[r];
                FqDot t[C];
#pragma unroll
                for (int c = 0; c < C; c++) t[c] = FqDot(0, m);
#pragma unroll
                for (int sd = 0; sd < A; sd++) {
                    if (sd < ns) {
                        const FqPair w = s_fq[sd * rows + r];
#pragma unroll
                        for (int c = 0; c < C; c++) {
                            if (narrow[sd]) t[c].narrow(y[c][sd], w.lo);
                            else t[c].wide(y[c][sd], w);
                        }
                    }
                }
#pragma unroll
                for (int c = 0; c < C; c++) o.w[c] = t[c].get(s_q[r], m);
            } else {
                const u64 q = s_q[r];
                u64 acc[C];
#pragma unroll
                for (int c = 0; c < C; c++) acc[c] = 0;
#pragma unroll
                for (int sd = 0; sd < A; sd++) {
                    if (sd < ns) {
                        const ShoupPair w = s_mod[sd * rows + r];
#pragma unroll
                        for (int c = 0; c < C; c++) acc[c] += shoup_lazy(y[c][sd], w.w, w.wp, q);
                    }
                }
                // < 2 A q <= 8q < 2^64
#pragma unroll
                for (int c = 0; c < C; c++) o.w[c] = reduce_any(acc[c], q, s_w1[r]);
            }
            store_words<C>(ob + (long)r * N, o);
        }
    }
}

template <int A>
static void modup_launch_a(Ctx *c, const u64 *coef, u64 *out, int B, int level, int nd, const ShoupPair *up_inv,
                           const ShoupPair *up_mod, const FqPair *up_fq, const u64 *own_ntt, long own_s,
                           cudaStream_t st) {
    const int nsm = sm_count(c->device);
    // two coefficients per thread once the launch fills the GPU with 8 CTAs
    // of 256 threads per SM, one below that
    const bool wide = (long)B * (c->N / 2) * nd >= (long)nsm * 8 * 256;
    const long units = (long)B * (c->N / (wide ? 2 : 1));
    long gx = std::max(1L, (long)nsm * 8 / nd);
    gx = std::min(gx, (long)nblk(units, 256));
    const dim3 grid((unsigned)gx, (unsigned)nd);
    const RowMap qp = c->map_qp(level);
    if (wide)
        launch_pdl(k_modup_bconv<A, 2>, dim3(grid), 256, 0, st, coef, out, B, level, nd, c->N, qp, c->d_mod, c->d_modf, up_inv, up_mod, up_fq, own_ntt, own_s);
    else
        launch_pdl(k_modup_bconv<A, 1>, dim3(grid), 256, 0, st, coef, out, B, level, nd, c->N, qp, c->d_mod, c->d_modf, up_inv, up_mod, up_fq, own_ntt, own_s);
}

static void modup_launch(Ctx *c, const u64 *coef, u64 *out, int B, int level, int nd, const ShoupPair *up_inv,
                         const ShoupPair *up_mod, const FqPair *up_fq, const u64 *own_ntt, long own_s,
                         cudaStream_t st) {
    switch (c->alpha) {
    case 1: modup_launch_a<1>(c, coef, out, B, level, nd, up_inv, up_mod, up_fq, own_ntt, own_s, st); break;
    case 2: modup_launch_a<2>(c, coef, out, B, level, nd, up_inv, up_mod, up_fq, own_ntt, own_s, st); break;
    case 3: modup_launch_a<3>(c, coef, out, B, level, nd, up_inv, up_mod, up_fq, own_ntt, own_s, st); break;
    default: modup_launch_a<4>(c, coef, out, B, level, nd, up_inv, up_mod, up_fq, own_ntt, own_s, st); break;
    }
}

void launch_modup_bconv(Ctx *c, const u64 *coef, u64 *out, int B, int level, cudaStream_t st, const u64 *own_ntt,
                        long own_s) {
    const LevelConsts &L = c->lc(level);
    c->n_launch++;
    cudaEvent_t e0;
    c->trace_begin(3, e0);
    modup_launch(c, coef, out, B, level, L.ndig, L.d_up_inv, L.d_up_mod, L.d_up_fq, own_ntt, own_s, st);
    // the input limbs once, every digit's extended limbs once
    c->trace_end(3, e0, 8.0 * B * c->N * ((level + 1) + (double)L.ndig * c->qp_rows(level)));
}

// Same conversion with caller-supplied constants (layout of LevelConsts).
void launch_modup_bconv_with(Ctx *c, const u64 *coef, u64 *out, int B, int level, const ShoupPair *up_inv,
                             const ShoupPair *up_mod, cudaStream_t st) {
    c->n_launch++;
    modup_launch(c, coef, out, B, level, c->ndig(level), up_inv, up_mod, nullptr, nullptr, 0, st);
}

// ----------------------------------------------------- constants per limb
// Multiplying by a constant polynomial m (or adding it) acts on every
// NTT-domain slot of limb i with the scalar m mod q_i.
struct ScalarList {
    ShoupPair w[64];
};
__global__ void k_scalar_mul_rows(u64 *o, const u64 *a, long rows, int rpi, int N, ScalarList s, RowMap rm,
                                  const ModQ *mods) {
    pdl_trigger();
    pdl_wait();
    long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= rows * (long)N) return;
    long row = idx / N;
    int r = (int)(row % rpi);
    o[idx] = shoup(a[idx], s.w[r].w, s.w[r].wp, mods[rm.at(row)].q);
}
void launch_scalar_mul_rows(Ctx *c, u64 *out, const u64 *a, long rows, int rpi, const ShoupPair *vals,
                            const RowMap &rm, cudaStream_t st) {
    ScalarList s;
    for (int i = 0; i < rpi && i < 64; i++) s.w[i] = vals[i];
    long n = rows * (long)c->N;
    c->n_launch++;
    launch_pdl(k_scalar_mul_rows, dim3(nblk(n, 256)), 256, 0, st, out, a, rows, rpi, c->N, s, rm, c->d_mod);
}
__global__ void k_scalar_add_rows(u64 *o, long rows, int N, ScalarList s, RowMap rm, const ModQ *mods) {
    pdl_trigger();
    pdl_wait();
    long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= rows * (long)N) return;
    long row = idx / N;
    u64 q = mods[rm.at(row)].q;
    o[idx] = addmod(o[idx], s.w[row].w, q);
}
void launch_scalar_add_rows(Ctx *c, u64 *data, long rows, const u64 *vals, const RowMap &rm, cudaStream_t st) {
    ScalarList s;
    for (int i = 0; i < rows && i < 64; i++) s.w[i].w = vals[i];
    long n = rows * (long)c->N;
    c->n_launch++;
    launch_pdl(k_scalar_add_rows, dim3(nblk(n, 256)), 256, 0, st, data, rows, c->N, s, rm, c->d_mod);
}
// centred lift of a residue mod q_0 to a signed integer
__global__ void k_centre_i64_q0(const u64 *a, i64 *out, int N, const ModQ *mods) {
    pdl_trigger();
    pdl_wait();
    int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= N) return;
    u64 q = mods[0].q, v = a[x];
    out[x] = v > (q >> 1) ? -(i64)(q - v) : (i64)v;
}
void launch_centre_i64_q0(Ctx *c, const u64 *a, i64 *out, cudaStream_t st) {
    c->n_launch++;
    launch_pdl(k_centre_i64_q0, dim3(nblk(c->N, 256)), 256, 0, st, a, out, c->N, c->d_mod);
}

// ------------------------------------------------------------- ModDown
// Rounding ModDown (App. A KeySwitch: round(P^-1 x)) as floor((x + h) / P),
// h = (P-1)/2.  With v_j = u_{p_j} + h mod p_j and y_j = [v_j (P/p_j)^-1]_{p_j},
// the exact residue (x + h) mod P is S - e P with S = sum_j y_j (P/p_j) and
// the overflow count e = floor(S / P) < A, taken exactly: S is summed in
// 64-bit limbs and compared with P, 2P, ...
// conv_r = ((x + h) mod P) - h mod q_r, coefficient form (h is added to
// every coefficient, so it is folded in here, before the forward NTT):
// conv_r = sum_j y_j (P/p_j mod q_r) + E_{e,r} with E_{e,r} = -(e P + h) mod q_r.
// pcoef: [items][A][N]; out: [items][l+1][N].

// C adjacent coefficients per thread (2: 16-byte loads and stores, on
// launches that fill the GPU; 1 on small ones), a grid stride over (item,
// coefficient group); per row the products are summed with one float quotient
// (40-bit rows) or as lazy Shoup products reduced once.
//
// RS: the ModDown of a ciphertext that is rescaled by q_l next.  With
// conv_r = ((x + h) mod P) - h as above, ModDown is d_r = (u_r - conv_r) P^-1, and
// the rescale takes t = d_l centred (coefficient form, from row l of u):
// (d_i - t) q_l^-1 = (u_i - (conv_i + t P)) (P q_l)^-1, so one forward NTT of
// z_i = conv_i + t P does for both: out [items][l][N] holds z.  pcoef:
// [items][1 + A][N], row q_l first.  E: [neg][e][r], -q_l P folded in where the
// centred t is negative.
template <int A, int C, bool RS>
__global__ void __launch_bounds__(256) k_moddown_bconv(const u64 *pcoef, u64 *out, int items, int level, int N,
                                                       const __grid_constant__ MdExact k, const ModQ *mods,
                                                       const ModF *modf, const ShoupPair *pmod, const FqPair *pfq,
                                                       const ShoupPair *Pmod, const ShoupPair *Pinv, const u64 *E,
                                                       int Es, const u64 *El, int L) {
    pdl_trigger();
    constexpr int S = RS ? A + 1 : A;   // sources: y_j, then t
    __shared__ ShoupPair s_c[S * 64];
    __shared__ FqPair s_fq[S * 64];
    __shared__ ModF s_f[64];
    __shared__ u64 s_E[(RS ? 2 : 1) * A * 64], s_El[A], s_q[64], s_w1[64];
    const int nr = RS ? level : level + 1, nt = level + 1;   // rows written; rows with constants
    for (int r = threadIdx.x; r < nt; r += blockDim.x) s_q[r] = mods[r].q, s_w1[r] = mods[r].wone, s_f[r] = modf[r];
    for (int e = threadIdx.x; e < S * nt; e += blockDim.x) {
        const int j = e / nt, r = e - j * nt;
        s_c[e] = j < A ? pmod[j * (L + 1) + r] : Pmod[r];
        s_fq[e] = pfq[j * (L + 1) + r];
    }
    for (int e = threadIdx.x; e < (RS ? 2 : 1) * A * nr; e += blockDim.x) {
        const int j = e / nr, r = e - j * nr;
        s_E[e] = E[j * Es + r];
    }
    if (RS && threadIdx.x < A) s_El[threadIdx.x] = El[threadIdx.x * (L + 1) + level];
    const ShoupPair pil = RS ? Pinv[level] : ShoupPair{0, 0};
    __syncthreads();
    pdl_wait();
    const int per = N / C;
    const long units = (long)items * per;
    // sum_j y_j w_jr + e for the first n sources
    auto dot = [&](const u64 *y, int n, int r, u64 e) -> u64 {
        if (s_f[r].on) {   // uniform over the CTA
            const ModF m = s_f[r];
            FqDot t(e, m);
#pragma unroll
            for (int j = 0; j < S; j++)
                if (j < n) t.wide(y[j], s_fq[j * nt + r]);
            return t.get(s_q[r], m);
        }
        const u64 q = s_q[r];
        u64 acc = e;   // < (2 S + 1) q <= 11 q < 2^64
#pragma unroll
        for (int j = 0; j < S; j++)
            if (j < n) acc += shoup_lazy(y[j], s_c[j * nt + r].w, s_c[j * nt + r].wp, q);
        return reduce_any(acc, q, s_w1[r]);
    };
    for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < units; idx += (long)gridDim.x * blockDim.x) {
        const int it = (int)(idx / per);
        const int x = C * (int)(idx - (long)it * per);
        const u64 *pi = pcoef + (long)it * S * N + x;
        u64 y[C][S];
#pragma unroll
        for (int j = 0; j < A; j++) {
            const Words<C> v = load_words<C>(pi + (long)(RS ? j + 1 : j) * N);
            const u64 p = k.p[j];
#pragma unroll
            for (int c = 0; c < C; c++) y[c][j] = shoup(addmod(v.w[c], k.hp[j], p), k.pinv[j].w, k.pinv[j].wp, p);
        }
        int e[C];
#pragma unroll
        for (int c = 0; c < C; c++) {
            u64 ya[A];
#pragma unroll
            for (int j = 0; j < A; j++) ya[j] = y[c][j];
            e[c] = md_overflow<A>(ya, k);
        }
        if constexpr (RS) {
            const Words<C> v = load_words<C>(pi);
            const u64 ql = s_q[level];
#pragma unroll
            for (int c = 0; c < C; c++) {
                const u64 cl = dot(y[c], A, level, s_El[e[c]]);
                const u64 t = shoup(submod(v.w[c], cl, ql), pil.w, pil.wp, ql);
                y[c][A] = t;
                if (t > (ql >> 1)) e[c] += A;
            }
        }
        u64 *op = out + (long)it * nr * N + x;
        for (int r = 0; r < nr; r++) {
            Words<C> o;
#pragma unroll
            for (int c = 0; c < C; c++) o.w[c] = dot(y[c], S, r, s_E[e[c] * nr + r]);
            store_words<C>(op + (long)r * N, o);
        }
    }
}

template <int A, bool RS>
static void moddown_launch_a(Ctx *c, const u64 *pcoef, u64 *out, int items, int level, cudaStream_t st) {
    const int nsm = sm_count(c->device);
    const bool wide = (long)items * (c->N / 2) >= (long)nsm * 8 * 256;
    const long units = (long)items * (c->N / (wide ? 2 : 1));
    const unsigned grid = (unsigned)std::min<long>((long)nsm * 8, nblk(units, 256));
    const MdExact &k = c->md_exact;
    const u64 *E = RS ? c->lc(level).d_mr_E : c->d_dn_E;
    const int Es = RS ? level : c->L + 1;
    if (wide)
        launch_pdl(k_moddown_bconv<A, 2, RS>, dim3(grid), 256, 0, st, pcoef, out, items, level, c->N, k, c->d_mod, c->d_modf, c->d_dn_pmod, c->d_dn_fq, c->d_Pmod, c->d_dn_Pinv, E, Es, c->d_dn_E, c->L);
    else
        launch_pdl(k_moddown_bconv<A, 1, RS>, dim3(grid), 256, 0, st, pcoef, out, items, level, c->N, k, c->d_mod, c->d_modf, c->d_dn_pmod, c->d_dn_fq, c->d_Pmod, c->d_dn_Pinv, E, Es, c->d_dn_E, c->L);
}

template <bool RS>
static void moddown_launch(Ctx *c, const u64 *pcoef, u64 *out, int items, int level, cudaStream_t st) {
    c->n_launch++;
    cudaEvent_t e0;
    c->trace_begin(4, e0);
    switch (c->alpha) {
    case 1: moddown_launch_a<1, RS>(c, pcoef, out, items, level, st); break;
    case 2: moddown_launch_a<2, RS>(c, pcoef, out, items, level, st); break;
    case 3: moddown_launch_a<3, RS>(c, pcoef, out, items, level, st); break;
    default: moddown_launch_a<4, RS>(c, pcoef, out, items, level, st); break;
    }
    c->trace_end(4, e0, 8.0 * items * c->N * (c->alpha + level + 1));
}

void launch_moddown_bconv(Ctx *c, const u64 *pcoef, u64 *out, int items, int level, cudaStream_t st) {
    moddown_launch<false>(c, pcoef, out, items, level, st);
}

void launch_moddown_rescale_bconv(Ctx *c, const u64 *pcoef, u64 *out, int items, int level, cudaStream_t st) {
    moddown_launch<true>(c, pcoef, out, items, level, st);
}

// out_r = (u_r - conv_r) P^-1 mod q_r (+ addend_r), NTT domain, r <= level.
__global__ void k_moddown_final(u64 *out, const u64 *u, const u64 *conv, const u64 *add, int items, int level,
                                int N, long us, long os, long as, const ModQ *mods, const ShoupPair *Pinv) {
    pdl_trigger();
    pdl_wait();
    long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    long per = (long)(level + 1) * N;
    if (idx >= (long)items * per) return;
    int it = (int)(idx / per);
    long off = idx - (long)it * per;
    int r = (int)(off / N);
    u64 q = mods[r].q;
    ShoupPair w = Pinv[r];
    u64 v = shoup(submod(u[it * us + off], conv[idx], q), w.w, w.wp, q);
    if (add) v = addmod(v, add[it * as + off], q);
    out[it * os + off] = v;
}
void launch_moddown_final(Ctx *c, u64 *out, const u64 *u, const u64 *conv, const u64 *addend, int items, int level,
                          long us, long os, long as, cudaStream_t st) {
    long n = (long)items * (level + 1) * c->N;
    c->n_launch++;
    launch_pdl(k_moddown_final, dim3(nblk(n, 256)), 256, 0, st, out, u, conv, addend, items, level, c->N, us, os, as, c->d_mod,
                                                  c->d_dn_Pinv);
}

// Permutes key rows into the layout of msum.cu: out[row][pi_g(x)] = in[row][x].
__global__ void k_permute_key(u64 *out, const u64 *in, long rows, int logN, u32 g) {
    const int N = 1 << logN;
    long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= rows * (long)N) return;
    long row = idx / N;
    int x = (int)(idx - row * N);
    out[row * N + auto_index(x, g, logN)] = in[idx];
}
void launch_permute_key(Ctx *c, u64 *out, const u64 *in, long rows, uint32_t g, cudaStream_t st) {
    long n = rows * (long)c->N;
    c->n_launch++;
    k_permute_key<<<nblk(n, 256), 256, 0, st>>>(out, in, rows, c->logN, g);
}

// ------------------------------------------------------ double hoisting
// S[b][k][r][x] = sum_t ptM_t[r][x] * R_t[b][k][r][x] over Q_l P (one REDC).
// One launch for several sums over the same R: term t of sum y is plaintext
// pt[t] times R[ri[t]], first[y] <= t < first[y + 1].  The sums are the fastest
// grid index: the CTAs of one block of coefficients run together and find its R
// words in L2 (with the coefficients fastest the 15 giants of a sigma read R
// from DRAM 15 times, twice the plaintexts' bytes: 480 us against the 170 of
// one pass over both at the copy rate).  Two adjacent words per thread; a
// thread's words of the next three terms are on their way to a ring of its own
// in shared memory while a term is multiplied (with only the next term's in
// flight it waited for memory: the 15 giants of a sigma, 16 terms each, took 385
// us at 2.9 TB/s, both launches of the transform 430 us, now 251: N = 2^15, level
// 11, one ciphertext).  One REDC per output word: up to 32 products below q^2 stay below q 2^64 for q < 2^59; on wider
// rows (q_0, the special primes) the sum is kept below it term by term
// (mac128_q).
struct PmulArgs {
    const u64 *pt[kMaxPmulTerms];
    const u64 *R[kMaxPmulRots];
    unsigned char ri[kMaxPmulTerms];
    short first[kMaxPmulSums + 1];
};
constexpr int kPmulThreads = 128, kPmulStages = 4;
// FQ: plaintexts plain and centred, sums as in MultSum; else in Montgomery form.
template <bool FQ, bool WIDE>
__device__ __forceinline__ void pmul_item(const PmulArgs &pa, int t0, int t1, long idx, long per, long ro, u64 *ob,
                                          const ModQ &m, const ModF &f, ulonglong2 (*ring)[3][kPmulThreads]) {
    const int tx = threadIdx.x;
    auto issue = [&](int t) {
        if (t < t1) {
            ulonglong2 (*s)[kPmulThreads] = ring[(t - t0) % kPmulStages];
            const u64 *rb = pa.R[pa.ri[t]] + ro + idx;
            bc_copy16(bc_smem(&s[0][tx]), pa.pt[t] + idx);
            bc_copy16(bc_smem(&s[1][tx]), rb);
            bc_copy16(bc_smem(&s[2][tx]), rb + per);
        }
        bc_commit();
    };
    u64 o[2][2];
    ulonglong2 pv, v0, v1;
    auto next = [&](int t) {   // the term's words; its slot is the next one's
        bc_wait_groups<kPmulStages - 2>();
        const ulonglong2 (*s)[kPmulThreads] = ring[(t - t0) % kPmulStages];
        pv = s[0][tx], v0 = s[1][tx], v1 = s[2][tx];
        issue(t + kPmulStages - 1);
    };
#pragma unroll
    for (int i = 0; i < kPmulStages - 1; i++) issue(t0 + i);
    if constexpr (FQ) {
        const FqMacC c(f, m.q);
        FqMac a[2][2] = {};
        for (int t = t0, run = 0; t < t1; t++, run++) {
            next(t);
            if (run == c.lim) {
                run = 0;
#pragma unroll
                for (int i = 0; i < 4; i++) a[i >> 1][i & 1].fold(c, f);
            }
            const float p0 = FqMac::part(pv.x), p1 = FqMac::part(pv.y);
            a[0][0].add(v0.x, FqMac::part(v0.x), pv.x, p0), a[0][1].add(v0.y, FqMac::part(v0.y), pv.y, p1);
            a[1][0].add(v1.x, FqMac::part(v1.x), pv.x, p0), a[1][1].add(v1.y, FqMac::part(v1.y), pv.y, p1);
        }
#pragma unroll
        for (int i = 0; i < 4; i++) o[i >> 1][i & 1] = a[i >> 1][i & 1].get(c, m.q, f);
    } else {
        U128 a[2][2] = {};
        for (int t = t0; t < t1; t++) {
            next(t);
            if (WIDE) {
                mac128_q(a[0][0], pv.x, v0.x, m.q), mac128_q(a[0][1], pv.y, v0.y, m.q);
                mac128_q(a[1][0], pv.x, v1.x, m.q), mac128_q(a[1][1], pv.y, v1.y, m.q);
            } else {
                mac128(a[0][0], pv.x, v0.x), mac128(a[0][1], pv.y, v0.y);
                mac128(a[1][0], pv.x, v1.x), mac128(a[1][1], pv.y, v1.y);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; i++) o[i >> 1][i & 1] = redc(a[i >> 1][i & 1].lo, a[i >> 1][i & 1].hi, m);
    }
#pragma unroll
    for (int c = 0; c < 2; c++) *(ulonglong2 *)(ob + c * per + idx) = make_ulonglong2(o[c][0], o[c][1]);
}
__global__ void __launch_bounds__(kPmulThreads) k_pmul_acc(u64 *out, long out_s, const __grid_constant__ PmulArgs pa, int B,
                                                  int rows, int logN, long Rs, RowMap qp, const ModQ *mods,
                                                  const ModF *modf) {
    __shared__ ulonglong2 ring[kPmulStages][3][kPmulThreads];   // a thread reads only what it copied
    pdl_trigger();
    pdl_wait();
    const long idx = 2 * ((long)blockIdx.y * 128 + threadIdx.x), per = (long)rows << logN;   // 256 | N
    const int pi = qp.at32((unsigned)(idx >> logN));
    const ModQ m = mods[pi];
    const ModF f = modf[pi];
    const int t0 = pa.first[blockIdx.x], t1 = pa.first[blockIdx.x + 1];
    u64 *o = out + blockIdx.x * out_s;
    for (int b = 0; b < B; b++) {   // the branches are uniform over the CTA
        u64 *ob = o + (long)b * 2 * per;
        if (f.on) pmul_item<true, false>(pa, t0, t1, idx, per, b * Rs, ob, m, f, ring);
        else if (m.q >= (1ull << 59)) pmul_item<false, true>(pa, t0, t1, idx, per, b * Rs, ob, m, f, ring);
        else pmul_item<false, false>(pa, t0, t1, idx, per, b * Rs, ob, m, f, ring);
    }
}
void launch_pmul_sums(Ctx *c, u64 *out, long out_s, const PmulTerm *terms, const int *first, int sums,
                      const u64 *const *R, int nR, int B, int level, long Rs, cudaStream_t st) {
    const int rows = level + 1 + c->alpha;
    // what PmulArgs holds, and what one reduction per output word takes
    if (nR > kMaxPmulRots) throw HeError(HE_ERR_ARG, "a plaintext sum takes at most 32 rotations");
    for (int y = 0; y < sums; y++)
        if (first[y + 1] - first[y] > kMaxPmulRots) throw HeError(HE_ERR_ARG, "a plaintext sum takes at most 32 terms");
    for (int y0 = 0, y1; y0 < sums; y0 = y1) {
        PmulArgs a;
        for (int j = 0; j < nR; j++) a.R[j] = R[j];
        for (y1 = y0 + 1; y1 < sums && y1 - y0 < kMaxPmulSums && first[y1 + 1] - first[y0] <= kMaxPmulTerms;) y1++;
        for (int y = y0; y <= y1; y++) a.first[y - y0] = (short)(first[y] - first[y0]);
        for (int t = first[y0]; t < first[y1]; t++)
            a.pt[t - first[y0]] = terms[t].pt, a.ri[t - first[y0]] = (unsigned char)terms[t].r;
        c->n_launch++;
        launch_pdl(k_pmul_acc, dim3((unsigned)(y1 - y0), (unsigned)((long)rows * c->N / 256)), 128, 0, st, 
            out + y0 * out_s, out_s, a, B, rows, c->logN, Rs, c->map_qp(level), c->d_mod, c->d_modf);
    }
}

__global__ void k_add_lifted(u64 *u, const u64 *d, int level, int rows, int logN, const ModQ *mods,
                             const ShoupPair *Pmod) {
    pdl_trigger();
    pdl_wait();
    const long N = 1L << logN, x = (long)blockIdx.x * 256 + threadIdx.x;   // 256 | N
    const int r = blockIdx.y;
    const u64 q = mods[r].q;
    const ShoupPair w = Pmod[r];
    u64 *o = u + ((long)blockIdx.z * rows + r) * N + x;
    *o = addmod(*o, shoup(d[((long)blockIdx.z * (level + 1) + r) * N + x], w.w, w.wp, q), q);
}
void launch_add_lifted(Ctx *c, u64 *u, const u64 *d, int B, int level, cudaStream_t st) {
    c->n_launch++;
    launch_pdl(k_add_lifted, dim3((unsigned)(c->N / 256), (unsigned)(level + 1), (unsigned)(2 * B)), 256, 0, st, u, d, level,
               c->qp_rows(level), c->logN, c->d_mod, c->d_Pmod);
}

// P * a over Q_l P: rows q_r get (P mod q_r) a_r, the p rows are zero.
// in: [items][l+1][N] (stride in_s), out: [items][l+1+alpha][N] (stride out_s)
__global__ void k_lift_P(u64 *out, const u64 *in, int items, int level, int alpha, int N, long is, long os,
                         const ModQ *mods, const ShoupPair *Pmod) {
    pdl_trigger();
    pdl_wait();
    long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    int rows = level + 1 + alpha;
    long per = (long)rows * N;
    if (idx >= (long)items * per) return;
    int it = (int)(idx / per);
    long off = idx - (long)it * per;
    int r = (int)(off / N);
    u64 v = 0;
    if (r <= level) {
        ShoupPair w = Pmod[r];
        v = shoup(in[it * is + off], w.w, w.wp, mods[r].q);
    }
    out[it * os + off] = v;
}
void launch_lift_P(Ctx *c, u64 *out_qp, const u64 *in_q, int items, int level, long is, long os, cudaStream_t st) {
    long n = (long)items * (level + 1 + c->alpha) * c->N;
    c->n_launch++;
    launch_pdl(k_lift_P, dim3(nblk(n, 256)), 256, 0, st, out_qp, in_q, items, level, c->alpha, c->N, is, os, c->d_mod,
                                           c->d_Pmod);
}

// ------------------------------------------------------------- Rescale
// t_i = [c_l]_{q_l} mod q_i for i < l (coefficient form): the centred residue
// of the last limb (reading of App. A Rescaling: round(c / q_l)).
// last: [items][N]; out: [items][l][N]
__global__ void k_rescale_prep(const u64 *last, u64 *out, int items, int level, int logN, const ModQ *mods,
                               const ModF *modf, const u64 *qlmod) {
    pdl_trigger();
    pdl_wait();
    const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long)items << logN) return;
    const int N = 1 << logN, x = (int)(idx & (N - 1)), it = (int)(idx >> logN);
    const u64 ql = mods[level].q;
    const u64 v = last[idx];
    const bool neg = v > (ql >> 1);
    const u64 t = neg ? v - ql : v;   // signed
    u64 *op = out + (long)it * level * N + x;
    for (int i = 0; i < level; i++) {
        const u64 q = mods[i].q;
        const ModF m = modf[i];
        u64 r;
        if (m.on && ql < 8 * q) {   // |t| <= 4 q
            r = fq_pos(fq_red(t, m), q);
        } else {
            r = reduce_any(v, q, mods[i].wone);
            if (neg) r = submod(r, qlmod[i], q);  // v - q_l
        }
        op[(long)i * N] = r;
    }
}
void launch_rescale_prep(Ctx *c, const u64 *lastcoef, u64 *out, int items, int level, cudaStream_t st) {
    const LevelConsts &L = c->lc(level);
    long n = (long)items * c->N;
    c->n_launch++;
    launch_pdl(k_rescale_prep, dim3(nblk(n, 256)), 256, 0, st, lastcoef, out, items, level, c->logN, c->d_mod, c->d_modf, L.d_rs_qlmod);
}

// out_i = (c_i - t_i) q_l^-1 mod q_i (NTT domain), i < l.
// in: [items][l+1][N] stride is; t: [items][l][N]; out: [items][l][N] stride os
__global__ void k_rescale_final(u64 *out, const u64 *in, const u64 *t, int items, int level, int N, long is, long os,
                                const ModQ *mods, const ShoupPair *inv) {
    pdl_trigger();
    pdl_wait();
    long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    long per = (long)level * N;
    if (idx >= (long)items * per) return;
    int it = (int)(idx / per);
    long off = idx - (long)it * per;
    int i = (int)(off / N);
    u64 q = mods[i].q;
    ShoupPair w = inv[i];
    out[it * os + off] = shoup(submod(in[it * is + off], t[idx], q), w.w, w.wp, q);
}
void launch_rescale_final(Ctx *c, u64 *out, const u64 *in, const u64 *t, int items, int level, long is, long os,
                          cudaStream_t st) {
    const LevelConsts &L = c->lc(level);
    long n = (long)items * level * c->N;
    c->n_launch++;
    launch_pdl(k_rescale_final, dim3(nblk(n, 256)), 256, 0, st, out, in, t, items, level, c->N, is, os, c->d_mod, L.d_rs_inv);
}

// ------------------------------------------------------------- decrypt
// m = c0 + c1 s on limb q_0 (NTT domain), written into out (u64 view).
__global__ void k_dec_q0(const u64 *c0, const u64 *c1, const u64 *skM, u64 *out, int N, const ModQ *mods) {
    pdl_trigger();
    pdl_wait();
    int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= N) return;
    const ModQ &m = mods[0];
    out[x] = addmod(c0[x], mulmont(c1[x], skM[x], m), m.q);
}
__global__ void k_centre_q0(const u64 *a, double *out, int N, const ModQ *mods) {
    pdl_trigger();
    pdl_wait();
    int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= N) return;
    u64 q = mods[0].q, v = a[x];
    out[x] = v > (q >> 1) ? -(double)(q - v) : (double)v;
}

// -------------------------------------------------------------- diagonals
// Slot vector (length S, period n^2) of a permutation-matrix diagonal,
// rotated left by `rot` (mod n^2) and multiplied by `value`:
//   kind 0  Z (sigma), eq. 5, index t in (-n, n)
//   kind 1  T (tau), eq. 6, index t = k n
//   kind 2  G (transpose), index t = (n-1) k, ones where column - row = k
//   kind 3  C^k mask 1 (columns j < n-k); kind 4  C^k mask 2 (j >= n-k)
//   kind 5  all ones (constant)
//   kind 6  first column (j == 0); kind 7  identity (i == j)
//   kind 10 row k (i == k); kind 11 column k (j == k)
__global__ void k_diag_fill(double *out, int S, int kind, int n, long t, long rot, double value, int k) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= S) return;
    long n2 = (long)n * n;
    long l = ((long)(p % n2) + rot) % n2;
    long i = l / n, j = l % n;
    bool one = false;
    switch (kind) {
    case 0:
        if (t >= 0) one = (l - n * t >= 0) && (l - n * t < n - t);
        else one = (l - (n + t) * n >= -t) && (l - (n + t) * n < n);
        break;
    case 1: one = (j == t / n); break;
    case 2: one = ((j - i) * (n - 1) == t); break;
    case 3: one = j < n - k; break;
    case 4: one = j >= n - k; break;
    case 5: one = true; break;
    case 6: one = (j == 0); break;
    case 7: one = (i == j); break;
    case 10: one = (i == k); break;
    case 11: one = (j == k); break;
    }
    out[p] = one ? value : 0.0;
}
void launch_diag_fill(Ctx *c, double *out, int kind, int n, long t, long rot, double value, int k, cudaStream_t st) {
    c->n_launch++;
    k_diag_fill<<<nblk(c->S, 256), 256, 0, st>>>(out, c->S, kind, n, t, rot, value, k);
}

void launch_copy_rows(u64 *dst, long dst_stride, const u64 *src, long src_stride, int items, long words,
                      cudaStream_t st) {
    cudaMemcpy2DAsync(dst, dst_stride * 8, src, src_stride * 8, words * 8, items, cudaMemcpyDeviceToDevice, st);
}

}  // namespace he

// exported for decrypt
namespace he {
void launch_dec_q0(Ctx *c, const u64 *c0, const u64 *c1, u64 *out, cudaStream_t st) {
    c->n_launch++;
    launch_pdl(k_dec_q0, dim3(nblk(c->N, 256)), 256, 0, st, c0, c1, c->d_skM, out, c->N, c->d_mod);
}
void launch_centre_q0(Ctx *c, const u64 *a, double *out, cudaStream_t st) {
    c->n_launch++;
    launch_pdl(k_centre_q0, dim3(nblk(c->N, 256)), 256, 0, st, a, out, c->N, c->d_mod);
}
}  // namespace he

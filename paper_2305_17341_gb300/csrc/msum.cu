// msum.cu -- the key switch's inner products (MultSum + Permute, Sec. 3.3.1).
//
// For G rotations that share one Decompose output (hoisting).  Rotation keys
// are stored permuted, K'_g[y] = K_g[x] with y = pi_g(x) the NTT-domain index of
// kappa_g, so that
//   out_g[x] = sum_d D[d][pi_g(x)] K_g[d][x] = T_g[pi_g(x)],
//   T_g[y]   = sum_d D[d][y] K'_g[d][y]
// and the result is written to x = pi_g^{-1}(y), which stays inside the aligned
// 32-word block of y (kappa permutes the low bits of the bit-reversed index
// only).  With c0 given, P c0[y] is added on the Q rows of poly 0 (the hoisted
// rotation kept in Q_l P of double hoisting).
// digits: [B][ndig][rows][N]; key_k: [dnum][2][nprimes][N]; out_k: [B][2][rows][N].
//
// Key words (and the masks and diagonals they meet) of a limb with ModF constants
// are plain and centred (|k| <= q/2), those of the others in Montgomery form
// (launch_key_form).
//
// What bounds it: with one load per product in flight the digit loop waited one
// memory round trip per digit (1.9 TB/s for the C^k babies of 8 items), and the
// 96-bit sums cost 7.5 multiply slots a product.  So
//  * the CTA's digit and key rows go through a four-deep ring of cp.async
//    stages, one digit a stage;
//  * a CTA takes the rotations of a chunk for a group of items, and the CTAs of
//    one block of coefficients are adjacent in the grid: each row comes from
//    DRAM once and from L2 for the others;
//  * a product is a wrapping 64-bit sum and an FP32 estimate of the quotient (4
//    slots), reduced once per output (FqMac).
// 8 items under 15 keys (N = 2^15, 10 digits): 1.80 -> 1.44 ms; one key: 180 ->
// 140 us; the C^k babies of a giant (8 items, N = 2^16, level 19): 7.09 -> 6.22
// ms, 1.1 of the 3.86 T products/s that the sums alone reach in registers: shared
// memory reads, folds, masks and the 60-bit rows (a tenth of the rows, four times
// the multiplies) take the rest of the issue slots.
#include <cstdio>
#include <set>

#include "bulkcopy.cuh"
#include "kernels.cuh"

namespace he {

// NTT-domain index of the automorphism X -> X^g
__device__ __forceinline__ int msum_auto(int x, u32 g, int logN) {
    const u32 sh = 32 - logN, e = 2u * (__brev((u32)x) >> sh) + 1u;
    const u32 e2 = (e * g) & ((2u << logN) - 1u);
    return (int)(__brev((e2 - 1) >> 1) >> sh);
}

constexpr int kMsKeys = 32, kMsStages = 4, kMsRows = 80;

struct MsumArgs {
    const u64 *key[kMsKeys];
    u64 *out[kMsKeys];
    const u64 *m1[kMsKeys], *m2[kMsKeys];   // C^k masks over Q_l P, [rows][N]
    u32 ginv[kMsKeys];                      // pi_g^{-1} = pi_{g^{-1} mod 2N}; 1 = identity
};
struct MsumGeom {
    int G, B;
    int wi, kw, xt;     // warps = wi (items) x kw (keys) x xt (blocks of 64 coefficients)
    int nig, nkc;       // item groups, key chunks
    int level, rows, L, ndig, nprimes, logN;
};

// A thread: two adjacent coefficients, NS digit streams (NS items; with CK the two
// sources of one item) and GK keys.
//
// CK: the C^k babies with their masks (Sec. 4.1, Table 1 "Optimized C^k"):
//   S_b = m_k (.) rot_qp(A_g; b) + m'_k (.) rot_qp(A'_g; b),
// both sources under the same keys; only S_b reaches memory.
template <int NS, int GK, bool CK>
__global__ void __launch_bounds__(256, NS * GK <= 2 ? 3 : 2) k_msum(const __grid_constant__ MsumArgs ma, const u64 *dig1, const u64 *dig2,
                                                 const MsumGeom g, const ModQ *mods, const ModF *modf, const u64 *c01,
                                                 const u64 *c02, long c0s, const ShoupPair *Pmod) {
    extern __shared__ __align__(16) u64 ms_ring[];
    __shared__ const u64 *s_src[kMsRows];
    __shared__ long s_str[kMsRows];
    pdl_trigger();
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long N = 1L << g.logN;
    const int kc = blockIdx.x % g.nkc, t1 = blockIdx.x / g.nkc, ig = t1 % g.nig, tile = t1 / g.nig;
    const int r = blockIdx.y, kr = r <= g.level ? r : g.L + 1 + (r - g.level - 1);   // the row's global prime
    const ModQ m = mods[kr];
    const ModF f = modf[kr];
    const int xi = w / (g.wi * g.kw), rem = w - xi * g.wi * g.kw, wi = rem % g.wi, kwi = rem / g.wi;
    const int R = g.wi * NS + 2 * g.kw * GK, tot = g.xt * R;
    const long ds = (long)g.rows * N, kd = 2L * g.nprimes * N, kk = (long)g.nprimes * N;
    for (int e = threadIdx.x; e < tot; e += 256) {
        const int x = e / R, q = e - x * R;
        const long y = (long)(tile * g.xt + x) * 64;
        if (q < g.wi * NS) {
            const int it = min(CK ? ig * g.wi + q / NS : ig * g.wi * NS + q, g.B - 1);   // rows past B repeat the last item
            s_src[e] = (CK && (q & 1) ? dig2 : dig1) + (long)it * g.ndig * ds + (long)r * N + y;
            s_str[e] = ds;
        } else {
            const int k = min(kc * g.kw * GK + (q - g.wi * NS) / 2, g.G - 1);
            s_src[e] = ma.key[k] + ((q - g.wi * NS) & 1) * kk + (long)kr * N + y;
            s_str[e] = kd;
        }
    }
    __syncthreads();
    pdl_wait();
    // a warp copies rows w, w + 8, ...: its first two rows' addresses run along in
    // registers (most splits have no more than 16 rows)
    const u64 *src0 = s_src[w < tot ? w : 0] + 2 * lane, *src1 = s_src[w + 8 < tot ? w + 8 : 0] + 2 * lane;
    const long str0 = s_str[w < tot ? w : 0], str1 = s_str[w + 8 < tot ? w + 8 : 0];
    const u32 ring = bc_smem(ms_ring + w * 64 + 2 * lane), stage = (u32)tot * 512;
    auto issue = [&](int d) {   // called for d = 0, 1, 2, ... in order
        if (d < g.ndig) {
            const u32 st = ring + (u32)(d & (kMsStages - 1)) * stage;
            if (w < tot) bc_copy16(st, src0);
            if (w + 8 < tot) bc_copy16(st + 8 * 512, src1);
            src0 += str0, src1 += str1;
            for (int e = w + 16; e < tot; e += 8) bc_copy16(st + (e - w) * 512, s_src[e] + d * s_str[e] + 2 * lane);
        }
        bc_commit();
    };
#pragma unroll
    for (int d = 0; d < kMsStages - 1; d++) issue(d);
    const int drow = (xi * R + wi * NS) * 64 + 2 * lane, krow = (xi * R + g.wi * NS + kwi * GK * 2) * 64 + 2 * lane;
    const u64 *digp = ms_ring + drow, *keyp = ms_ring + krow;
    const long y = (long)(tile * g.xt + xi) * 64 + 2 * lane;
    const bool q_row = r <= g.level;
    u64 o[NS][2 * GK][2];   // [stream][key, poly][coefficient]: residues
    if (f.on) {             // uniform over the CTA
        const FqMacC c(f, m.q);
        FqMac acc[NS][2 * GK][2];
#pragma unroll
        for (int j = 0; j < NS; j++)
#pragma unroll
            for (int k = 0; k < 2 * GK; k++)
#pragma unroll
                for (int e = 0; e < 2; e++) acc[j][k][e] = FqMac{0, 0, 0.0f};
        // runs of at most lim digits; the sums are folded between them (outside the
        // digit loop, whose registers the fold would otherwise constrain)
        for (int d0 = 0; d0 < g.ndig; d0 += c.lim) {
            if (d0) {
#pragma unroll
                for (int j = 0; j < NS; j++)
#pragma unroll
                    for (int k = 0; k < 2 * GK; k++)
#pragma unroll
                        for (int e = 0; e < 2; e++) acc[j][k][e].fold(c, f);
            }
            const int d1 = min(g.ndig, d0 + c.lim);
            for (int d = d0; d < d1; d++) {
                bc_wait_groups<kMsStages - 2>();
                __syncthreads();   // stage d has landed; stage d - 1's readers are done
                issue(d + kMsStages - 1);
                const int so = (d & (kMsStages - 1)) * tot * 64;
                ulonglong2 v[NS];
                float vf[NS][2];
#pragma unroll
                for (int j = 0; j < NS; j++) {
                    v[j] = *(const ulonglong2 *)(digp + so + j * 64);
                    vf[j][0] = FqMac::part(v[j].x), vf[j][1] = FqMac::part(v[j].y);
                }
#pragma unroll
                for (int k = 0; k < 2 * GK; k++) {
                    const ulonglong2 kv = *(const ulonglong2 *)(keyp + so + k * 64);
                    const float k0 = FqMac::part(kv.x), k1 = FqMac::part(kv.y);
#pragma unroll
                    for (int j = 0; j < NS; j++) {
                        acc[j][k][0].add(v[j].x, vf[j][0], kv.x, k0);
                        acc[j][k][1].add(v[j].y, vf[j][1], kv.y, k1);
                    }
                }
            }
        }
        if (c01 && q_row) {
            // P c0 is one more product of each poly-0 sum
            const u64 Pw = Pmod[r].w, Pc = Pw > m.q / 2 ? Pw - m.q : Pw;
            const float Pf = FqMac::part(Pc);
#pragma unroll
            for (int j = 0; j < NS; j++) {
                const int it = min(CK ? ig * g.wi + wi : (ig * g.wi + wi) * NS + j, g.B - 1);
                const ulonglong2 cv = *(const ulonglong2 *)((CK && j ? c02 : c01) + it * c0s + (long)r * N + y);
                const float f0 = FqMac::part(cv.x), f1 = FqMac::part(cv.y);
#pragma unroll
                for (int k = 0; k < GK; k++) {
                    acc[j][2 * k][0].add(cv.x, f0, Pc, Pf);
                    acc[j][2 * k][1].add(cv.y, f1, Pc, Pf);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < NS; j++)
#pragma unroll
            for (int k = 0; k < 2 * GK; k++)
#pragma unroll
                for (int e = 0; e < 2; e++) {
                    if constexpr (CK) {   // signed, |.| < 1.5 q: the masks' products reduce
                        acc[j][k][e].fold(c, f);
                        o[j][k][e] = ((u64)acc[j][k][e].a1 << 32) | acc[j][k][e].a0;
                    } else {
                        o[j][k][e] = acc[j][k][e].get(c, m.q, f);
                    }
                }
    } else {
        WideMac acc[NS][2 * GK][2];
#pragma unroll
        for (int j = 0; j < NS; j++)
#pragma unroll
            for (int k = 0; k < 2 * GK; k++) acc[j][k][0] = acc[j][k][1] = WideMac{0, 0, 0, 0};
        for (int d = 0; d < g.ndig; d++) {
            bc_wait_groups<kMsStages - 2>();
            __syncthreads();
            issue(d + kMsStages - 1);
            const long so = (long)(d & (kMsStages - 1)) * tot * 64;
            ulonglong2 v[NS];
#pragma unroll
            for (int j = 0; j < NS; j++) v[j] = *(const ulonglong2 *)(digp + so + j * 64);
#pragma unroll
            for (int k = 0; k < 2 * GK; k++) {
                const ulonglong2 kv = *(const ulonglong2 *)(keyp + so + k * 64);
#pragma unroll
                for (int j = 0; j < NS; j++) {
                    acc[j][k][0].add(v[j].x, kv.x);
                    acc[j][k][1].add(v[j].y, kv.y);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < NS; j++)
#pragma unroll
            for (int k = 0; k < 2 * GK; k++)
#pragma unroll
                for (int e = 0; e < 2; e++) o[j][k][e] = acc[j][k][e].get(m);
    }
    // the copies still in flight are empty groups (issue past ndig): nothing to drain
    const ShoupPair wP = c01 && q_row && !f.on ? Pmod[r] : ShoupPair{0, 0};
#pragma unroll
    for (int j = 0; j < NS; j++) {
        const int it = CK ? ig * g.wi + wi : (ig * g.wi + wi) * NS + j;
        if (it >= g.B) continue;
        if (c01 && q_row && !f.on) {
            const u64 *cp = (CK && j ? c02 : c01) + it * c0s + (long)r * N + y;
            const ulonglong2 cv = *(const ulonglong2 *)cp;
            const u64 p0 = shoup(cv.x, wP.w, wP.wp, m.q), p1 = shoup(cv.y, wP.w, wP.wp, m.q);
#pragma unroll
            for (int k = 0; k < GK; k++) {
                o[j][2 * k][0] = addmod(o[j][2 * k][0], p0, m.q);
                o[j][2 * k][1] = addmod(o[j][2 * k][1], p1, m.q);
            }
        }
        if (CK && j == 0) continue;
#pragma unroll
        for (int k = 0; k < GK; k++) {
            const int ki = kc * g.kw * GK + kwi * GK + k;
            if (ki >= g.G) continue;
            u64 *ob = ma.out[ki] + (long)it * 2 * ds + (long)r * N;
            const u32 gi = ma.ginv[ki];
#pragma unroll
            for (int e = 0; e < 2; e++) {
                const int x = gi == 1u ? (int)y + e : msum_auto((int)y + e, gi, g.logN);
                u64 o0 = o[j][2 * k][e], o1 = o[j][2 * k + 1][e];
                if constexpr (CK) {
                    const u64 w1 = __ldg(ma.m1[ki] + (long)r * N + x), w2 = __ldg(ma.m2[ki] + (long)r * N + x);
                    if (f.on) {   // |sums| < 1.5 q, masks plain and centred
                        const float c = FqMacC(f, m.q).c;
                        const ulonglong2 v1 = fq_svar(w1, c), v2 = fq_svar(w2, c);
                        o0 = fq_pos(fq_red(fq_mul(o[0][2 * k][e], v1, f) + fq_mul(o0, v2, f), f), m.q);
                        o1 = fq_pos(fq_red(fq_mul(o[0][2 * k + 1][e], v1, f) + fq_mul(o1, v2, f), f), m.q);
                    } else {
                        U128 s0 = {0, 0}, s1 = {0, 0};   // two products below q^2: below q 2^64
                        mac128(s0, w1, o[0][2 * k][e]);
                        mac128(s0, w2, o0);
                        mac128(s1, w1, o[0][2 * k + 1][e]);
                        mac128(s1, w2, o1);
                        o0 = redc(s0.lo, s0.hi, m);
                        o1 = redc(s1.lo, s1.hi, m);
                    }
                }
                ob[x] = o0;
                ob[ds + x] = o1;
            }
        }
    }
}

// ------------------------------------------------------------------ launches
// Ways to split a launch's 8 warps over items, keys and coefficients.
struct MsumCfg {
    int ns, gk, wi, kw, xt;
    int rows() const { return xt * (wi * ns + 2 * kw * gk); }
};
static std::vector<MsumCfg> msum_cfgs(int B, int G, bool ck) {
    std::vector<MsumCfg> v;
    const int ns = ck || B >= 2 ? 2 : 1, per = ck ? 1 : ns;
    const int ni = (B + per - 1) / per;
    auto splits = [&](int gk) {
        const int nk = (G + gk - 1) / gk;
        for (int wi = 1; wi <= 8 && wi < 2 * ni; wi *= 2)
            for (int kw = 1; kw * wi <= 8 && kw < 2 * nk; kw *= 2) {
                const MsumCfg c{ns, gk, wi, kw, 8 / (wi * kw)};
                if (c.rows() <= kMsRows) v.push_back(c);
            }
    };
    // one item leaves registers for four keys a thread, but their rows take the
    // shared memory of a whole SM: two keys a thread are timed as well (the 15
    // babies of a sigma, the best split of each: 188 us with four, 145 with two at
    // N = 2^15, level 11; 834 and 684 at N = 2^16, level 20)
    splits(G < 2 ? 1 : 2);
    if (ns == 1 && G >= 4) splits(4);
    // fewest rows first: the most products per word brought in
    std::stable_sort(v.begin(), v.end(), [](const MsumCfg &a, const MsumCfg &b) { return a.rows() < b.rows(); });
    return v;
}

template <auto KERN, class... A>
static void msum_go(const Ctx *c, dim3 grid, size_t smem, cudaStream_t st, A... args) {
    static std::atomic<bool> raised[64];
    // dynamic and static shared memory together pass 48 KB
    if (smem > 40 * 1024 && !raised[c->device & 63].load(std::memory_order_acquire)) {
        cudaFuncSetAttribute(KERN, cudaFuncAttributeMaxDynamicSharedMemorySize, kMsStages * kMsRows * 512);
        raised[c->device & 63].store(true, std::memory_order_release);
    }
    launch_pdl(KERN, grid, 256, smem, st, args...);
}

struct MsumCall {
    u64 *const *outs;
    const u64 *dig1, *dig2;
    const u64 *const *keys;
    const uint32_t *gs;
    const u64 *const *m1, *const *m2;
    int B, level, rows;
    const u64 *c01, *c02;
    long c0s;
};

// keys k0 .. k0 + G (at most kMsKeys) in one launch
static void msum_launch(Ctx *c, const MsumCall &a, const MsumCfg &cf, int k0, int G, cudaStream_t st) {
    MsumArgs ma = {};
    const u32 M = 2u * (u32)c->N;
    for (int k = 0; k < G; k++) {
        ma.key[k] = a.keys[k0 + k];
        ma.out[k] = a.outs[k0 + k];
        if (a.m1) ma.m1[k] = a.m1[k0 + k], ma.m2[k] = a.m2[k0 + k];
        u32 g = a.gs[k0 + k], inv = g;   // inverse of the odd g modulo 2N (Newton on 32-bit words)
        for (int it = 0; it < 5; it++) inv *= 2u - g * inv;
        ma.ginv[k] = inv & (M - 1);
    }
    const bool ck = a.m1 != nullptr;
    MsumGeom g;
    const int per = ck ? 1 : cf.ns;
    g.G = G, g.B = a.B, g.wi = cf.wi, g.kw = cf.kw, g.xt = cf.xt;
    g.nig = (a.B + cf.wi * per - 1) / (cf.wi * per), g.nkc = (G + cf.kw * cf.gk - 1) / (cf.kw * cf.gk);
    g.level = a.level, g.rows = a.rows, g.L = c->L, g.ndig = c->ndig(a.level), g.nprimes = c->nprimes, g.logN = c->logN;
    const dim3 grid((unsigned)((long)(c->N / (64 * cf.xt)) * g.nig * g.nkc), (unsigned)a.rows);
    const size_t smem = (size_t)kMsStages * cf.rows() * 512;
    c->n_launch++;
#define MS_GO(NS, GK, CK)                                                                                         \
    msum_go<k_msum<NS, GK, CK>>(c, grid, smem, st, ma, a.dig1, a.dig2, g, (const ModQ *)c->d_mod,                 \
                                (const ModF *)c->d_modf, a.c01, a.c02, a.c0s, (const ShoupPair *)c->d_Pmod)
    if (ck) {
        if (cf.gk == 2) MS_GO(2, 2, true);
        else MS_GO(2, 1, true);
    } else if (cf.ns == 2) {
        if (cf.gk == 2) MS_GO(2, 2, false);
        else MS_GO(2, 1, false);
    } else {
        if (cf.gk == 4) MS_GO(1, 4, false);
        else if (cf.gk == 2) MS_GO(1, 2, false);
        else MS_GO(1, 1, false);
    }
#undef MS_GO
}

static void msum_run(Ctx *c, const MsumCall &a, const MsumCfg &cf, int G, bool traced, cudaStream_t st) {
    const bool ck = a.m1 != nullptr;
    for (int k0 = 0; k0 < G; k0 += kMsKeys) {
        const int g = std::min(kMsKeys, G - k0);
        cudaEvent_t e0 = nullptr;
        if (traced) c->trace_begin(0, e0);
        msum_launch(c, a, cf, k0, g, st);
        if (traced) {
            // algorithmic bytes: every key (and mask) read once, every item's
            // digits (of both sources) and c0 once, every output written once
            const double nd = c->ndig(a.level), W = 8.0 * c->N, s = ck ? 2.0 : 1.0;
            const double bytes = W * (g * (2.0 * nd + (ck ? 2.0 : 0.0)) * a.rows +
                                      (double)a.B * (s * nd * a.rows + g * 2.0 * a.rows + (a.c01 ? s * (a.level + 1) : 0.0)));
            c->trace_end(0, e0, bytes, (double)a.B * nd * a.rows * c->N * 2.0 * s * g);
        }
    }
}

// Split of a launch: pinned, tuned on its first use (every split timed twice on
// these very launches; the words do not depend on it), or the one with the
// fewest rows.
static void msum_tuned(Ctx *c, const MsumCall &a, int G, std::map<std::tuple<int, int, int>, int> &tuned, cudaStream_t st) {
    const bool ck = a.m1 != nullptr;
    const std::vector<MsumCfg> cf = msum_cfgs(a.B, std::min(G, kMsKeys), ck);
    int pick = 0;
    if (c->force_multsum >= 0) {
        pick = c->force_multsum % (int)cf.size();
    } else if (c->autotune && cf.size() > 1) {
        const auto key = std::make_tuple(a.level * 64 + a.rows - a.level, a.B, G);
        auto it = tuned.find(key);
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        cudaStreamIsCapturing(st, &cap);
        if (it != tuned.end()) {
            pick = it->second;
        } else if (cap == cudaStreamCaptureStatusNone) {
            cudaEvent_t e0 = c->ev_get(), e1 = c->ev_get();
            float best = 1e30f;
            for (int i = 0; i < (int)cf.size(); i++) {
                float t = 1e30f;
                for (int rep = 0; rep < 2; rep++) {
                    cudaEventRecord(e0, st);
                    msum_run(c, a, cf[i], G, false, st);
                    cudaEventRecord(e1, st);
                    cudaEventSynchronize(e1);
                    float ms = 0;
                    cudaEventElapsedTime(&ms, e0, e1);
                    t = std::min(t, ms);
                }
                if (t < best) best = t, pick = i;
                char line[160];
                if (ck)
                    snprintf(line, sizeof line, "multsum_ck level %d B %d G %d chunk %d BI %d ms %.4f\n", a.level, a.B, G,
                             cf[i].kw * cf[i].gk, cf[i].wi, t);
                else
                    snprintf(line, sizeof line, "multsum level %d B %d G %d chunk %d BI %d stream %d ms %.4f\n", a.level,
                             a.B, G, cf[i].kw * cf[i].gk, cf[i].wi * cf[i].ns, 0, t);
                c->tune_log += line;
            }
            c->ev_free.push_back(e0);
            c->ev_free.push_back(e1);
            tuned[key] = pick;
        }
    }
    msum_run(c, a, cf[pick], G, true, st);
}

void launch_multsum_multi(Ctx *c, u64 *const *outs, const u64 *digits, const u64 *const *keys, const uint32_t *gs, int G,
                          int B, int level, const u64 *c0_for_P, long c0s, cudaStream_t st) {
    if (G <= 0) return;
    const MsumCall a{outs, digits, nullptr, keys, gs, nullptr, nullptr, B, level, level + 1 + c->alpha, c0_for_P, nullptr, c0s};
    msum_tuned(c, a, G, c->tune_multsum, st);
}

void launch_multsum(Ctx *c, u64 *out, const u64 *digits, const u64 *key, uint32_t g, int B, int level,
                    const u64 *c0_for_P, long c0s, cudaStream_t st) {
    launch_multsum_multi(c, &out, digits, &key, &g, 1, B, level, c0_for_P, c0s, st);
}

// The inner product with one key on the rows of Q alone: digits [B][ndig][l+1][N]
// -> out [B][2][l+1][N] (the key without permutation).
void launch_multsum_q(Ctx *c, u64 *out, const u64 *digits, const u64 *key, int B, int level, cudaStream_t st) {
    const uint32_t g = 1;
    const MsumCall a{&out, digits, nullptr, &key, &g, nullptr, nullptr, B, level, level + 1, nullptr, nullptr, 0};
    msum_tuned(c, a, 1, c->tune_multsum, st);
}

// The C^k babies of a giant with their masks (CK above): G rotations of two
// sources with the same keys.
void launch_multsum_ck(Ctx *c, u64 *const *outs, const u64 *dig1, const u64 *dig2, const u64 *const *keys,
                       const uint32_t *gs, const u64 *const *m1, const u64 *const *m2, int G, int B, int level,
                       const u64 *c01, const u64 *c02, long c0s, cudaStream_t st) {
    if (G <= 0) return;
    const MsumCall a{outs, dig1, dig2, keys, gs, m1, m2, B, level, level + 1 + c->alpha, c01, c02, c0s};
    msum_tuned(c, a, G, c->tune_ck, st);
}

// ------------------------------------------------------------ summed giants
// MultSum + Permute of the G giants of a BSGS transform, summed: every giant
// has its own digits, key and automorphism, and
//   out[x] = in[x] + sum_g (T_g[y_g] + P c0_g[y_g]),  y_g = pi_g(x).
// A thread owns the output word, so the sum over giants and digits is one
// accumulation with one reduction; the words of a giant are read at permuted
// positions inside aligned 32-word blocks.  digits: [G][B][ndig][rows][N]; c0:
// [G][B] ciphertexts at stride c0s; in (may be null, or equal out), out: [B][2]
// [rows][N].
// Only the keys are loaded through the read-only path: the digits are written by
// the kernel before, which may still run when this grid starts.
struct GiantArgs {
    const u64 *key[kMaxGiants];
    u32 g[kMaxGiants];
};
__global__ void __launch_bounds__(256, 4) k_multsum_giants(const __grid_constant__ GiantArgs ga, int G, u64 *out,
                                                           const u64 *in, const u64 *digits, int B, int BI, int level,
                                                           int alpha, int L, int ndig, int nprimes, int logN,
                                                           const ModQ *mods, const ModF *modf, const u64 *c0, long c0s,
                                                           const ShoupPair *Pmod) {
    pdl_trigger();
    pdl_wait();
    const int N = 1 << logN;
    const int XW = 256 / BI;
    const int tx = threadIdx.x % XW, ti = threadIdx.x / XW;
    const int x = blockIdx.x * XW + tx;
    const int r = blockIdx.y;
    const int b = blockIdx.z * BI + ti;
    if (b >= B || x >= N) return;
    const int rows = level + 1 + alpha;
    const int kr = r <= level ? r : L + 1 + (r - level - 1);
    const ModQ m = mods[kr];
    const ModF f = modf[kr];
    const long ds = (long)rows * N, kd = 2L * nprimes * N, kk = (long)nprimes * N;
    const bool q_row = r <= level;
    const ShoupPair w = q_row ? Pmod[r] : ShoupPair{0, 0};
    u64 pc = 0, o0, o1;
    auto giant = [&](int g, const u64 *&dp, const u64 *&kp) {
        const int y = msum_auto(x, ga.g[g], logN);
        dp = digits + ((long)g * B + b) * ndig * ds + (long)r * N + y;
        kp = ga.key[g] + (long)kr * N + y;
        if (q_row) pc = addmod(pc, shoup(c0[((long)g * B + b) * c0s + (long)r * N + y], w.w, w.wp, m.q), m.q);
    };
    if (f.on) {   // uniform over the CTA
        const FqMacC c(f, m.q);
        FqMac a0 = {0, 0, 0.0f}, a1 = {0, 0, 0.0f};
        int run = 0;
        for (int g = 0; g < G; g++) {
            const u64 *dp, *kp;
            giant(g, dp, kp);
#pragma unroll 4
            for (int d = 0; d < ndig; d++) {
                const u64 v = dp[d * ds], k0 = __ldg(kp + d * kd), k1 = __ldg(kp + d * kd + kk);
                if (run == c.lim) run = 0, a0.fold(c, f), a1.fold(c, f);
                run++;
                const float vf = FqMac::part(v);
                a0.add(v, vf, k0, FqMac::part(k0));
                a1.add(v, vf, k1, FqMac::part(k1));
            }
        }
        o0 = a0.get(c, m.q, f), o1 = a1.get(c, m.q, f);
    } else {
        // giant by giant: one giant's digits (at most 48) stay below 2^128
        o0 = o1 = 0;
        for (int g = 0; g < G; g++) {
            const u64 *dp, *kp;
            giant(g, dp, kp);
            WideMac a0 = {0, 0, 0, 0}, a1 = {0, 0, 0, 0};
#pragma unroll 4
            for (int d = 0; d < ndig; d++) {
                const u64 v = dp[d * ds];
                a0.add(v, __ldg(kp + d * kd));
                a1.add(v, __ldg(kp + d * kd + kk));
            }
            o0 = addmod(o0, a0.get(m), m.q), o1 = addmod(o1, a1.get(m), m.q);
        }
    }
    o0 = addmod(o0, pc, m.q);
    const long o = (long)b * 2 * ds + (long)r * N + x;
    if (in) o0 = addmod(o0, in[o], m.q), o1 = addmod(o1, in[o + ds], m.q);
    out[o] = o0;
    out[o + ds] = o1;
}
void launch_multsum_giants(Ctx *c, u64 *out, const u64 *in, const u64 *digits, const u64 *const *keys,
                           const uint32_t *gs, int G, int B, int level, const u64 *c0, long c0s, cudaStream_t st) {
    GiantArgs ga;
    for (int g = 0; g < G; g++) ga.key[g] = keys[g], ga.g[g] = gs[g];
    int BI = 8;
    while (BI > 1 && BI > B) BI >>= 1;
    const int XW = 256 / BI, rows = level + 1 + c->alpha, nd = c->ndig(level);
    c->n_launch++;
    cudaEvent_t e0;
    c->trace_begin(0, e0);
    launch_pdl(k_multsum_giants, dim3((unsigned)((c->N + XW - 1) / XW), (unsigned)rows, (unsigned)((B + BI - 1) / BI)), 256,
               0, st, ga, G, out, in, digits, B, BI, level, c->alpha, c->L, nd, c->nprimes, c->logN, c->d_mod, c->d_modf,
               c0, c0s, c->d_Pmod);
    const double W = 8.0 * c->N;
    c->trace_end(0, e0, W * (G * 2.0 * nd * rows + (double)B * (G * ((double)nd * rows + level + 1) + (in ? 4.0 : 2.0) * rows)),
                 (double)B * G * nd * rows * c->N * 2.0);
}

// The relinearisation's inner product on the P rows of a run's terms: u [items][2]
// [A][N] = sum_d digP[item][d][j] key[d][poly][L + 1 + j], A = alpha; two adjacent
// words per thread, 8 items per CTA sharing the key words (the only ones loaded
// through the read-only path, as in k_multsum_giants).
__global__ void __launch_bounds__(256, 4) k_relin_ms(u64 *u, const u64 *digP, const u64 *key, int items, int A, int ndig,
                                                     int logN, int Lp1, int nprimes, const ModQ *mods, const ModF *modf) {
    pdl_trigger();
    pdl_wait();
    const long N = 1L << logN;
    const int tx = threadIdx.x & 31, ti = threadIdx.x >> 5;
    const int x = 2 * (blockIdx.x * 32 + tx), j = blockIdx.y;
    const long it = (long)blockIdx.z * 8 + ti;
    if (it >= items) return;
    const ModQ m = mods[Lp1 + j];
    const ModF f = modf[Lp1 + j];
    const u64 *kp = key + (long)(Lp1 + j) * N + x, *dp = digP + (it * ndig * A + j) * N + x;
    const long kd = 2L * nprimes * N, kk = (long)nprimes * N;
    u64 o[2][2];
    if (f.on) {   // uniform over the CTA
        const FqMacC c(f, m.q);
        FqMac a[2][2] = {};
        for (int d = 0, run = 0; d < ndig; d++, run++) {
            const ulonglong2 v = *(const ulonglong2 *)(dp + (long)d * A * N);
            if (run == c.lim) {
                run = 0;
#pragma unroll
                for (int i = 0; i < 4; i++) a[i >> 1][i & 1].fold(c, f);
            }
#pragma unroll
            for (int p = 0; p < 2; p++) {
                const ulonglong2 k = __ldg((const ulonglong2 *)(kp + d * kd + p * kk));
                a[p][0].add(v.x, FqMac::part(v.x), k.x, FqMac::part(k.x));
                a[p][1].add(v.y, FqMac::part(v.y), k.y, FqMac::part(k.y));
            }
        }
#pragma unroll
        for (int i = 0; i < 4; i++) o[i >> 1][i & 1] = a[i >> 1][i & 1].get(c, m.q, f);
    } else {
        WideMac a[2][2] = {};
        for (int d = 0; d < ndig; d++) {
            const ulonglong2 v = *(const ulonglong2 *)(dp + (long)d * A * N);
#pragma unroll
            for (int p = 0; p < 2; p++) {
                const ulonglong2 k = __ldg((const ulonglong2 *)(kp + d * kd + p * kk));
                a[p][0].add(v.x, k.x);
                a[p][1].add(v.y, k.y);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; i++) o[i >> 1][i & 1] = a[i >> 1][i & 1].get(m);
    }
#pragma unroll
    for (int p = 0; p < 2; p++) *(ulonglong2 *)(u + ((it * 2 + p) * A + j) * N + x) = make_ulonglong2(o[p][0], o[p][1]);
}
void launch_relin_ms(Ctx *c, u64 *u, const u64 *digP, int items, int ndig, cudaStream_t st) {
    c->n_launch++;
    launch_pdl(k_relin_ms, dim3((unsigned)(c->N / 64), (unsigned)c->alpha, (unsigned)((items + 7) / 8)), 256, 0, st, u, digP,
               c->rlk, items, c->alpha, ndig, c->logN, c->L + 1, c->nprimes, c->d_mod, c->d_modf);
}

// ------------------------------------------------------------------ key form
// Rows (row r of prime rm.at(r)) into the form above, in place.
__global__ void k_key_form(u64 *k, long rows, RowMap rm, int logN, const ModQ *mods, const ModF *modf) {
    const long idx = (long)blockIdx.x * 256 + threadIdx.x;   // 256 | N
    const long row = idx >> logN;
    if (row >= rows) return;
    const int p = rm.at32((unsigned)row);
    const ModQ m = mods[p];
    const u64 v = k[idx];
    k[idx] = modf[p].on ? (v > m.q / 2 ? v - m.q : v) : mulmont(v, m.r2, m);
}
void launch_key_form(Ctx *c, u64 *key, long rows, const RowMap &rm, cudaStream_t st) {
    c->n_launch++;
    k_key_form<<<(unsigned)(rows * (long)c->N / 256), 256, 0, st>>>(key, rows, rm, c->logN, c->d_mod, c->d_modf);
}

// Integer roofline of MultSum: the rate of its inner step on the 40-bit limbs
// (FqMac::add with both factors' float parts at hand), operands in registers, 16
// independent sums per thread, 8 CTAs of 256 threads per SM.  Only the
// instruction stream matters; a store that never happens keeps it alive.
__global__ void __launch_bounds__(256, 3) k_mac_peak(u64 *sink, int iters, u64 seed) {
    FqMac a[16];
    u64 kk[4];
    float kf[4];
    u64 v = (seed ^ threadIdx.x) & ((1ull << 40) - 1);
#pragma unroll
    for (int k = 0; k < 16; k++) a[k] = FqMac{0, 0, 0.0f};
#pragma unroll
    for (int k = 0; k < 4; k++) kk[k] = (seed * (k + 3) + threadIdx.x) & ((1ull << 39) - 1), kf[k] = FqMac::part(kk[k]);
    for (int it = 0; it < iters; it++) {
        v = (v + 0x9E3779B97F4A7C15ull) & ((1ull << 40) - 1);
        const float vf = FqMac::part(v);
#pragma unroll
        for (int k = 0; k < 16; k++) a[k].add(v, vf, kk[k & 3] ^ it, kf[k & 3]);
    }
    u64 acc = 0;
#pragma unroll
    for (int k = 0; k < 16; k++) acc ^= (((u64)a[k].a1 << 32) | a[k].a0) ^ __float_as_uint(a[k].s);
    if (acc == 0x1234567ull) sink[0] = acc;
}

double mac_peak(int iters) {
    int nsm = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    u64 *sink;
    cudaMalloc(&sink, 8);
    const int blocks = nsm * 8, threads = 256;
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    k_mac_peak<<<blocks, threads>>>(sink, 16, 12345);   // warm-up
    cudaEventRecord(a);
    k_mac_peak<<<blocks, threads>>>(sink, iters, 12345);
    cudaEventRecord(b);
    cudaEventSynchronize(b);
    float ms = 0;
    cudaEventElapsedTime(&ms, a, b);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    cudaFree(sink);
    return (double)blocks * threads * iters * 16.0 / (ms * 1e-3);
}

}  // namespace he

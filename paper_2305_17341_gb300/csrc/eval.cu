// eval.cu -- key switching, rotations, products, rescale, the double-hoisted
// linear transforms and the JKLS matrix product, all on batches of B
// ciphertexts laid out contiguously as [B][2][level+1][N] (NTT domain).
#include <algorithm>
#include <cmath>
#include <memory>
#include <sstream>

#include "eval.h"

namespace he {

// ------------------------------------------------------------ key switch
// Decompose (Sec. 3.3): poly of every item (stride item_s) -> digits
// [B][ndig][l+1+alpha][N] in the NTT domain.
void modup(Ctx *c, const u64 *poly, long item_s, int B, int level, u64 *digits) {
    const int N = c->N, nq = level + 1;
    Buf coef(&c->pool, (size_t)B * nq * N);
    ntt_inv(c, coef.p, (long)B * nq, c->map_q(level), c->stream, NttSrc{poly, item_s, nq});
    const long rows = (long)B * c->ndig(level) * c->qp_rows(level);
    if (c->logN >= 14 && c->logN <= 16) {
        // the digit's own rows are the input's NTT-domain rows: copy them and
        // transform only the extended rows
        launch_modup_bconv(c, coef.p, digits, B, level, c->stream, poly, item_s);
        RowSkip sk;
        sk.rows_per_digit = c->qp_rows(level);
        sk.ndig = c->ndig(level);
        sk.alpha = c->alpha;
        sk.nq = nq;
        ntt_fwd(c, digits, rows, c->map_qp(level), c->stream, &sk);
    } else {
        launch_modup_bconv(c, coef.p, digits, B, level, c->stream);
        ntt_fwd(c, digits, rows, c->map_qp(level), c->stream);
    }
    c->n_dp += B;
}

// ModDown: items of [rows][N] over Q_l P (contiguous) -> out items of [l+1][N]
// with item stride out_s.
void moddown(Ctx *c, const u64 *u, int items, int level, u64 *out, long out_s, const u64 *add, long add_s) {
    const int N = c->N, rows = c->qp_rows(level), a = c->alpha;
    Buf pc(&c->pool, (size_t)items * a * N), conv(&c->pool, (size_t)items * (level + 1) * N);
    ntt_inv(c, pc.p, (long)items * a, c->map_p(), c->stream, NttSrc{u + (long)(level + 1) * N, (long)rows * N, a});
    launch_moddown_bconv(c, pc.p, conv.p, items, level, c->stream);
    if (c->logN >= 14 && c->logN <= 16) {
        // the NTT's last pass writes out = (u_Q - conv) P^-1 directly
        SubScale ep;
        ep.u = u, ep.us = (long)rows * N, ep.out = out, ep.os = out_s, ep.w = c->d_dn_Pinv, ep.wf = c->d_dn_Pinvf;
        ep.rows_per_item = level + 1;
        ep.add = add, ep.as = add_s;
        ntt_fwd_subscale(c, conv.p, (long)items * (level + 1), c->map_q(level), c->stream, ep);
    } else {
        ntt_fwd(c, conv.p, (long)items * (level + 1), c->map_q(level), c->stream);
        launch_moddown_final(c, out, u, conv.p, add, items, level, (long)rows * N, out_s, add_s, c->stream);
    }
}

const u64 *need_key(Ctx *c, uint32_t g) {
    auto it = c->rtk.find(g);
    if (it == c->rtk.end()) {
        std::ostringstream os;
        os << "rotation key for Galois element " << g << " missing";
        throw HeError(HE_ERR_KEY_MISSING, os.str());
    }
    return it->second;
}

// Hoisted rotation kept in Q_l P: u = <kappa_g(digits), rtk_g> + (P kappa_g(c0), 0).
// ct: [B][2][l+1][N]; out: [B][2][rows][N].
void rot_qp(Ctx *c, const u64 *ct, int B, int level, const u64 *digits, uint32_t g, u64 *out) {
    const u64 *key = need_key(c, g);
    launch_multsum(c, out, digits, key, g, B, level, ct, 2L * (level + 1) * c->N, c->stream);
    c->n_ms += B;
}

// G hoisted rotations of the same Decompose output, kept in Q_l P; the
// digits are read once per launch for the keys of a launch.
void rot_qp_multi(Ctx *c, const u64 *ct, int B, int level, const u64 *digits, const uint32_t *gs, int G,
                  u64 *const *outs) {
    if (G <= 0) return;
    std::vector<const u64 *> keys(G);
    for (int k = 0; k < G; k++) keys[k] = need_key(c, gs[k]);
    launch_multsum_multi(c, outs, digits, keys.data(), gs, G, B, level, ct, 2L * (level + 1) * c->N, c->stream);
    c->n_ms += (long long)B * G;
}

// Full rotation from precomputed digits: ModDown(rot_qp) = kappa(c0) + ModDown(IP0), ModDown(IP1).
void rotate_digits(Ctx *c, const u64 *ct, int B, int level, const u64 *digits, uint32_t g, u64 *out) {
    const int rows = c->qp_rows(level);
    Buf u(&c->pool, (size_t)B * 2 * rows * c->N);
    rot_qp(c, ct, B, level, digits, g, u.p);
    moddown(c, u.p, 2 * B, level, out, (long)(level + 1) * c->N);
    c->n_md += B;
}

void rotate(Ctx *c, const u64 *ct, int B, int level, uint32_t g, u64 *out) {
    const int rows = c->qp_rows(level);
    Buf dg(&c->pool, (size_t)B * c->ndig(level) * rows * c->N);
    modup(c, ct + (long)(level + 1) * c->N, 2L * (level + 1) * c->N, B, level, dg.p);
    rotate_digits(c, ct, B, level, dg.p, g, out);
}

// Rescale (App. A): [B][2][l+1][N] -> [B][2][l][N], round(c / q_l).
void rescale(Ctx *c, const u64 *in, int B, int level, u64 *out) {
    const int N = c->N;
    if (level < 1) throw HeError(HE_ERR_LEVEL, "rescale at level 0");
    Buf last(&c->pool, (size_t)2 * B * N), t(&c->pool, (size_t)2 * B * level * N);
    RowMap one = RowMap::single(level);
    ntt_inv(c, last.p, 2L * B, one, c->stream, NttSrc{in + (long)level * N, (long)(level + 1) * N, 1});
    launch_rescale_prep(c, last.p, t.p, 2 * B, level, c->stream);
    if (c->logN >= 14 && c->logN <= 16) {
        // the NTT's last pass writes out = (in - t) q_l^-1 directly
        SubScale ep;
        ep.u = in, ep.us = (long)(level + 1) * N, ep.out = out, ep.os = (long)level * N, ep.w = c->lc(level).d_rs_inv, ep.wf = c->lc(level).d_rs_invf;
        ep.rows_per_item = level;
        ntt_fwd_subscale(c, t.p, 2L * B * level, c->map_q(level - 1), c->stream, ep);
    } else {
        ntt_fwd(c, t.p, 2L * B * level, c->map_q(level - 1), c->stream);
        launch_rescale_final(c, out, in, t.p, 2 * B, level, (long)(level + 1) * N, (long)level * N, c->stream);
    }
}

// ModDown then Rescale of items over Q_l P ([2 B][rows][N]) -> [B][2][l][N]:
// the words of moddown and rescale in a row, with one forward NTT of l rows per
// polynomial for the two (k_moddown_bconv, RS).
void moddown_rescale(Ctx *c, const u64 *u, int B, int level, u64 *out, u64 *const *outs) {
    const int N = c->N, rows = c->qp_rows(level), a1 = c->alpha + 1;
    if (level < 1) throw HeError(HE_ERR_LEVEL, "rescale at level 0");
    if (c->logN < 14 || c->logN > 16) {
        Buf t(&c->pool, (size_t)B * 2 * (level + 1) * N);
        moddown(c, u, 2 * B, level, t.p, (long)(level + 1) * N);
        if (!outs) rescale(c, t.p, B, level, out);
        else
            for (int b = 0; b < B; b++) rescale(c, t.p + (size_t)b * 2 * (level + 1) * N, 1, level, outs[b]);
        return;
    }
    Buf pc(&c->pool, (size_t)2 * B * a1 * N), z(&c->pool, (size_t)2 * B * level * N);
    ntt_inv(c, pc.p, 2L * B * a1, c->map_lp(level), c->stream, NttSrc{u + (long)level * N, (long)rows * N, a1});
    launch_moddown_rescale_bconv(c, pc.p, z.p, 2 * B, level, c->stream);
    SubScale ep;
    ep.u = u, ep.us = (long)rows * N, ep.out = out, ep.os = (long)level * N;
    ep.w = c->lc(level).d_mr_inv, ep.wf = c->lc(level).d_mr_invf, ep.rows_per_item = level;
    if (outs) {
        ep.n_out = B;
        for (int b = 0; b < B; b++) ep.outs[b] = outs[b];
    }
    ntt_fwd_subscale(c, z.p, 2L * B * level, c->map_q(level - 1), c->stream, ep);
}

// Level drop: keep limbs 0..to of both polys.
void drop(Ctx *c, const u64 *in, int B, int level, int to, u64 *out) {
    const int N = c->N;
    launch_copy_rows(out, (long)(to + 1) * N, in, (long)(level + 1) * N, 2 * B, (long)(to + 1) * N, c->stream);
}

// out (holding (d0, d1)) += KeySwitch(d2, rlk): the relinearisation of Mult.
// The ModDown's last store adds into out in place.
static void relin_into(Ctx *c, const u64 *d2, int B, int level, u64 *out) {
    if (!c->rlk) throw HeError(HE_ERR_KEY_MISSING, "relinearisation key missing");
    const int N = c->N, nq = level + 1, rows = c->qp_rows(level);
    Buf dg(&c->pool, (size_t)B * c->ndig(level) * rows * N);
    modup(c, d2, (long)nq * N, B, level, dg.p);
    Buf u(&c->pool, (size_t)B * 2 * rows * N);
    launch_multsum(c, u.p, dg.p, c->rlk, 1u, B, level, nullptr, 0, c->stream);
    c->n_ms += B;
    moddown(c, u.p, 2 * B, level, out, (long)nq * N, out, (long)nq * N);
    c->n_md += B;
}

// Mult (App. A): tensor (d0, d1, d2), then (d0, d1) + KeySwitch(d2, rlk).
void mult_relin(Ctx *c, const u64 *a, const u64 *b, int B, int level, u64 *out) {
    if (!c->rlk) throw HeError(HE_ERR_KEY_MISSING, "relinearisation key missing");
    const int N = c->N, nq = level + 1;
    Buf d2(&c->pool, (size_t)B * nq * N);
    launch_tensor(c, out, d2.p, a, b, B, nq, c->map_q(level), c->stream);
    relin_into(c, d2.p, B, level, out);
}

void add(Ctx *c, const u64 *a, const u64 *b, int B, int level, u64 *out) {
    launch_add(c, out, a, b, 2L * B * (level + 1), c->map_q(level), c->stream);
}

// --------------------------------------------------- plaintext diagonals
// Cached encodings (NTT, in the form their kernels take) over Q_l P of a diagonal slot vector at
// scale q_l.  kind/n/t/rot/value/k as in k_diag_fill.
const u64 *get_pt(Ctx *c, int kind, int n, long t, long rot, double value, int k, int level,
                  const DcdFactor *fac) {
    std::ostringstream os;
    os << kind << ':' << n << ':' << t << ':' << rot << ':' << k << ':' << level << ':';
    if (fac) os << fac->id << ':';
    os.precision(17);
    os << value;
    std::string key = os.str();
    auto it = c->ptcache.find(key);
    if (it != c->ptcache.end()) return it->second;
    const int N = c->N, rows = c->qp_rows(level);
    Buf zr(&c->pool, c->S), zi(&c->pool, c->S), m(&c->pool, N);
    u64 *pt = (u64 *)device_alloc(c, (size_t)rows * N * 8);
    if (!pt) throw HeError(HE_ERR_OOM, "plaintext cache allocation failed");
    if (fac)
        launch_dcd_fill(c, (double *)zr.p, fac->dev, n, t, rot, value, c->stream);
    else
        launch_diag_fill(c, (double *)zr.p, kind, n, t, rot, value, k, c->stream);
    cudaMemsetAsync(zi.p, 0, (size_t)c->S * 8, c->stream);
    launch_encode(c, (double *)zr.p, (double *)zi.p, (double)c->primes[level], (i64 *)m.p, c->stream);
    RowMap qp = c->map_qp(level);
    launch_small_to_rns(c, (const i64 *)m.p, pt, rows, qp, c->stream);
    ntt_fwd(c, pt, rows, qp, c->stream);
    // the PowerMethod's masks (kinds 6, 7, 10, 11) multiply by themselves, in
    // Montgomery form; diagonals and column masks enter sums
    if (kind == 6 || kind == 7 || kind == 10 || kind == 11) launch_to_mont(c, pt, pt, rows, qp, c->stream);
    else launch_key_form(c, pt, rows, qp, c->stream);
    c->ptcache[key] = pt;
    c->ptcache_bytes += (size_t)rows * N * 8;
    return pt;
}

// Does diagonal `t` of transform `kind` hold a non-zero entry?
static bool diag_nonzero(int kind, int n, long t) {
    switch (kind) {
    case 0: return t > -n && t < n;                         // Z, eq. 5
    case 1: return t >= 0 && t % n == 0 && t / n < n;       // T, eq. 6
    case 2: {                                                // G, (n-1) k
        long a = n - 1;
        if (a == 0) return t == 0;
        if (t % a != 0) return false;
        long kk = t / a;
        return kk > -n && kk < n;
    }
    }
    return false;
}

static long mod_pos(long x, long m) { return ((x % m) + m) % m; }

// Double-hoisted BSGS linear transform (eq. 3', Sec. 3.3):
//   U m = sum_i rho( sum_j rho(u_{a(n1 i + j)}; -a n1 i) . rho(m; a j) ; a n1 i ),
// babies kept in Q_l P from one Decompose; giant groups summed in Q_l P,
// ModDown'd, rotated (kept in Q_l P) and accumulated; one final ModDown and a
// rescale by q_l (plaintexts at scale q_l keep the ciphertext scale).
// in: [B][2][l+1][N]; out: [B][2][l][N].
//
// n1_sub > 0 (simple key substitution, Sec. 4.2): the babies use only the
// keys a s, 0 < s < n1_sub.  They come in groups of n1_sub - 1: the first
// rotates the input by a s; every later group takes the last baby of the
// previous one, ModDown'd to a ciphertext c and Decomposed, and rotates c by
// a s, so that baby j = b + s is rho(c; a s) with c = rho(m; a b).
static void lintrans_once(Ctx *c, const u64 *in, int B, int level, int kind, int n, long a, int n1, int gi0, int gi1,
                          double value, u64 *out, const DcdFactor *fac, int n1_sub) {
    const int N = c->N, nq = level + 1, rows = c->qp_rows(level);
    const long n2 = (long)n * n;
    const size_t qpct = (size_t)2 * rows * N;   // one item over Q_l P
    Buf dg(&c->pool, (size_t)B * c->ndig(level) * rows * N);
    modup(c, in + (long)nq * N, 2L * nq * N, B, level, dg.p);
    std::vector<Buf> R;
    R.emplace_back(&c->pool, B * qpct);
    launch_lift_P(c, R[0].p, in, 2 * B, level, (long)nq * N, (long)rows * N, c->stream);
    for (int j = 1; j < n1; j++) R.emplace_back(&c->pool, B * qpct);
    // Giants i != 0 go in groups of G: their sums, ModDowns, Decomposes and
    // rotations run as one batch of G B items, so that a few ciphertexts fill
    // the GPU (one giant of one ciphertext at N = 2^15 leaves most of it idle).
    // 16 items of N = 2^16 bound the digits' memory.
    std::vector<int> giants;
    std::vector<PmulTerm> terms;
    std::vector<int> first(1, 0);
    int i0 = -1;   // position of giant 0, which needs no rotation: it comes first
    auto add_giant = [&](int i) {
        const size_t n0 = terms.size();
        for (int j = 0; j < n1; j++) {
            long t = a * ((long)n1 * i + j);
            if (fac ? !fac->diags.count(mod_pos(t, n2)) : !diag_nonzero(kind, n, t)) continue;
            terms.push_back({get_pt(c, kind, n, t, mod_pos(-a * n1 * i, n2), value, 0, level, fac), j});
        }
        if (terms.size() == n0) return;
        giants.push_back(i);
        first.push_back((int)terms.size());
    };
    if (gi0 <= 0 && gi1 > 0) {
        add_giant(0);
        if (!giants.empty()) i0 = 0;
    }
    for (int i = gi0; i < gi1; i++)
        if (i) add_giant(i);
    const int ng = (int)giants.size(), nrot = ng - (i0 == 0 ? 1 : 0);
    const bool one = c->scratch == Ctx::kSingle;
    const int Gmax = std::min(nrot, one ? 1 : (int)std::max<long>(1, std::min<long>(kMaxGiants, (16L << 16) / ((long)B * N))));
    const size_t dgw = (size_t)B * c->ndig(level) * rows * N;
    Buf acc(&c->pool, B * qpct), ctmp(&c->pool, std::max(1, Gmax) * (size_t)B * 2 * nq * N),
        dg2(&c->pool, std::max(1, Gmax) * dgw);
    // the plaintext sums of up to 64 items of N = 2^16 at a time: more sums a launch
    // share more of its reads of R
    const int Smax = std::max(1, one ? 1 : std::min(nrot, (int)std::max<long>(Gmax, (64L << 16) / ((long)B * N))));
    Buf S(&c->pool, (size_t)Smax * B * qpct);
    const int head = n1_sub > 1 && n1_sub < n1 ? n1_sub : n1;
    for (int j0 = 1, base = 0; j0 < n1; j0 += head - 1) {
        const u64 *src = in, *sdg = dg.p;
        if (j0 > 1) {
            // the previous group's last baby as the next source
            base = j0 - 1;
            moddown(c, R[base].p, 2 * B, level, ctmp.p, (long)nq * N);
            c->n_md += B;
            modup(c, ctmp.p + (long)nq * N, 2L * nq * N, B, level, dg2.p);
            src = ctmp.p, sdg = dg2.p;
        }
        std::vector<uint32_t> gs;
        std::vector<u64 *> outs;
        for (int j = j0; j < std::min(n1, j0 + head - 1); j++) {
            gs.push_back(galois_of_step(c, mod_pos(a * (j - base), n2)));
            outs.push_back(R[j].p);
        }
        rot_qp_multi(c, src, B, level, sdg, gs.data(), (int)gs.size(), outs.data());
    }
    std::vector<const u64 *> Rp;
    for (auto &r : R) Rp.push_back(r.p);
    if (i0 == 0) launch_pmul_sums(c, acc.p, (long)(B * qpct), terms.data(), first.data(), 1, Rp.data(), n1, B, level, (long)qpct, c->stream);
    bool have = i0 == 0;
    for (int p0 = have ? 1 : 0, G, s0 = 0, s1 = 0; p0 < ng; p0 += G) {
        if (p0 >= s1) {
            s0 = p0, s1 = std::min(ng, p0 + Smax);
            launch_pmul_sums(c, S.p, (long)(B * qpct), terms.data(), first.data() + s0, s1 - s0, Rp.data(), n1, B, level,
                             (long)qpct, c->stream);
        }
        G = std::min(Gmax, s1 - p0);
        moddown(c, S.p + (size_t)(p0 - s0) * B * qpct, 2 * B * G, level, ctmp.p, (long)nq * N);
        c->n_md += (long long)B * G;
        modup(c, ctmp.p + (long)nq * N, 2L * nq * N, B * G, level, dg2.p);
        std::vector<const u64 *> keys;
        std::vector<uint32_t> gs;
        for (int t = 0; t < G; t++) {
            gs.push_back(galois_of_step(c, mod_pos(a * n1 * giants[p0 + t], n2)));
            keys.push_back(need_key(c, gs.back()));
        }
        launch_multsum_giants(c, acc.p, have ? acc.p : nullptr, dg2.p, keys.data(), gs.data(), G, B, level, ctmp.p,
                              2L * nq * N, c->stream);
        c->n_ms += (long long)B * G;
        have = true;
    }
    moddown_rescale(c, acc.p, B, level, out);
    c->n_md += B;
}

void lintrans(Ctx *c, const u64 *in, int B, int level, int kind, int n, long a, int n1, int gi0, int gi1,
              double value, u64 *out, const DcdFactor *fac, int n1_sub) {
    with_scratch(c, [&] { lintrans_once(c, in, B, level, kind, n, a, n1, gi0, gi1, value, out, fac, n1_sub); });
}

// The ModDown's last store adds into ct in place.
void rotate_add(Ctx *c, u64 *ct, int B, int level, uint32_t g) {
    const int rows = c->qp_rows(level);
    const size_t N = c->N;
    const long nq = level + 1;
    Buf dg(&c->pool, (size_t)B * c->ndig(level) * rows * N), u(&c->pool, (size_t)B * 2 * rows * N);
    modup(c, ct + nq * N, 2L * nq * N, B, level, dg.p);
    rot_qp(c, ct, B, level, dg.p, g, u.p);
    moddown(c, u.p, 2 * B, level, ct, nq * N, ct, nq * N);
    c->n_md += B;
}

// ct <- ct + Rot(ct, -n^2 2^j) for j = 0 .. log2(S/n^2)-1 (period n^2).
void replicate(Ctx *c, u64 *ct, int B, int level, int n) {
    const long n2 = (long)n * n;
    for (long s = n2; s < c->S; s *= 2) rotate_add(c, ct, B, level, galois_of_step(c, c->S - s));
}

// JKLS product (eq. 4) with the hoisting of Sec. 4.1; A, B: [Bn][2][l+1][N]
// replicated with period n^2; out: [Bn][2][l-2][N].
// A chain of decomposition factors (application order) on B items at
// `level`; the output, one level per factor lower, goes to out.
static void apply_chain(Ctx *c, const u64 *in, int B, int level, const DcdChain &ch, int n, long a_left, int n1,
                        int gi0, int gi1, u64 *out) {
    const size_t w = (size_t)2 * (level + 1) * c->N;
    Buf t0(&c->pool, B * w), t1(&c->pool, B * w);
    const u64 *cur = in;
    int lv = level;
    for (size_t f = 0; f + 1 < ch.factors.size(); f++) {
        u64 *dst = (f % 2 == 0) ? t0.p : t1.p;
        lintrans(c, cur, B, lv, 8, n, ch.factors[f].step, 2, 0, 1, 1.0, dst, &ch.factors[f]);
        cur = dst;
        lv--;
    }
    lintrans(c, cur, B, lv, 8, n, a_left, n1, gi0, gi1, 1.0, out, &ch.factors.back());
}

// sigma (Z) or tau (T) of B items at `level`, undecomposed (one level) or
// through the decomposition chains (Sec. 4.2 DMatrixMult), then dropped to
// level `to`.
static void zt_stage(Ctx *c, const u64 *in, int B, int level, bool is_t, int n, int n1, int np, int to, u64 *out) {
    const int N = c->N;
    const int m = dcd_levels(n, np, is_t), lo = level - m;
    const size_t wlo = (size_t)2 * (lo + 1) * N;
    Buf r(&c->pool, lo == to ? 1 : B * wlo);
    u64 *dst = lo == to ? out : r.p;   // no copy when no level has to be dropped
    if (!np) {
        if (is_t) lintrans(c, in, B, level, 1, n, n, n1, 0, n / n1, 1.0, dst);
        else lintrans(c, in, B, level, 0, n, 1, n1, -(n / n1), n / n1, 1.0, dst);
    } else if (is_t) {
        apply_chain(c, in, B, level, dcd_chain(c, 2, n, np), n, n, n1, 0, np / n1 + 1, dst);
    } else {
        Buf r2(&c->pool, B * wlo);
        apply_chain(c, in, B, level, dcd_chain(c, 0, n, np), n, 1, n1, 0, np / n1, dst);
        apply_chain(c, in, B, level, dcd_chain(c, 1, n, np), n, 1, n1, -(np / n1), 1, r2.p);
        add(c, dst, r2.p, B, lo, dst);
    }
    if (lo != to) drop(c, r.p, B, lo, to, out);
}

void zt_stage_public(Ctx *c, const u64 *in, int B, int level, bool is_t, int n, int n1, int np, int to, u64 *out) {
    zt_stage(c, in, B, level, is_t, n, n1, np, to, out);
}

// Products A[ia[p]] B[ib[p]], p < P, of nA distinct left and nB distinct
// right operands: sigma, C^k and their hoisted rotations run once per left
// operand, tau and R^k once per right operand, whatever the number of
// products each takes part in (Sec. 5.2, covariance Optimizations 1 and 2:
// C^k Z X_j^T and R^k T X_i computed once for every product that uses
// them; the batch of products is the row segment).  Only the current k's
// A^(k), B^(k) are held, so the memory grows with nA + nB + P, not with n.
static void hmatmul_once(Ctx *c, const u64 *A, int nA, const u64 *Bm, int nB, const int *ia, const int *ib, int P,
                         int level, int n, int n1z, int n1t, u64 *out, bool relin_once, int dcd_z, int dcd_t) {
    const int depth = hmatmul_depth(n, dcd_z, dcd_t);
    if (level < depth) throw HeError(HE_ERR_LEVEL, "matrix product needs more levels");
    if ((dcd_z && (dcd_z >= n || dcd_z % n1z)) || (dcd_t && (dcd_t >= n || dcd_t % n1t)))
        throw HeError(HE_ERR_ARG, "a decomposition needs n' < n with n1 dividing n'");
    if (!c->rlk) throw HeError(HE_ERR_KEY_MISSING, "relinearisation key missing");
    const int N = c->N;
    const long n2m = (long)n * n;
    const int l1 = level - (depth - 2), l2 = l1 - 1;
    const size_t ct1 = (size_t)2 * (l1 + 1) * N, ct2 = (size_t)2 * (l2 + 1) * N;
    const int rows1 = c->qp_rows(l1);
    const size_t qp1 = (size_t)2 * rows1 * N, dig1 = (size_t)c->ndig(l1) * rows1 * N;
    for (int p = 0; p < P; p++)
        if (ia[p] < 0 || ia[p] >= nA || ib[p] < 0 || ib[p] >= nB) throw HeError(HE_ERR_ARG, "bad operand index");
    Buf A0(&c->pool, nA * ct1), B0(&c->pool, nB * ct1);
    zt_stage(c, A, nA, level, false, n, n1z, dcd_z, l1, A0.p);
    zt_stage(c, Bm, nB, level, true, n, n1t, dcd_t, l1, B0.p);

    // C^k sources A_g, A'_g and R^k sources B_g with their digits
    Buf Ag(&c->pool, nA * ct1), Apg(&c->pool, nA * ct1), Bg(&c->pool, nB * ct1);
    Buf dA(&c->pool, nA * dig1), dAp(&c->pool, nA * dig1), dB(&c->pool, nB * dig1);
    Buf tmpA(&c->pool, nA * ct1), tmpB(&c->pool, nB * ct1);
    cudaMemcpyAsync(Ag.p, A0.p, nA * ct1 * 8, cudaMemcpyDeviceToDevice, c->stream);
    modup(c, Ag.p + (long)(l1 + 1) * N, (long)ct1, nA, l1, dA.p);
    rotate_digits(c, Ag.p, nA, l1, dA.p, galois_of_step(c, mod_pos(-n, n2m)), Apg.p);
    modup(c, Apg.p + (long)(l1 + 1) * N, (long)ct1, nA, l1, dAp.p);
    cudaMemcpyAsync(Bg.p, B0.p, nB * ct1 * 8, cudaMemcpyDeviceToDevice, c->stream);
    modup(c, Bg.p + (long)(l1 + 1) * N, (long)ct1, nB, l1, dB.p);
    int gA = 0;

    // Terms k run by run: kn consecutive k of one A giant and one B giant, all
    // their ModDowns, rescales, tensors and key switches in one set of launches
    // (SA, BB: slot b of a giant's baby b, slot 0 the giant itself).  A run holds
    // kn P items; the bound keeps its temporaries in proportion to the batch's
    // (64 items of N = 2^16 fill the GPU many times over).
    const int nbA = n1z - 1, nbB = n1t - 1;
    const int kmax =
        c->scratch == Ctx::kSingle
            ? 1
            : (int)std::max<long>(1, std::min<long>(n, (64L << 16) / ((long)std::max(P, std::max(nA, nB)) * N)));
    const bool summed = c->logN >= 14 && c->logN <= 16;   // the register-blocked NTT's row layouts
    Buf SA(&c->pool, (size_t)n1z * nA * qp1), BB(&c->pool, (size_t)n1t * nB * ct1);
    Buf Ak(&c->pool, (size_t)std::min(kmax, n1z) * nA * ct2);
    Buf acc(&c->pool, P * ct2), D2(&c->pool, (size_t)P * (l2 + 1) * N);
    Buf d2(&c->pool, relin_once ? 1 : (size_t)std::min(kmax, n1z) * P * (l2 + 1) * N);
    std::unique_ptr<RelinSum> sum;
    if (!relin_once && summed) sum.reset(new RelinSum(c, P, l2));
    // the giant's own sources, lifted to Q_l P, masked and summed (slot 0)
    auto giant_A = [&]() {
        const int k = n1z * gA;
        if (k) {
            Buf R1(&c->pool, nA * qp1), R2(&c->pool, nA * qp1);
            launch_lift_P(c, R1.p, Ag.p, 2 * nA, l1, (long)(l1 + 1) * N, (long)rows1 * N, c->stream);
            launch_lift_P(c, R2.p, Apg.p, 2 * nA, l1, (long)(l1 + 1) * N, (long)rows1 * N, c->stream);
            const u64 *pts[2] = {get_pt(c, 3, n, 0, 0, 1.0, k, l1), get_pt(c, 4, n, 0, 0, 1.0, k, l1)};
            const u64 *Rs[2] = {R1.p, R2.p};
            const PmulTerm two[2] = {{pts[0], 0}, {pts[1], 1}};
            const int range[2] = {0, 2};
            launch_pmul_sums(c, SA.p, 0, two, range, 1, Rs, 2, nA, l1, (long)qp1, c->stream);
        }
        if (nbA <= 0) return;
        // the babies, masked and summed in one pass:
        // SA_b = m_k (.) rot_qp(A_g; b) + m'_k (.) rot_qp(A'_g; b), k = n1z g + b
        std::vector<uint32_t> gs;
        std::vector<u64 *> o;
        std::vector<const u64 *> m1, m2, keys;
        for (int b = 1; b <= nbA; b++) {
            gs.push_back(galois_of_step(c, b % n2m));
            o.push_back(SA.p + (size_t)b * nA * qp1);
            m1.push_back(get_pt(c, 3, n, 0, 0, 1.0, k + b, l1));
            m2.push_back(get_pt(c, 4, n, 0, 0, 1.0, k + b, l1));
            keys.push_back(need_key(c, gs.back()));
        }
        launch_multsum_ck(c, o.data(), dA.p, dAp.p, keys.data(), gs.data(), m1.data(), m2.data(), nbA, nA, l1,
                          Ag.p, Apg.p, (long)ct1, c->stream);
        c->n_ms += 2LL * nA * nbA;
    };
    // B_g in slot 0, its hoisted rotations by n b (ModDown'd) in the others
    auto giant_B = [&]() {
        cudaMemcpyAsync(BB.p, Bg.p, nB * ct1 * 8, cudaMemcpyDeviceToDevice, c->stream);
        if (nbB <= 0) return;
        Buf UB(&c->pool, (size_t)nbB * nB * qp1);
        std::vector<uint32_t> gs;
        std::vector<u64 *> o;
        for (int b = 1; b <= nbB; b++) {
            gs.push_back(galois_of_step(c, ((long)n * b) % n2m));
            o.push_back(UB.p + (size_t)(b - 1) * nB * qp1);
        }
        rot_qp_multi(c, Bg.p, nB, l1, dB.p, gs.data(), nbB, o.data());
        moddown(c, UB.p, 2 * nB * nbB, l1, BB.p + nB * ct1, (long)(l1 + 1) * N);
        c->n_md += (long long)nB * nbB;
    };
    giant_A();
    giant_B();
    for (int k = 0, kn; k < n; k += kn) {
        const int b = k % n1z, bb = k % n1t;
        kn = std::min(std::min(kmax, n - k), std::min(n1z - b, n1t - bb));
        if (k && b == 0) {
            rotate_digits(c, Ag.p, nA, l1, dA.p, galois_of_step(c, n1z % n2m), tmpA.p);
            std::swap(Ag, tmpA);
            modup(c, Ag.p + (long)(l1 + 1) * N, (long)ct1, nA, l1, dA.p);
            rotate_digits(c, Apg.p, nA, l1, dAp.p, galois_of_step(c, n1z % n2m), tmpA.p);
            std::swap(Apg, tmpA);
            modup(c, Apg.p + (long)(l1 + 1) * N, (long)ct1, nA, l1, dAp.p);
            gA++;
            giant_A();
        }
        if (k && bb == 0) {
            rotate_digits(c, Bg.p, nB, l1, dB.p, galois_of_step(c, ((long)n * n1t) % n2m), tmpB.p);
            std::swap(Bg, tmpB);
            modup(c, Bg.p + (long)(l1 + 1) * N, (long)ct1, nB, l1, dB.p);
            giant_B();
        }
        // ---- A^(k) = C^k A^(0) at level l2
        const int k0 = k == 0 ? 1 : 0;   // A^(0) is A0 itself
        if (k0) drop(c, A0.p, nA, l1, l2, Ak.p);
        if (kn > k0) {
            moddown_rescale(c, SA.p + (size_t)(b + k0) * nA * qp1, (kn - k0) * nA, l1, Ak.p + (size_t)k0 * nA * ct2);
            c->n_md += (long long)(kn - k0) * nA;
        }
        // ---- products with B^(k) = R^k B^(0) (at level l1: the tensor reads its
        // first l2 + 1 limbs), relinearised and accumulated at level l2
        launch_tensor_run(c, acc.p, D2.p, relin_once ? nullptr : d2.p, Ak.p, BB.p + (size_t)bb * nB * ct1, kn, P, nA, nB, ia,
                          ib, l2 + 1, (long)ct1, (long)(l1 + 1) * N, k > 0);
        if (relin_once) continue;
        if (summed) relin_sum_run(c, *sum, d2.p, kn);
        else
            for (int t = 0; t < kn; t++) relin_into(c, d2.p + (size_t)t * P * (l2 + 1) * N, P, l2, acc.p);
    }
    if (relin_once) relin_into(c, D2.p, P, l2, acc.p);
    else if (summed) relin_sum_finish(c, *sum, D2.p, acc.p);
    rescale(c, acc.p, P, l2, out);
}

void hmatmul_pairs(Ctx *c, const u64 *A, int nA, const u64 *Bm, int nB, const int *ia, const int *ib, int P,
                   int level, int n, int n1z, int n1t, u64 *out, bool relin_once, int dcd_z, int dcd_t) {
    with_scratch(c, [&] {
        hmatmul_once(c, A, nA, Bm, nB, ia, ib, P, level, n, n1z, n1t, out, relin_once, dcd_z, dcd_t);
    });
}

void hmatmul(Ctx *c, const u64 *A, const u64 *Bm, int Bn, int level, int n, int n1z, int n1t, u64 *out,
             bool relin_once, int dcd_z, int dcd_t) {
    std::vector<int> id(Bn);
    for (int i = 0; i < Bn; i++) id[i] = i;
    hmatmul_pairs(c, A, Bn, Bm, Bn, id.data(), id.data(), Bn, level, n, n1z, n1t, out, relin_once, dcd_z, dcd_t);
}

}  // namespace he

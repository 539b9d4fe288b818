// eval.h -- batched evaluation routines (see eval.cu).
#pragma once
#include <stdexcept>

#include "he_internal.h"

namespace he {

// Runs f, a routine whose groups and runs of many items only make it faster
// (its words do not depend on their size), and where their scratch does not fit
// the device runs it again with groups and runs of one, which take no more than
// a loop over the items.  f reads its inputs and writes its output last, so it
// may be run again; the operation counters are those of one run.
struct ScratchMode {
    Ctx *c;
    const Ctx::Scratch keep;
    ScratchMode(Ctx *cc, Ctx::Scratch m) : c(cc), keep(cc->scratch) { c->scratch = m; }
    ~ScratchMode() { c->scratch = keep; }
};
template <class F>
void with_scratch(Ctx *c, F f) {
    if (c->scratch != Ctx::kAdapt) return f();
    const long long ms = c->n_ms, dp = c->n_dp, md = c->n_md;
    try {
        return f();
    } catch (const std::bad_alloc &) {
    } catch (const HeError &e) {
        if (e.code != HE_ERR_OOM) throw;
    }
    c->n_ms = ms, c->n_dp = dp, c->n_md = md;
    ScratchMode single(c, Ctx::kSingle);
    f();
}

uint32_t galois_of_step(const Ctx *c, long step);
void create_keys(Ctx *c);
u64 *gen_rotation_key(Ctx *c, uint32_t g);
u64 *gen_relin_key(Ctx *c);
void encrypt_poly(Ctx *c, const u64 *m_ntt, int level, uint32_t obj, bool refresh, u64 *out);
void encode_to(Ctx *c, const double *d_zr, const double *d_zi, double scale, u64 *out, int rows, const RowMap &rm);
const char *last_error();
double bfly_peak(int iters);
double mac_peak(int iters);

void modup(Ctx *c, const u64 *poly, long item_s, int B, int level, u64 *digits);
// add (may be null, item stride add_s; may equal out): out = add + ModDown(u)
void moddown(Ctx *c, const u64 *u, int items, int level, u64 *out, long out_s, const u64 *add = nullptr,
             long add_s = 0);
void rot_qp(Ctx *c, const u64 *ct, int B, int level, const u64 *digits, uint32_t g, u64 *out);
void rot_qp_multi(Ctx *c, const u64 *ct, int B, int level, const u64 *digits, const uint32_t *gs, int G,
                  u64 *const *outs);
void rotate_digits(Ctx *c, const u64 *ct, int B, int level, const u64 *digits, uint32_t g, u64 *out);
void rotate(Ctx *c, const u64 *ct, int B, int level, uint32_t g, u64 *out);
void rescale(Ctx *c, const u64 *in, int B, int level, u64 *out);
// out: [B][2][l][N], or outs[b] for each of at most 8 items
void moddown_rescale(Ctx *c, const u64 *u, int B, int level, u64 *out, u64 *const *outs = nullptr);
constexpr int kMultMany = 8;
void mult_rescale_many(Ctx *c, const u64 *const *a, const int *a_level, const u64 *const *b, const int *b_level, int n,
                       int level, u64 *const *out);
// ct [B][2][l+1][N] += Rot(ct; g)
void rotate_add(Ctx *c, u64 *ct, int B, int level, uint32_t g);
void drop(Ctx *c, const u64 *in, int B, int level, int to, u64 *out);
void mult_relin(Ctx *c, const u64 *a, const u64 *b, int B, int level, u64 *out);
// Sum of at most kRelinTerms relinearised terms (relin.cu): the integers of the
// runs so far.
constexpr int kRelinTerms = 256;
struct RelinSum {
    int P, level, terms = 0;
    Buf SY, YP;
    RelinSum(Ctx *c, int P, int level);
};
void relin_sum_run(Ctx *c, RelinSum &S, u64 *d2, int K);
void relin_sum_finish(Ctx *c, RelinSum &S, const u64 *D2, u64 *out);
void launch_tensor_run(Ctx *c, u64 *d01, u64 *D2, u64 *d2, const u64 *a, const u64 *b, int K, int P, int nA, int nB,
                       const int *ia, const int *ib, int limbs, long bs, long bp, bool accumulate);
void add(Ctx *c, const u64 *a, const u64 *b, int B, int level, u64 *out);
const u64 *get_pt(Ctx *c, int kind, int n, long t, long rot, double value, int k, int level,
                  const DcdFactor *fac = nullptr);
void lintrans(Ctx *c, const u64 *in, int B, int level, int kind, int n, long a, int n1, int gi0, int gi1,
              double value, u64 *out, const DcdFactor *fac = nullptr, int n1_sub = 0);
// Decompositions (dcd.cu): which = 0 (Z_1), 1 (Z_2), 2 (T); levels a chain consumes.
const DcdChain &dcd_chain(Ctx *c, int which, int n, int n_prime);
// Factors (levels) of the decomposed Z (is_t false) or T; 1 without n'.
int dcd_levels(int n, int n_prime, bool is_t);
void launch_dcd_fill(Ctx *c, double *out, const int *diag, int n, long t, long rot, double value, cudaStream_t st);
// Levels a product consumes: the Z/T stage (1, or the longer decomposition
// chain), C^k, and the multiplication.
// sigma (is_t false) or tau of B items through the undecomposed transform or
// the decomposition chains, output dropped to level `to`.
void zt_stage_public(Ctx *c, const u64 *in, int B, int level, bool is_t, int n, int n1, int np, int to, u64 *out);
inline int hmatmul_depth(int n, int dcd_z, int dcd_t) {
    int mz = dcd_levels(n, dcd_z, false), mt = dcd_levels(n, dcd_t, true);
    return (mz > mt ? mz : mt) + 2;
}
void replicate(Ctx *c, u64 *ct, int B, int level, int n);
void hmatmul(Ctx *c, const u64 *A, const u64 *Bm, int Bn, int level, int n, int n1z, int n1t, u64 *out,
             bool relin_once = false, int dcd_z = 0, int dcd_t = 0);
// products A[ia[p]] B[ib[p]] of shared operands (each operand's transforms once)
void hmatmul_pairs(Ctx *c, const u64 *A, int nA, const u64 *Bm, int nB, const int *ia, const int *ib, int P,
                   int level, int n, int n1z, int n1t, u64 *out, bool relin_once = false, int dcd_z = 0,
                   int dcd_t = 0);

}  // namespace he

"""The key switch's inner product (k_msum): every split of a launch over items,
keys and coefficients, ragged numbers of both, sums long enough to be folded
several times, and special primes in the float-quotient range, word for word
against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _open(qb, pb, seed, logN=14):
    import paper_2305_17341_gb300 as pk
    from oracle.ckks import CKKS, Params
    pk.build()
    P = Params(logN, qb, pb)
    return pk, pk.he_ctx_create(pk.make_params(logN, qb, pb), seed), P, CKKS(P, seed)


# 26 digits of one prime (folded at 11 and 22), 41-bit primes above the
# float-quotient range, a special prime inside it
CHAINS = [([60] + [40] * 25, [60]), ([60, 40, 41, 36, 40], [39]), ([60, 40, 40, 50, 41, 40, 40], [60, 39])]


@pytest.mark.parametrize("chain", range(len(CHAINS)))
def test_rotations_in_every_split(chain):
    qb, pb = CHAINS[chain]
    pk, ctx, P, he = _open(qb, pb, 11)
    try:
        steps = [1, 3, 64, -5, 17, 100, 2]
        pk.he_keygen(ctx, steps, False)
        for s in steps:
            he.gen_rotation_key(s)
        rng = np.random.default_rng(chain)
        level = P.L
        # residues at the edges of their range in the NTT domain's sums: the
        # largest values everywhere for one ciphertext, uniform for the others
        cts, want = [], []
        for i in range(5):
            r = np.stack([[rng.integers(0, q, P.N, dtype=np.uint64) if i else np.full(P.N, q - 1, dtype=np.uint64)
                           for q in P.qs(level)] for _ in range(2)])
            cts.append(pk.he_ct_import(ctx, r, level, float(2 ** 40), P.S))
        z = rng.uniform(-1, 1, P.S)
        o = he.encrypt_slots(z, level, obj=3)
        g = pk.he_encrypt_slots(ctx, z, level, 3)
        for s in steps[:3]:
            h = pk.he_rotate(ctx, g, s)
            w = he.rotate(o, s)
            assert np.array_equal(pk.he_ct_export(ctx, h), np.stack([w.c0, w.c1])), s
            pk.he_ct_free(h)
        for c in cts:
            want.append([])
            for s in steps:
                h = pk.he_rotate(ctx, c, s)
                want[-1].append(pk.he_ct_export(ctx, h))
                pk.he_ct_free(h)
        for B, G in ((1, 7), (2, 3), (5, 7), (3, 1), (5, 2)):
            for v in (0, 1, 2, 3, 4, 5, 6, 7, 8, 9):
                pk.he_ctx_set_multsum_variant(ctx, v)
                got = pk.he_rotate_hoisted(ctx, cts[:B], steps[:G])
                for b in range(B):
                    for k in range(G):
                        assert np.array_equal(pk.he_ct_export(ctx, got[b][k]), want[b][k]), (B, G, v, b, k)
                        pk.he_ct_free(got[b][k])
        for h in cts + [g]:
            pk.he_ct_free(h)
    finally:
        pk.he_ctx_destroy(ctx)


def test_product_with_a_narrow_special_prime():
    """The relinearisation's P rows in the float-quotient form."""
    from oracle.hmm import HMM, matmul_rot_steps
    pk, ctx, P, he = _open([60, 40, 40, 40, 40], [39], 12)
    try:
        n, n1 = 4, 2
        steps = matmul_rot_steps(n, n1, n1, P.S)
        pk.he_keygen(ctx, steps, True)
        for s in steps:
            he.gen_rotation_key(s)
        he.gen_relin_key()
        rng = np.random.default_rng(1)
        A, B = rng.uniform(-1, 1, (2, n * n))
        za, zb = np.zeros(P.S), np.zeros(P.S)
        za[:n * n], zb[:n * n] = A, B
        ga = pk.he_encrypt_matrix(ctx, A.reshape(n, n), P.L, 1)
        gb = pk.he_encrypt_matrix(ctx, B.reshape(n, n), P.L, 2)
        w = HMM(he).hmatmul(he.encrypt_slots(za, P.L, obj=1), he.encrypt_slots(zb, P.L, obj=2), n, n1, n1)
        h = pk.he_hmatmul(ctx, ga, gb, n, n1, n1)
        assert np.array_equal(pk.he_ct_export(ctx, h), np.stack([w.c0, w.c1]))
        for x in (ga, gb, h):
            pk.he_ct_free(x)
    finally:
        pk.he_ctx_destroy(ctx)

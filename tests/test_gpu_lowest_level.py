"""Products whose relinearisation lies at a level of a single digit.

There (l2 + 1 <= alpha) every row of the summed digits is the digit's own and
the forward transform of that launch has nothing to do; the kernels after it
must still wait for the ones before it.  Single, batched and planned products,
repeated, word for word against the oracle; and a key switch whose transforms
are launched in chunks of a digit's own rows only."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LOGN, N_MAT, N1, ITEMS = 14, 8, 2, 24


def res(ct):
    return np.stack([ct.c0, ct.c1])


@pytest.mark.parametrize("alpha,levels", [(2, (3,)), (3, (3, 4)), (4, (3, 4, 5))])
def test_product_at_a_level_of_one_digit(alpha, levels):
    import paper_2305_17341_gb300 as pk
    from oracle.ckks import CKKS, Params
    from oracle.hmm import HMM, matmul_rot_steps
    pk.build()
    qb, pb = [60] + [40] * 5, [60] * alpha
    P = Params(LOGN, qb, pb)
    ctx = pk.he_ctx_create(pk.make_params(LOGN, qb, pb), 30 + alpha)
    he = CKKS(P, 30 + alpha)
    n = N_MAT
    try:
        steps = matmul_rot_steps(n, N1, N1, P.S)
        pk.he_keygen(ctx, steps, want_relin=True)
        for s in steps:
            he.gen_rotation_key(s)
        he.gen_relin_key()
        rng = np.random.default_rng(alpha)
        for level in levels:
            assert level - 2 + 1 <= alpha
            mats = rng.uniform(-1, 1, (ITEMS, 2, n, n))
            cts = [tuple(pk.he_encrypt_matrix(ctx, mats[i, t], level, 2 * i + t) for t in (0, 1)) for i in range(ITEMS)]
            single = []
            for a, b in cts:
                h = pk.he_hmatmul(ctx, a, b, n, N1, N1)
                single.append(pk.he_ct_export(ctx, h))
                pk.he_ct_free(h)
            for i in (0, ITEMS - 1):
                z = np.zeros((2, P.S))
                z[:, :n * n] = mats[i].reshape(2, n * n)
                want = HMM(he).hmatmul(he.encrypt_slots(z[0], level, obj=2 * i),
                                       he.encrypt_slots(z[1], level, obj=2 * i + 1), n, N1, N1)
                assert np.array_equal(single[i], res(want)), (level, i)
            jobs = [(a, b, n, N1, N1) for a, b in cts]
            plan = pk.he_mm_plan_create(jobs)
            try:
                for rep in range(3):
                    for how, outs in (("batch", pk.he_hmatmul_batch(jobs)), ("plan", pk.he_mm_plan_run(plan))):
                        for i, h in enumerate(outs):
                            assert np.array_equal(pk.he_ct_export(ctx, h), single[i]), (level, how, rep, i)
                            pk.he_ct_free(h)
            finally:
                pk.he_mm_plan_destroy(plan)
            # chunks of the transforms that hold a digit's own rows only
            pk.he_ctx_set_ntt_chunk(ctx, alpha)
            try:
                h = pk.he_hmatmul(ctx, cts[0][0], cts[0][1], n, N1, N1)
            finally:
                pk.he_ctx_set_ntt_chunk(ctx, 0)
            assert np.array_equal(pk.he_ct_export(ctx, h), single[0]), level
            pk.he_ct_free(h)
            for c in cts:
                for h in c:
                    pk.he_ct_free(h)
    finally:
        pk.he_ctx_destroy(ctx)

"""Every build that a launch may take gives the same words: the NTT passes
compiled for 2, 3 and 4 CTAs per SM, and every split of the inner products'
warps, of the plain kernel and of the one with the C^k masks.

A product runs all of them (Decompose with its skipped rows, the fused ModDown
and rescale epilogues, hoisted rotations, masked babies, the relinearisation),
one item, and several with a ragged last group."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NTT_BUILDS = (2, 3, 5)
# the launches of a product have at most ten splits: pins 0..9 reach each
SPLITS = range(10)


@pytest.mark.parametrize("logN", [14, 16])
def test_products_in_every_build(logN):
    import paper_2305_17341_gb300 as pk
    pk.build()
    n, n1, level = 16, 8, 5
    ctx = pk.he_ctx_create(pk.make_params(logN, [60] + [40] * 5, [60, 60]), 23)
    try:
        pk.he_ctx_set_autotune(ctx, False)
        pk.he_keygen(ctx, pk.he_rot_steps_for_matmul(n, n1, n1, 1 << (logN - 1)), want_relin=True)
        mats = np.random.default_rng(logN).uniform(-1, 1, (3, 2, n, n))
        cts = [tuple(pk.he_encrypt_matrix(ctx, m, level, 2 * i + t) for t, m in enumerate(p)) for i, p in enumerate(mats)]
        jobs = [(a, b, n, n1, n1) for a, b in cts]

        def words(js):
            outs = pk.he_hmatmul_batch(js)
            r = [pk.he_ct_export(ctx, h) for h in outs]
            for h in outs:
                pk.he_ct_free(h)
            return r

        want = words(jobs)
        h = pk.he_hmatmul(ctx, *cts[0], n, n1, n1)
        assert np.abs(pk.he_decrypt_matrix(ctx, h, n, n) - mats[0][0] @ mats[0][1]).max() < 1e-4
        pk.he_ct_free(h)

        def check(what):
            for js in (jobs[:1], jobs):
                for i, w in enumerate(words(js)):
                    assert np.array_equal(w, want[i]), (what, len(js), i)

        for v in NTT_BUILDS:
            pk.he_ctx_set_ntt_variant(ctx, v)
            check(("ntt", v))
        pk.he_ctx_set_ntt_variant(ctx, -1)
        for v in SPLITS:
            pk.he_ctx_set_multsum_variant(ctx, v)
            check(("split", v))
        pk.he_ctx_set_multsum_variant(ctx, -1)
        for p in cts:
            for h in p:
                pk.he_ct_free(h)
    finally:
        pk.he_ctx_destroy(ctx)

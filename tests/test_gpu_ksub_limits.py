"""The key-substituted transform takes at most 32 babies: its plaintext sums
hold 32 rotations.  More are refused before anything is launched, with the
code of every other schedule check, and the context stays usable."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_more_babies_than_a_sum_holds_are_refused():
    import paper_2305_17341_gb300 as pk
    from oracle.ckks import CKKS, Params
    from oracle.hmm import HMM
    pk.build()
    n = n1 = 64
    P = Params(14, [60, 40, 40, 40], [60])
    ctx = pk.he_ctx_create(pk.he_params_default(1), 5)
    he = CKKS(P, 5)
    try:
        steps = set(pk.he_rot_steps_for_ksub(32, 0, 32, 32, P.S)) | set(pk.he_rot_steps_for_ksub(n, 0, n1, 2, P.S))
        pk.he_keygen(ctx, sorted(steps), want_relin=False)
        A = np.random.default_rng(1).uniform(-1, 1, (32, 32))
        a = pk.he_encrypt_matrix(ctx, A, P.L, 3)
        for kind in (0, 1):
            for head in (2, n1):
                with pytest.raises(pk.HeError) as e:
                    pk.he_linear_transform_ksub(ctx, a, kind, n, n1, head)
                assert e.value.code == pk.HE_ERR_ARG
        # the largest number that is taken, against the oracle
        for s in pk.he_rot_steps_for_ksub(32, 0, 32, 32, P.S):
            he.gen_rotation_key(s)
        z = np.zeros(P.S)
        z[:1024] = A.ravel()
        H = HMM(he)
        want = H.sigma(H.replicate(he.encrypt_slots(z, P.L, obj=3), 32), 32, 32, 32)
        got = pk.he_linear_transform_ksub(ctx, a, 0, 32, 32, 32)
        assert np.array_equal(pk.he_ct_export(ctx, got), np.stack([want.c0, want.c1]))
        pk.he_ct_free(got)
        pk.he_ct_free(a)
    finally:
        pk.he_ctx_destroy(ctx)

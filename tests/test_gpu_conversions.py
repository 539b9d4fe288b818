"""Basis conversions, the fused ModDown + Rescale and the summed key switch of
a product's relinearisations on chains that mix every kind of limb (40-bit,
just above and below the narrow and float-quotient bounds, 50 and 60 bits) with
one to four special primes, word for word against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# q_1.. on both sides of 2^41 (the narrow source bound), 2^36 and 2^40; q_l wide
# (50, 60 bits) at some levels, so that the rescale divides by a wide prime
CHAINS = {
    1: ([60, 41, 41, 36, 40, 50], [60]),
    2: ([60, 40, 50, 41, 40, 41, 36], [60, 50]),
    3: ([60, 40, 40, 36, 41, 50, 40], [60, 59, 45]),
    4: ([60, 50, 41, 41, 40, 40, 36, 38, 60], [60, 60, 58, 44]),
}


def _open(alpha, logN=14):
    import paper_2305_17341_gb300 as pk
    from oracle.ckks import CKKS, Params
    pk.build()
    qb, pb = CHAINS[alpha]
    P = Params(logN, qb, pb)
    return pk, pk.he_ctx_create(pk.make_params(logN, qb, pb), 9), P, CKKS(P, 9)


@pytest.mark.parametrize("alpha", [1, 2, 3, 4])
def test_conversions_on_mixed_limbs(alpha):
    import torch
    pk, ctx, P, he = _open(alpha)

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(a).view(np.int64).copy()).cuda()

    try:
        rng = np.random.default_rng(alpha)
        for level in (P.L, P.L - 1, 1, 0):
            nq, rows, nd = level + 1, level + 1 + P.alpha, P.ndigits(level)
            c = np.stack([rng.integers(0, q, P.N, dtype=np.uint64) for q in P.qs(level)])
            c[:, :3], c[:, 3:6] = 0, np.array([[q - 1] for q in P.qs(level)], dtype=np.uint64)
            d = dev(c)
            pk.he_ntt(ctx, d.data_ptr(), nq, level)
            dig = torch.empty((nd, rows, P.N), dtype=torch.int64, device="cuda")
            torch.cuda.synchronize()
            pk.he_decompose(ctx, d.data_ptr(), 1, level, dig.data_ptr())
            for k in range(nd):
                pk.he_ntt(ctx, dig[k].data_ptr(), rows, level, inverse=True)
            got = dig.cpu().numpy().view(np.uint64)
            for k, want in enumerate(he.modup(c, level)):
                assert np.array_equal(got[k], want), (level, k)
            u = np.stack([rng.integers(0, q, P.N, dtype=np.uint64) for q in P.qp(level)])
            u[:, :3], u[:, 3:6] = 0, np.array([[q - 1] for q in P.qp(level)], dtype=np.uint64)
            d = dev(u)
            pk.he_ntt(ctx, d.data_ptr(), rows, level)
            out = torch.empty((nq, P.N), dtype=torch.int64, device="cuda")
            torch.cuda.synchronize()
            pk.he_moddown(ctx, d.data_ptr(), 1, level, out.data_ptr())
            pk.he_ntt(ctx, out.data_ptr(), nq, level, inverse=True)
            assert np.array_equal(out.cpu().numpy().view(np.uint64), he.moddown(u, level)), level
    finally:
        pk.he_ctx_destroy(ctx)


@pytest.mark.parametrize("alpha,n,n1z,n1t", [(1, 8, 2, 4), (2, 8, 4, 2), (3, 4, 2, 1), (4, 8, 8, 8)])
def test_products_on_mixed_limbs(alpha, n, n1z, n1t):
    """One product and a batch with shared operands: BSGS transforms, C^k / R^k
    with unequal baby counts, the products' summed relinearisation."""
    from oracle.hmm import HMM, matmul_rot_steps
    pk, ctx, P, he = _open(alpha)
    try:
        steps = matmul_rot_steps(n, n1z, n1t, P.S)
        pk.he_keygen(ctx, steps, want_relin=True)
        for s in steps:
            he.gen_rotation_key(s)
        he.gen_relin_key()
        rng = np.random.default_rng(10 + alpha)
        g, o = [], []
        for i in range(3):
            z = np.zeros(P.S)
            z[:n * n] = rng.uniform(-1, 1, n * n)
            o.append(he.encrypt_slots(z, P.L, obj=20 + i))
            g.append(pk.he_encrypt_matrix(ctx, z[:n * n].reshape(n, n), P.L, 20 + i))
        hm = HMM(he)
        pairs = [(0, 1), (0, 2)]     # a shared left operand
        for once in (False, True):
            want = [hm.hmatmul(o[a], o[b], n, n1z, n1t, relin_once=once) for a, b in pairs]
            outs = pk.he_hmatmul_batch([(g[a], g[b], n, n1z, n1t, once) for a, b in pairs])
            outs.append(pk.he_hmatmul(ctx, g[0], g[1], n, n1z, n1t, once))
            for h, w in zip(outs, want + want[:1]):
                assert np.array_equal(pk.he_ct_export(ctx, h), np.stack([w.c0, w.c1])), once
                pk.he_ct_free(h)
        for h in g:
            pk.he_ct_free(h)
    finally:
        pk.he_ctx_destroy(ctx)

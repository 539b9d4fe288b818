"""The register-blocked NTT's three kinds of butterfly (float-quotient on
primes 2^36 <= q < 1.5 2^40, lazy Shoup below 2^57, reducing Shoup above) at
the edges of their ranges, and the row pass's grouping of limbs of one prime
(1, 2 or 4 per CTA, with a ragged last group)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# primes on both sides of 2^b for b = 36, 38, 39, 40, 41, and in the ranges of
# the Shoup butterflies
QBITS = [60, 36, 36, 37, 38, 38, 39, 39, 40, 40, 41, 41, 42, 50, 57, 57, 58]
PBITS = [60, 60]


@pytest.mark.parametrize("logN", [14, 15, 16])
def test_ntt_at_the_edges_of_the_butterfly_ranges(logN):
    import torch

    import paper_2305_17341_gb300 as pk
    from oracle import _c
    pk.build()
    ctx = pk.he_ctx_create(pk.make_params(logN, QBITS, PBITS), 3)
    try:
        q, p = pk.he_ctx_primes(ctx)
        primes = [int(v) for v in list(q) + list(p)]
        assert any(v < 1 << 36 for v in primes) and any(1 << 36 < v < (1 << 36) + (1 << 30) for v in primes)
        n, N, level = len(primes), 1 << logN, len(QBITS) - 1

        def words(kind, m, rng):
            if kind == 0:
                return rng.integers(0, m, N, dtype=np.uint64)
            if kind == 1:      # the largest values, the longest runs of equal signs
                return np.full(N, m - 1, dtype=np.uint64)
            return np.where(rng.integers(0, 2, N) == 0, np.uint64(0), np.uint64(m - 1))

        def run(rows, inverse=False):
            d = torch.from_numpy(rows.view(np.int64).copy()).cuda()
            torch.cuda.synchronize()
            pk.he_ntt(ctx, d.data_ptr(), rows.shape[0], level, inverse)
            return d.cpu().numpy().view(np.uint64)

        rng = np.random.default_rng(logN)
        single = {}
        for kind in range(3):
            a = np.stack([words(kind, primes[i], rng) for i in range(n)])
            b = np.stack([rng.integers(0, primes[i], N, dtype=np.uint64) for i in range(n)])
            fa, fb = run(a), run(b)
            for i in range(n):
                assert int(fa[i].max()) < primes[i] and int(fb[i].max()) < primes[i]
            prod = np.stack([np.array([x * y % primes[i] for x, y in zip(fa[i].tolist(), fb[i].tolist())],
                                      dtype=np.uint64) for i in range(n)])
            got = run(prod, True)
            for i in range(n):
                assert np.array_equal(got[i], _c.polymul(primes[i], a[i], b[i])), (kind, primes[i])
            assert np.array_equal(run(fa, True), a), kind
            single[kind] = (a, fa)
        # several limbs per prime: the same words as one limb per prime
        for R in (2 * n, 4 * n, 4 * n + 3, 8 * n - 1):
            a = np.stack([single[(r // n) % 3][0][r % n] for r in range(R)])
            f = np.stack([single[(r // n) % 3][1][r % n] for r in range(R)])
            assert np.array_equal(run(a), f), R
            assert np.array_equal(run(f, True), a), R
    finally:
        pk.he_ctx_destroy(ctx)

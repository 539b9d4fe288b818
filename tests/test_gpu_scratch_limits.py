"""What fits the device one item at a time runs when the scratch of groups does
not: a transform, a captured plan and the PowerMethod with little free memory
give the words, and the operation counts, that they give with plenty.

The room left is between the two: a sigma of one 64 x 64 matrix (level 12, 13
digits, 14 rows of 128 KB) takes 15 giants' digits and sums together in about
550 MB, one giant at a time in about 90 MB, beside 222 MB of plaintexts; eight
products of the PowerMethod's step together take 277 MB, one at a time 35 MB."""
import contextlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LOGN, QBITS, PBITS, SEED = 14, [60] + [40] * 12, [60], 91
LEVEL = len(QBITS) - 1
MB = 1 << 20


@contextlib.contextmanager
def room(mb):
    """Leaves about `mb` MB of the device's memory free."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = []
    try:
        for _ in range(4):
            free = torch.cuda.mem_get_info()[0]
            if free <= (mb + 8) * MB:
                break
            hold.append(torch.empty(free - mb * MB, dtype=torch.uint8, device="cuda"))
        assert torch.cuda.mem_get_info()[0] <= (mb + 16) * MB
        yield
    finally:
        hold.clear()
        torch.cuda.empty_cache()


def _open(pk, steps, relin):
    ctx = pk.he_ctx_create(pk.make_params(LOGN, QBITS, PBITS), SEED)
    pk.he_ctx_set_autotune(ctx, False)
    pk.he_keygen(ctx, sorted(steps), want_relin=relin)
    return ctx


def _counts(pk, ctx):
    c = pk.he_counters(ctx)
    return c["MS"], c["Dp"], c["MD"]


def test_transform_and_plan_with_little_room():
    import paper_2305_17341_gb300 as pk
    pk.build()
    n, n1, S = 64, 8, 1 << (LOGN - 1)
    steps = pk.he_rot_steps_for_matmul(n, n1, n1, S)
    rng = np.random.default_rng(6)
    A, B = rng.uniform(-1, 1, (2, n, n))

    def run(ctx, squeezed):
        a, b = pk.he_encrypt_matrix(ctx, A, LEVEL, 1), pk.he_encrypt_matrix(ctx, B, LEVEL, 2)
        ar = pk.he_replicate(ctx, a, n)
        pk.he_counters(ctx, reset=True)
        with room(460) if squeezed else contextlib.nullcontext():
            s = pk.he_linear_transform(ctx, ar, 0, n, n1)
        out = [pk.he_ct_export(ctx, s), _counts(pk, ctx)]
        # a product fills the context's caches; then the plan has little room
        p = pk.he_hmatmul(ctx, a, b, n, n1, n1)
        out.append(pk.he_ct_export(ctx, p))
        with room(100) if squeezed else contextlib.nullcontext():
            plan = pk.he_mm_plan_create([(a, b, n, n1, n1)])
            bytes_ = pk.he_mm_plan_info(plan)["bytes"]
            for _ in range(2):
                r = pk.he_mm_plan_run(plan)[0]
                out.append(pk.he_ct_export(ctx, r))
                pk.he_ct_free(r)
            pk.he_mm_plan_destroy(plan)
        for h in (a, b, ar, s, p):
            pk.he_ct_free(h)
        return out, bytes_

    wide = _open(pk, steps, True)
    try:
        want, most = run(wide, False)
    finally:
        pk.he_ctx_destroy(wide)
    tight = _open(pk, steps, True)
    try:
        got, least = run(tight, True)
        # with room again, groups again
        full = pk.he_mm_plan_create([(h, h, n, n1, n1) for h in [pk.he_encrypt_matrix(tight, A, LEVEL, 1)]])
        again = pk.he_mm_plan_info(full)["bytes"]
        pk.he_mm_plan_destroy(full)
    finally:
        pk.he_ctx_destroy(tight)
    assert got[1] == want[1]
    for i in (0, 2, 3, 4):
        assert np.array_equal(got[i], want[i]), i
    assert least < 0.6 * most and again == most


def test_power_method_with_little_room():
    import paper_2305_17341_gb300 as pk
    from oracle.pca import lazy_normalization_schedule
    pk.build()
    n, k, l_P, S = 16, 3, 1, 1 << (LOGN - 1)
    steps, i = set(), 1
    while i < n * n:
        steps |= {i, n * n - i}
        i <<= 1
    rng = np.random.default_rng(9)
    X = rng.standard_normal((100, k * n))
    C = X.T @ X / 100
    C *= 1.5 / np.linalg.eigvalsh(C)[-1]
    v = rng.standard_normal(k * n)
    v /= np.linalg.norm(v)
    counts = lazy_normalization_schedule(l_P)

    def run(ctx, mb):
        def enc(blk, obj):
            h = pk.he_encrypt_slots(ctx, np.tile(blk.ravel(), S // (n * n)), LEVEL, obj)
            r = pk.he_ct_import(ctx, pk.he_ct_export(ctx, h), LEVEL, pk.he_ct_info(h)[1], n * n)
            pk.he_ct_free(h)
            return r

        cov = [enc(C[a * n:(a + 1) * n, b * n:(b + 1) * n], 10 + a * k + b) for a in range(k) for b in range(k)]
        v0 = [enc(np.tile(v[j * n:(j + 1) * n], n), 30 + j) for j in range(k)]
        rs = pk.he_refresh_state(1 << 20, 0)
        pk.he_counters(ctx, reset=True)
        with room(mb) if mb else contextlib.nullcontext():
            lam, V, VT, ax = pk.he_power_method(ctx, cov, k, n, v0, 0, l_P, counts, 2.0 ** 16, rs)
        out = [pk.he_ct_export(ctx, h) for h in [lam] + V + VT], (ax, rs.count) + _counts(pk, ctx)
        for h in cov + v0 + V + VT + [lam]:
            pk.he_ct_free(h)
        return out

    wide = _open(pk, steps, True)
    try:
        want, meta = run(wide, 0)
    finally:
        pk.he_ctx_destroy(wide)
    tight = _open(pk, steps, True)
    try:
        got, meta_t = run(tight, 140)
    finally:
        pk.he_ctx_destroy(tight)
    assert meta_t == meta
    for g, w in zip(got, want):
        assert np.array_equal(g, w)

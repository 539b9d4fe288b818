"""The work that users of this framework have it do, as cases to be timed.

Every case goes through the package's public functions: device transforms and
key-switch parts on tensors, ciphertext operations, matrix products (single,
batched, replayed from a captured plan), the covariance circuit and the
PowerMethod.  Results leave the way a cloud program sends them back: residues
exported into pinned host memory, and, where the client's side belongs to the
call, decrypted values.

A context with its keys is what a program sets up once and keeps, so contexts
are shared by the states of equal parameters; every state has its own inputs,
drawn from its seed.

Residues are whole numbers: they have no nearest 64-bit floating value, so
exact() speaks only for the decrypted outputs.
"""
import collections
import ctypes
import math

import numpy as np
import torch

import paper_2305_17341_gb300 as pk
from paper_2305_17341_gb300 import _lib, workloads

_u64p = ctypes.POINTER(ctypes.c_uint64)


# --------------------------------------------------------------------- cases
def listed():
    return [
        # a user's smallest call: one polynomial of the 32 x 32 preset
        # (5 limbs) into the NTT domain
        dict(name="ntt_one_poly", kind="ntt", logN=14, n_q=4, n_p=1, level=3, rows=5, inverse=False),
        # the polynomials of a ragged group of ciphertexts back to
        # coefficients before a download (19 limbs, an odd number of rows)
        dict(name="ntt_inverse", kind="ntt", logN=15, n_q=17, n_p=2, level=16, rows=209, inverse=True),
        # the bench's transform workload: 8 items x 11 digits x 23 rows
        dict(name="ntt_batch", kind="ntt", logN=16, n_q=21, n_p=2, level=20, rows=2024, inverse=False),
        # the two halves of a key switch by themselves, for a pipeline that
        # has its own inner product: Decompose and ModDown of 3 items
        dict(name="keyswitch_parts", kind="parts", logN=16, n_q=21, n_p=2, level=19, items=3),
        # a rotation in caller-owned memory: one small call on the latency path
        dict(name="rotate_noalloc", kind="rotate", logN=14, n_q=4, n_p=1, level=3, step=100),
        # one product of two ciphertexts and its rescale at the top level
        dict(name="mult_rescale", kind="mult", logN=16, n_q=21, n_p=2, level=20),
        # sigma of one 128 x 128 matrix in the paper's Table 3 setting
        dict(name="transform_sigma", kind="transform", logN=15, n_q=15, n_p=2, level=11, which=0, n=128, n1=16,
             n_prime=0),
        # the client's whole round trip: encrypt two 32 x 32 matrices,
        # multiply, decrypt (the 32 x 32 preset)
        dict(name="product_one", kind="product", logN=14, n_q=4, n_p=1, level=3, n=32, n1=8, relin_once=False, dcd=0),
        # 16 resident 32 x 32 products replayed from a captured plan
        dict(name="product_plan", kind="batch", logN=14, n_q=4, n_p=1, level=3, n=32, n1=8, relin_once=False, dcd=0,
             count=16, plan=True),
        # the headline: 8 resident 128 x 128 products in one batch
        dict(name="product_batch", kind="batch", logN=16, n_q=21, n_p=2, level=20, n=128, n1=16, relin_once=False,
             dcd=0, count=8, plan=False),
        # covariance of 256 samples x 256 features in 128 x 128 blocks with
        # the decomposed products of the paper's Sec. 7
        dict(name="covariance", kind="covariance", logN=16, n_q=21, n_p=2, level=20, n=128, n1=16, dcd=32,
             samples=256, features=256),
        # two normalised PowerMethod iterations on a 256 x 256 covariance, with
        # the Lazy Normalization counts of two iterations
        dict(name="power_method", kind="power", logN=16, n_q=14, n_p=2, level=13, n=128, features=256, newton="7 24"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same kinds; sizes spread over the kinds' ranges."""
    kind = rng.choice(["ntt", "ntt", "parts", "rotate", "mult", "transform", "product", "batch"])
    logN = rng.choice([14, 15, 16])
    n_p = rng.choice([1, 2, 2])
    n_q = rng.randint(4, 21 if n_p == 2 else 10)
    if kind == "ntt":
        return dict(kind=kind, logN=logN, n_q=n_q, n_p=n_p, level=rng.randint(0, n_q - 1),
                    rows=_log_int(rng, 1, 2024), inverse=rng.random() < 0.5)
    if kind == "parts":
        return dict(kind=kind, logN=logN, n_q=n_q, n_p=n_p, level=rng.randint(0, n_q - 1), items=_log_int(rng, 1, 8))
    if kind == "rotate":
        # the reserved scratch bounds the level (levels up to 3 fit at every N)
        return dict(kind=kind, logN=logN, n_q=n_q, n_p=n_p, level=rng.randint(0, 3), step=_log_int(rng, 1, 4000))
    if kind == "mult":
        return dict(kind=kind, logN=logN, n_q=n_q, n_p=n_p, level=rng.randint(1, n_q - 1))
    if kind == "transform":
        logN = rng.choice([14, 15])
        which = rng.choice([0, 1, 2])
        n = rng.choice([16, 32, 64])
        n1 = rng.choice([2, 4, 8])
        n_prime = n // 2 if which < 2 and rng.random() < 0.4 else 0
        return dict(kind=kind, logN=logN, n_q=n_q, n_p=n_p, level=rng.randint(2, n_q - 1), which=which, n=n, n1=n1,
                    n_prime=n_prime)
    logN = rng.choice([14, 15])
    n = rng.choice([8, 16, 32])
    n1 = rng.choice([2, 4, 8])
    dcd = n // 2 if n1 <= n // 2 and n_q > 4 and rng.random() < 0.3 else 0
    level = rng.randint(4 if dcd else 3, n_q - 1)
    case = dict(kind=kind, logN=logN, n_q=n_q, n_p=n_p, level=level, n=n, n1=n1, relin_once=rng.random() < 0.3,
                dcd=dcd)
    if kind == "batch":
        case.update(count=_log_int(rng, 2, 12), plan=rng.random() < 0.4)
    return case


# ------------------------------------------------------------------- handles
class _Context:
    """A context and the ciphertext handles that belong to it."""

    def __init__(self, logN, n_q, n_p):
        self.h = pk.he_ctx_create(pk.make_params(logN, [60] + [40] * (n_q - 1), [60] * n_p), 42)
        self.S = 1 << (logN - 1)
        q, p = pk.he_ctx_primes(self.h)
        self.q, self.p = q, p

    def __del__(self):
        pk.he_ctx_destroy(self.h)


_contexts = collections.OrderedDict()


def _context(case):
    """The context of a case's parameters: made once and kept, like its keys
    (a program that moves on to other parameters lets the oldest go)."""
    key = (case["logN"], case["n_q"], case["n_p"])
    if key not in _contexts:
        while len(_contexts) >= 2:
            _contexts.popitem(last=False)
        _contexts[key] = _Context(*key)
    _contexts.move_to_end(key)
    return _contexts[key]


class _State:
    """One program's inputs: ciphertexts (freed with the state, before the
    context can go), tensors, and the pinned buffers results are sent from."""

    def __init__(self, case, ctx):
        self.case, self.ctx, self.cts, self.plan, self.out = case, ctx, [], None, []

    def sends(self, count):
        """Pinned memory for `count` results of at most the inputs' level."""
        words = 2 * (self.case["level"] + 1) << self.case["logN"]
        self.out = [torch.empty(words, dtype=torch.int64, pin_memory=True) for _ in range(count)]

    def export(self, handles):
        """Residues of the handles in pinned memory; the handles are freed."""
        got = []
        for buf, h in zip(self.out, handles):
            t = buf[:2 * (pk.he_ct_info(h)[0] + 1) << self.case["logN"]]
            _lib.check(pk.lib().he_ct_export(h, ctypes.cast(t.data_ptr(), _u64p)))
            pk.he_ct_free(h)
            got.append(t)
        return got

    def __del__(self):
        if self.plan is not None:
            pk.he_mm_plan_destroy(self.plan)
        for h in self.cts:
            pk.he_ct_free(h)


def _residues(ctx, rows, level, N, seed, with_p):
    """rows x N residues, row r uniform modulo prime r mod (number of primes)."""
    primes = ctx.q[:level + 1] + (ctx.p if with_p else [])
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    t = torch.randint(0, 1 << 62, (rows, N), dtype=torch.int64, device="cuda", generator=g)
    q = torch.tensor([primes[r % len(primes)] for r in range(rows)], dtype=torch.int64, device="cuda")
    t.remainder_(q[:, None])
    return t


def _pow2_steps(n):
    steps, i = set(), 1
    while i < n * n:
        steps |= {i % (n * n), (-i) % (n * n)}
        i <<= 1
    return steps - {0}


def _replication_steps(n, S):
    steps, r = set(), n * n
    while r < S:
        steps.add(S - r)
        r *= 2
    return steps


def _covariance_data(case, seed):
    return workloads.lowrank_dataset(case["samples"], case["features"], seed)


def _newton(case):
    return [int(v) for v in case["newton"].split()]


def _power_data(case, seed):
    """A covariance scaled like the client's (by the feature count), and a unit start vector."""
    t = case["features"]
    X = workloads.lowrank_dataset(t, t, seed)
    Xc = X - X.mean(0)
    v0 = np.random.default_rng(seed).standard_normal(t)
    return Xc.T @ Xc, v0 / np.linalg.norm(v0)


# ------------------------------------------------------------------- prepare
def prepare(case, seed):
    ctx = _context(case)
    s = _State(case, ctx)
    kind, N, level = case["kind"], 1 << case["logN"], case["level"]
    if kind == "ntt":
        s.rows = _residues(ctx, case["rows"], level, N, seed, True)
    elif kind == "parts":
        nq, rows, items = level + 1, level + 1 + case["n_p"], case["items"]
        nd = -(-nq // case["n_p"])
        s.poly = _residues(ctx, items * nq, level, N, seed, False)
        s.wide = _residues(ctx, items * rows, level, N, seed + 1000003, True)
        s.digits = torch.empty((items, nd, rows, N), dtype=torch.int64, device="cuda")
        s.down = torch.empty((items, nq, N), dtype=torch.int64, device="cuda")
    elif kind == "rotate":
        pk.he_keygen(ctx.h, [case["step"]], False)
        s.inp = _residues(ctx, 2 * (level + 1), level, N, seed, False)
        s.res = torch.empty_like(s.inp)
    elif kind == "mult":
        pk.he_keygen(ctx.h, [], True)
        rng = np.random.default_rng(seed)
        s.cts = [pk.he_encrypt_slots(ctx.h, rng.uniform(-1, 1, ctx.S), level, 2 * seed + i) for i in range(2)]
        s.sends(1)
    elif kind == "transform":
        n, n1, np_ = case["n"], case["n1"], case["n_prime"]
        if case["which"] == 2:
            steps = pk.he_rot_steps_for_transpose(n, n1, ctx.S)
        else:
            # each of the two uses its own part of the schedule's steps
            steps = pk.he_rot_steps_for_sched(n, n1, n1, ctx.S, np_, np_)
        pk.he_keygen(ctx.h, steps, False)
        s.cts = [pk.he_encrypt_matrix(ctx.h, workloads.matmul_pair(n, seed)[0], level, seed)]
        s.sends(1)
    elif kind in ("product", "batch"):
        n, n1, dcd = case["n"], case["n1"], case["dcd"]
        pk.he_keygen(ctx.h, pk.he_rot_steps_for_sched(n, n1, n1, ctx.S, dcd, dcd), True)
        s.mats = [workloads.matmul_pair(n, 64 * seed + i) for i in range(case.get("count", 1))]
        s.sends(len(s.mats))
        if kind == "batch":
            for i, ab in enumerate(s.mats):
                s.cts += [pk.he_encrypt_matrix(ctx.h, m, level, 2 * i + j) for j, m in enumerate(ab)]
            s.jobs = [(s.cts[2 * i], s.cts[2 * i + 1], n, n1, n1, case["relin_once"], dcd, dcd)
                      for i in range(case["count"])]
            if case["plan"]:
                s.plan = pk.he_mm_plan_create(s.jobs)
    elif kind == "covariance":
        n, n1, dcd = case["n"], case["n1"], case["dcd"]
        steps = set(pk.he_rot_steps_for_sched(n, n1, n1, ctx.S, dcd, dcd))
        steps |= set(pk.he_rot_steps_for_transpose(n, n1, ctx.S)) | _pow2_steps(n)
        pk.he_keygen(ctx.h, sorted(steps), True)
        X = _covariance_data(case, seed)
        s.nrb, s.k = case["samples"] // n, case["features"] // n
        s.cts = [pk.he_encrypt_matrix(ctx.h, X[l * n:(l + 1) * n, j * n:(j + 1) * n], level, 100 + l * s.k + j)
                 for l in range(s.nrb) for j in range(s.k)]
        s.sends(s.k * s.k)
    elif kind == "power":
        n = case["n"]
        s.k = case["features"] // n
        pk.he_keygen(ctx.h, sorted(_pow2_steps(n) | _replication_steps(n, ctx.S)), True)
        C, v0 = _power_data(case, seed)

        def enc(m, obj):
            a = pk.he_encrypt_matrix(ctx.h, m, level, obj)
            b = pk.he_replicate(ctx.h, a, n)
            pk.he_ct_free(a)
            return b

        blocks = [C[a * n:(a + 1) * n, b * n:(b + 1) * n] for a in range(s.k) for b in range(s.k)]
        s.cts = [enc(m, 200 + i) for i, m in enumerate(blocks)]
        s.cts += [enc(np.tile(v0[j * n:(j + 1) * n], (n, 1)), 300 + j) for j in range(s.k)]
        s.newton = _newton(case)
        s.sends(1 + 2 * s.k)
    else:
        raise ValueError(kind)
    torch.cuda.synchronize()   # the context's stream is not ordered after torch's
    return s


# ----------------------------------------------------------------------- run
def run(s):
    case, ctx = s.case, s.ctx.h
    kind, level = case["kind"], case["level"]
    if kind == "ntt":
        pk.he_ntt(ctx, s.rows.data_ptr(), case["rows"], level, case["inverse"])
        return s.rows
    if kind == "parts":
        pk.he_decompose(ctx, s.poly.data_ptr(), case["items"], level, s.digits.data_ptr())
        pk.he_moddown(ctx, s.wide.data_ptr(), case["items"], level, s.down.data_ptr())
        return [s.digits, s.down]
    if kind == "rotate":
        pk.he_rotate_noalloc(ctx, s.inp.data_ptr(), level, case["step"], s.res.data_ptr())
        return s.res
    if kind == "mult":
        m = pk.he_mult(ctx, s.cts[0], s.cts[1])
        r = pk.he_rescale(ctx, m)
        pk.he_ct_free(m)
        return s.export([r])
    if kind == "transform":
        return s.export([pk.he_linear_transform(ctx, s.cts[0], case["which"], case["n"], case["n1"],
                                                case["n_prime"])])
    if kind == "product":
        A, B = s.mats[0]
        a, b = pk.he_encrypt_matrix(ctx, A, level, 1), pk.he_encrypt_matrix(ctx, B, level, 2)
        c = pk.he_hmatmul(ctx, a, b, case["n"], case["n1"], case["n1"], case["relin_once"], case["dcd"], case["dcd"])
        m = pk.he_decrypt_matrix(ctx, c, case["n"], case["n"])
        pk.he_ct_free(a)
        pk.he_ct_free(b)
        return {"words": s.export([c]), "matrix": m}
    if kind == "batch":
        return s.export(pk.he_mm_plan_run(s.plan) if s.plan is not None else pk.he_hmatmul_batch(s.jobs))
    if kind == "covariance":
        n, n1, dcd = case["n"], case["n1"], case["dcd"]
        C = pk.he_covariance(ctx, s.cts, s.nrb, s.k, n, case["samples"], False, n1, n1, dcd_z=dcd, dcd_t=dcd)
        mats = [pk.he_decrypt_matrix(ctx, h, n, n) for h in C]
        return {"words": s.export(C), "blocks": mats}
    n, kk = case["n"], s.k * s.k
    rs = pk.he_refresh_state(1 << 20, 0)
    lam, V, VT, axis = pk.he_power_method(ctx, s.cts[:kk], s.k, n, s.cts[kk:], 0, len(s.newton), s.newton, 2.0 ** 16,
                                          rs)
    mats = [pk.he_decrypt_matrix(ctx, h, n, n) for h in V]
    value = pk.he_decrypt_slots(ctx, lam, n * n)
    return {"words": s.export([lam] + V + VT), "vector": mats, "value": value, "axis": axis, "refreshes": rs.count}


# ----------------------------------------------------------------------- work
class _Work:
    """Words every operation has to read and write once, and the modular
    products (counted as two operations each) of the paper's schedules."""

    def __init__(self, case):
        self.N, self.logN, self.a = 1 << case["logN"], case["logN"], case["n_p"]

    def ntt(self, rows):
        return rows * (self.N // 2) * self.logN

    def digits(self, level):
        return -(-(level + 1) // self.a)

    def decompose(self, level):
        rows, nd = level + 1 + self.a, self.digits(level)
        ext = nd * rows - (level + 1)
        return self.ntt(level + 1 + ext) + (level + 1) * rows * self.N

    def moddown(self, level):
        """One polynomial."""
        return self.ntt(self.a + level + 1) + self.a * (level + 1) * self.N

    def multsum(self, level):
        return 2 * self.digits(level) * (level + 1 + self.a) * self.N

    def rescale(self, level):
        return 2 * self.ntt(1 + level)

    def key_switch(self, ms, dp, md, level):
        return ms * self.multsum(level) + dp * self.decompose(level) + 2 * md * self.moddown(level)

    def ct(self, level):
        return 2 * (level + 1) * self.N * 8

    def key(self, level):
        return 2 * self.digits(level) * (level + 1 + self.a) * self.N * 8


def _zt_counts(n, n1, which):
    """(MultSum, Decompose, ModDown) of one undecomposed transform."""
    g = (n // n1 if which == 1 else 2 * (n // n1)) - 1   # giants with a rotation
    return n1 - 1 + g, 1 + g, 1 + g


def _product_products(w, n, n1, level, relin_once):
    z, t = _zt_counts(n, n1, 0), _zt_counts(n, n1, 1)
    g = n // n1
    top = tuple(a + b for a, b in zip(z, t))
    mid = (2 * (n - 1) + 1 + n - 1, 3 * g, 1 + 2 * (g - 1) + 2 * (n - 1))
    relins = 1 if relin_once else n
    return (w.key_switch(*top, level) + w.key_switch(*mid, level - 1) + w.key_switch(relins, relins, relins, level - 2)
            + 4 * n * (level - 1) * w.N + (n - 1) * w.rescale(level - 1) + w.rescale(level - 2))


def work(case):
    w = _Work(case)
    kind, level = case["kind"], case["level"]
    if kind == "ntt":
        return {"bytes": 16 * case["rows"] * w.N, "flops": 2 * w.ntt(case["rows"])}
    if kind == "parts":
        rows, nq, m = level + 1 + w.a, level + 1, case["items"]
        words = m * w.N * (nq + w.digits(level) * rows + rows + nq)
        return {"bytes": 8 * words, "flops": 2 * m * (w.decompose(level) + w.moddown(level))}
    if kind == "rotate":
        return {"bytes": 2 * w.ct(level) + w.key(level),
                "flops": 2 * (w.key_switch(1, 1, 1, level) + w.ntt(4 * (level + 1)))}
    if kind == "mult":
        return {"bytes": 2 * w.ct(level) + w.key(level) + w.ct(level - 1),
                "flops": 2 * (w.key_switch(1, 1, 1, level) + 4 * (level + 1) * w.N + w.rescale(level))}
    if kind == "transform":
        ms, dp, md = _zt_counts(case["n_prime"] or case["n"], case["n1"], case["which"])
        return {"bytes": w.ct(level) + ms * w.key(level) + w.ct(level - 1),
                "flops": 2 * (w.key_switch(ms, dp, md, level) + w.rescale(level))}
    if kind in ("product", "batch"):
        n, n1, count = case["n"], case["n1"], case.get("count", 1)
        keys = n1 - 1 + n // n1 * 3 + 2
        return {"bytes": count * (2 * w.ct(level) + w.ct(level - 3)) + keys * w.key(level),
                "flops": 2 * count * _product_products(w, n, n1, level, case["relin_once"])}
    n = case["n"]
    k = case["features"] // n
    if kind == "covariance":
        nrb, n1 = case["samples"] // n, case["n1"]
        pairs = nrb * k * (k + 1) // 2
        return {"bytes": (nrb * k + k * k) * w.ct(level) + (3 * n1 + 30) * w.key(level),
                "flops": 2 * (pairs * _product_products(w, n, n1, level - 4, False)
                              + (nrb * k + k) * w.key_switch(*_zt_counts(n, n1, 2), level))}
    # PowerMethod: per iteration k*k products with the covariance, log2(n)
    # rotations per segment and axis flip, and the Newton steps' products
    its = len(_newton(case)) + 1
    switches = its * (k * k + 3 * k * int(math.log2(n)) + 40)
    return {"bytes": (k * k + 3 * k + 1) * w.ct(level) + (2 * int(math.log2(n * n)) + 2) * w.key(level),
            "flops": 2 * w.key_switch(switches, switches, switches, level // 2)}


# ---------------------------------------------------------------------- exact
def exact(case, seed):
    """The decrypted outputs in 64-bit floats; None for the ciphertexts."""
    kind = case["kind"]
    if kind == "product":
        A, B = workloads.matmul_pair(case["n"], 64 * seed)
        return {"words": [None], "matrix": A @ B}
    if kind == "covariance":
        n, X = case["n"], _covariance_data(case, seed)
        Xc = X - X.mean(0)
        C, k = Xc.T @ Xc / case["samples"], case["features"] // case["n"]
        blocks = [C[a * n:(a + 1) * n, b * n:(b + 1) * n].copy() for a in range(k) for b in range(k)]
        return {"words": [None] * (k * k), "blocks": blocks}
    if kind == "power":
        # the same schedule in floating point: normalised iterations whose
        # inverse square root starts from the order-1 Taylor value at B2/2 + 1
        # and takes the Lazy Normalization's Newton counts
        n, k = case["n"], case["features"] // case["n"]
        C, v = _power_data(case, seed)
        x0 = 2.0 ** 15 + 1.0
        newton = _newton(case)
        for steps in newton:
            y = C @ v
            x = y @ y
            inv = x0 ** -0.5 * (1.5 - x / (2.0 * x0))
            for _ in range(steps):
                inv = 0.5 * inv * (3.0 - x * inv * inv)
            v = y * inv
        lam = float((C @ v) @ v)
        axis = len(newton) % 2   # every transformation flips the vector's axis
        mats = [np.tile(v[j * n:(j + 1) * n], (n, 1)) if axis == 0 else np.tile(v[j * n:(j + 1) * n, None], (1, n))
                for j in range(k)]
        return {"words": [None] * (1 + 2 * k), "vector": mats, "value": np.full(n * n, lam), "axis": None,
                "refreshes": None}
    return None

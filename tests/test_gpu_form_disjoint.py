"""Rows of a Form's operands that are large in different pivots: digits that are cut
relative to the row's largest entry say little of such a pair's product, so the
Form (single and batched) and the blocked Solve's updates must take it by FP64
multiply-adds.

Tolerances, entry by entry: the Form within (2 e + 8) 2^-53 |W21||L21|^T, as in
test_gpu_form_fp64; a Solve's Y satisfies Y L11^T = x + R with |R| <= (2 e + 8) 2^-53
|Y||L11|^T, so it is off by at most that times |L11^-T|.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1305_2353_gb300 import inputs
from test_gpu_form_fp64 import _check, _factor
from test_gpu_supernode import ctx  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

EPS = [1e-2, 1e-3, 1e-6, 1e-12, 1e-18]


def _classes(m, how, rng):
    """Which half of the pivots each row is large in."""
    i = np.arange(m)
    return {"tiles": (i // 32) % 2, "blocks": (i // 128) % 2, "columns": (i // 64) % 2, "rows": i % 2,
            "random": rng.integers(0, 2, m), "few": (rng.random(m) < 0.02).astype(int)}[how]


def _disjoint(m, p, eps, how, seed, zeros=0.0):
    rng = np.random.default_rng(seed)
    A = np.zeros((p + m, p), order="F")
    A[:p] = np.diag(rng.uniform(1, 2, p))  # L11 = I: W21 and L21 are A21 and A21 D^-1
    half = (np.arange(p) >= p // 2).astype(int)
    B = rng.uniform(0.5, 1, (m, p)) * rng.choice([-1, 1], (m, p))
    B[_classes(m, how, rng)[:, None] != half[None, :]] *= eps
    B[rng.random((m, p)) < zeros] = 0.0
    A[p:] = B
    return A


@pytest.mark.parametrize("how", ["tiles", "blocks", "columns", "rows", "random", "few"])
@pytest.mark.parametrize("eps", EPS)
def test_form_disjoint_rows(ctx, how, eps):
    for m, p, zeros in ((64, 32, 0.0), (300, 32, 0.0), (290, 96, 0.0), (200, 12, 0.5), (129, 256, 0.3)):
        res = _factor(ctx, _disjoint(m, p, eps, how, 3 * p + m, zeros), p, "restricted", "fp64")
        assert res["nelim"] == p
        _check(res, p, "fp64")


@pytest.mark.parametrize("eps", EPS)
def test_form_disjoint_rows_batched(ctx, eps):
    from paper_1305_2353_gb300 import ctp
    shapes = [(64, 32, "tiles"), (300, 48, "blocks"), (130, 96, "random"), (20, 8, "rows"), (40, 33, "few"),
              (200, 160, "columns")]
    fronts = [_disjoint(m, p, eps, how, p) for m, p, how in shapes]
    ps = [p for _, p, _ in shapes]
    b = ctp.Batch(ctx, fronts, ps, ctp.options(pivot="restricted", smode="fp64_packed"))
    b.run()
    assert np.all(b.flags() == 0)
    for k, p in enumerate(ps):
        res = b.result(k)
        assert res["nelim"] == p
        _check(res, p, "fp64")


@pytest.mark.parametrize("eps", EPS)
@pytest.mark.parametrize("m,p", [(40, 160), (700, 200), (9000, 96)])
def test_blocked_solve_disjoint_rows(ctx, m, p, eps):
    """y of the first block and the rows of L11 below it are large in different halves of the block."""
    rng = np.random.default_rng(p + m)
    A = np.zeros((p + m, p), order="F")
    half = np.arange(32) >= 16
    A[:p] = np.diag(np.r_[rng.uniform(1, 2, 32), rng.uniform(100, 200, p - 32)])
    below = rng.uniform(0.5, 1, (p - 32, 32)) * rng.choice([-1, 1], (p - 32, 32))
    below[:, ~half] *= eps
    A[32:p, :32], A[:32, 32:p] = below, below.T
    y = rng.uniform(0.5, 1, (m, 32)) * rng.choice([-1, 1], (m, 32))
    y[:, half] *= eps
    A[p:, :32] = y
    res = _factor(ctx, A, p, "restricted", "none")
    assert res["nelim"] == p and np.array_equal(np.sort(res["perm"][:32]), np.arange(32))
    L, Dm, _ = O.unpack(res, p)
    Lx = L[:p, :p].astype(np.longdouble)
    x = A[p:][:, res["perm"]].astype(np.longdouble)
    Y = np.zeros_like(x)
    for k in range(p):
        Y[:, k] = x[:, k] - Y[:, :k] @ Lx[k, :k]
    got = res["A"][p:].astype(np.longdouble) @ Dm.astype(np.longdouble)
    inv = np.abs(np.linalg.inv(L[:p, :p])).T
    bound = (2 * p + 8) * 2.0 ** -53 * (np.abs(Y) @ np.abs(Lx).T).astype(float) @ inv
    # Y D^-1 and back: two roundings more, and a 2x2 pivot's product
    bound = bound + 8 * 2.0 ** -53 * np.abs(res["A"][p:]) @ np.abs(Dm)
    assert np.all(np.abs(got - Y).astype(float) <= bound)


def test_random_rows_take_digits_only_where_sure(ctx):
    """Graded and sparse random rows: nothing lost whichever way an entry goes."""
    for seed, (m, p) in enumerate([(200, 20), (333, 130), (150, 256)]):
        A = inputs.supernode(p + m, p, seed=seed)
        rng = np.random.default_rng(seed)
        A[p:] *= 2.0 ** rng.uniform(-30, 0, (m, p)) * (rng.random((m, p)) < 0.5)
        res = _factor(ctx, A, p, "restricted", "fp64")
        assert res["nelim"] > p // 2
        _check(res, p, "fp64")

"""The FP64 Form from digit slices at the edges of its tiles (128 x 64), K blocks (32)
and K steps (16), in every layout of S, and its rows that take FP64 multiply-adds.

Tolerance: both sides form W21 = L21 D11 with at most three roundings per entry
and sum e products; the oracle's sum and the GPU's (whose digits lose less than
e FP64 roundings) are each within (e + 4) 2^-53 |W21||L21|^T of the exact one.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1305_2353_gb300 import inputs
from test_gpu_supernode import ctx  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CASES = [(1, 8, "tpp", "fp64"), (63, 16, "relaxed", "fp64_packed"), (64, 17, "restricted", "fp32"),
         (65, 32, "tpp", "fp32_packed"), (127, 33, "relaxed", "fp64"), (128, 64, "restricted", "fp64_packed"),
         (129, 65, "tpp", "fp64"), (500, 1, "relaxed", "fp64"), (641, 129, "restricted", "fp64_packed"),
         (1153, 256, "tpp", "fp64_packed"), (1100, 255, "relaxed", "fp64")]


def _factor(ctx, A, p, pivot, smode):
    from paper_1305_2353_gb300 import ctp
    sn = ctp.Supernode(ctx, A, p, ctp.options(pivot=pivot, smode=smode))
    sn.run()
    torch.cuda.synchronize()
    return sn.result()


def _bound(res, p):
    e = res["nelim"]
    L21 = res["A"][p:, :e]
    _, Dm, _ = O.unpack(res, p)
    W = np.abs(L21) @ np.abs(Dm)
    return (2 * e + 8) * 2.0 ** -53 * (W @ np.abs(L21).T)


def _check(res, p, smode, rows=slice(None)):
    e = res["nelim"]
    want = O.form(res["A"][p:, :e], res["piv"][:e], res["D"])
    lo = np.tril(np.ones_like(want, bool))
    bound = _bound(res, p)
    if smode.startswith("fp32"):
        bound = bound + 2.0 ** -24 * np.abs(want)
    got = res["S"].astype(np.float64)
    keep = lo & np.isfinite(want)
    assert np.all(np.abs(got - want)[keep] <= bound[keep])
    return keep


@pytest.mark.parametrize("m,p,pivot,smode", CASES)
def test_form_edges(ctx, m, p, pivot, smode):
    A = inputs.supernode(p + m, p, seed=7 * p + m, zero_diag_frac=0.2)
    res = _factor(ctx, A, p, pivot, smode)
    assert res["info"] == 0 and res["nelim"] > 0
    _check(res, p, smode)


@pytest.mark.parametrize("what", ["rows", "columns", "entries", "one_row"])
def test_form_wide_scales(ctx, what):
    """Row and column scales leave the slices as good as they are without; entries
    scattered over 2^40 fall to FP64 multiply-adds."""
    m, p = 300, 48
    A = inputs.supernode(p + m, p, seed=5)
    rng = np.random.default_rng(6)
    if what == "rows":
        A[p:] *= 2.0 ** rng.uniform(-300, 300, (m, 1))
    elif what == "columns":
        c = 2.0 ** rng.uniform(-8, 8, p)
        A[:p] *= c[:, None]
        A *= c
    elif what == "entries":
        A[p:] *= 2.0 ** rng.uniform(-40, 0, (m, p))
    else:
        A[p + 70] *= 2.0 ** rng.uniform(-40, 0, p)
    res = _factor(ctx, A, p, "restricted", "fp64")
    assert res["nelim"] > p // 2
    _check(res, p, "fp64")


def test_form_nonfinite_rows(ctx):
    """An Inf or NaN in a row of A21 reaches that row and column of S only."""
    m, p = 200, 40
    A = inputs.supernode(p + m, p, seed=8)
    ref = _factor(ctx, A, p, "restricted", "fp64")
    B = A.copy(order="F")
    B[p + 30, 3], B[p + 150, 7] = np.inf, np.nan
    res = _factor(ctx, B, p, "restricted", "fp64")
    hit = np.zeros((m, m), bool)
    hit[[30, 150], :] = hit[:, [30, 150]] = True
    lo = np.tril(np.ones((m, m), bool))
    assert np.array_equal(res["S"][lo & ~hit], ref["S"][lo & ~hit])
    assert not np.isfinite(res["S"][lo & hit]).any()

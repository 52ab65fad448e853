"""Batches whose fronts solve partly in blocks and partly in one pass within one
pivot-search class: fronts of the class without rows below the pivots (no slices are written
for them, and their sections have no room for any), with a few, and with many."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1305_2353_gb300 import inputs
from test_gpu_supernode import compare, ctx  # noqa: F401  (ctx is a fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("smode", ["none", "fp64_packed"])
@pytest.mark.parametrize("p,rows,pivot", [(96, [0, 400, 3, 0, 31, 33, 500, 400, 400, 400, 400, 400, 400, 400, 0, 1200], "restricted"),
                                          (200, [0, 300, 1, 40, 900, 700, 0], "restricted"),
                                          (200, [0, 300, 1, 40, 900, 700, 0], "strict")])
def test_fronts_without_rows_among_blocked_ones(ctx, p, rows, pivot, smode):
    from paper_1305_2353_gb300 import ctp
    # enough entries right of the first 32 columns for the class to solve in blocks
    # (restricted pivoting: one class, by p alone)
    assert sum(m * (p - 32) for m in rows if m >= 187) >= 3e5
    A = [inputs.supernode(p + m, p, seed=3 * k + p, zero_diag_frac=0.3) for k, m in enumerate(rows)]
    b = ctp.Batch(ctx, A, [p] * len(A), ctp.options(pivot=pivot, smode=smode))
    guard = b.ws.clone()  # same bytes behind the plan's tables on both runs: nothing reads stale slices
    b.run()
    first = [b.result(k) for k in range(len(A))]
    b.reset()
    b.ws.copy_(guard)
    b.run()
    assert np.all(b.flags() == 0)
    for k, a in enumerate(A):
        got = b.result(k)
        assert np.array_equal(got["A"], first[k]["A"]) and np.array_equal(got["perm"], first[k]["perm"])
        compare(O.factor(a, p, pivot, log_cap=400000), got, p, a)

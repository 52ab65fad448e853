"""FP64 fronts of few rows: their Form by FP64 multiply-adds (up to 32 rows), and the room
that a front's section takes in a batch's workspace.  Tolerances as in test_gpu_form_fp64."""
import numpy as np
import pytest

from paper_1305_2353_gb300 import inputs
from test_gpu_form_fp64 import _check, _factor
from test_gpu_supernode import ctx  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("m", [1, 2, 9, 31, 32, 33, 40])
@pytest.mark.parametrize("p,pivot,smode", [(1, "relaxed", "fp64"), (8, "strict", "fp64_packed"),
                                           (33, "restricted", "fp32"), (64, "tpp", "fp64_packed"),
                                           (100, "tpp", "fp32_packed"), (256, "relaxed", "fp64_packed")])
def test_form_of_few_rows(ctx, m, p, pivot, smode):
    A = inputs.supernode(p + m, p, seed=7 * p + m, zero_diag_frac=0.2)
    res = _factor(ctx, A, p, pivot, smode)
    assert res["info"] == 0 and res["nelim"] > 0
    _check(res, p, smode)


@pytest.mark.parametrize("smode", ["fp64_packed", "fp32_packed"])
def test_batched_form_of_few_rows(ctx, smode):
    from paper_1305_2353_gb300 import ctp
    shapes = [(p + m, p) for p in (1, 7, 16, 32, 33, 90, 200) for m in (0, 1, 5, 31, 32, 33, 65)]
    b = ctp.Batch(ctx, [inputs.supernode(n, p, seed=n, zero_diag_frac=0.2) for n, p in shapes],
                  [p for _, p in shapes], ctp.options(pivot="restricted", smode=smode))
    b.run()
    assert np.all(b.flags() == 0)
    for k, (n, p) in enumerate(shapes):
        if n > p:
            _check(b.result(k), p, smode)


@pytest.mark.parametrize("n,p", [(12, 4), (24, 8), (40, 16), (53, 33), (65, 33), (100, 40), (200, 64), (600, 200)])
@pytest.mark.parametrize("smode", ["fp64_packed", "none"])
def test_workspace_of_small_fronts(ctx, n, p, smode):
    """Per front: the compressed matrix, D^-1 and, with a Form, W21 of up to 32 rows or the slices of two
    operands, 16.5 bytes an entry with rows rounded up to 8 and pivots to 32, and 1040
    bytes per tile; two K blocks of slices more where the Solve may be blocked (p > 32);
    each piece rounded up to 256 bytes, and the plan's tables."""
    from paper_1305_2353_gb300 import ctp
    A = inputs.supernode(n, p, seed=1)
    nb, m = 64, n - p
    b = ctp.Batch(ctx, [A] * nb, [p] * nb, ctp.options(smode=smode))
    want = 8 * p * p + 16 * p + 16 + 4 * p + 4 * 256 + 2048
    r8 = lambda x: -(-x // 8) * 8  # noqa: E731
    if smode != "none":
        if m <= 32:
            want += 8 * m * p + 256
        else:
            tiles = -(-m // 128) * (-(-m // 128) + 1)
            want += 33 * r8(m) * (-(-p // 32) * 32) + 8 * m + 6 * 256 + 1040 * tiles
    if p > 32:
        tiles = -(-m // 128) * -(-(p - 32) // 64)
        want += 16.5 * 32 * (r8(m) + r8(p)) + 4 * n + 6 * 256 + 1040 * tiles
    assert b.ws.numel() / nb <= want

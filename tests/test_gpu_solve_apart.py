"""The large blocked Solve, whose columns are moved and scaled in passes of their own:
2x2 pairs across the scaling pass's 16 columns and the blocks' 32, zero pivots,
delayed columns, columns that stay and that move.  Against the oracle, with the
parity bars of test_gpu_supernode.compare."""
import pytest

from oracle import oracle as O
from paper_1305_2353_gb300 import inputs
from test_gpu_supernode import compare, ctx, run_gpu  # noqa: F401  (ctx is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p", [(23700, 256), (46300, 130), (92100, 66)])  # just above 6e6 entries
@pytest.mark.parametrize("pivot,zero_diag", [("relaxed", 0.0), ("relaxed", 0.4), ("strict", 0.2)])
def test_columns_apart(ctx, n, p, pivot, zero_diag):
    assert (n - p) * p >= 6000000
    A = inputs.supernode(n, p, seed=p, scale_cols=p // 16, scale=1e-7, zero_diag_frac=zero_diag)
    A[:, 3] = 0.0
    A[3, :] = 0.0
    got = run_gpu(ctx, A, p, pivot)
    compare(O.factor(A, p, pivot, log_cap=400000), got, p, A)

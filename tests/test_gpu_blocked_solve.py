"""The blocked FP64 Solve (32-column blocks, tensor-core updates from digit slices) at
the edges of its tiles (32 and 128 rows, 64 columns) and blocks: 2x2 pivots cut by a
block boundary, zero pivots, delayed columns, blocks past the last pivot, pivots
past the blocks, rows that take FP64 multiply-adds.  Against the oracle, with the
parity bars of test_gpu_supernode.compare."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1305_2353_gb300 import inputs
from test_gpu_supernode import compare, ctx, run_gpu  # noqa: F401  (ctx is a fixture)

pytestmark = pytest.mark.gpu

CASES = [  # m, p, pivot, fraction of zero diagonals, diagonal boost
    (1, 129, "relaxed", 0.5, 0.0), (31, 160, "relaxed", 0.5, 0.0), (33, 200, "restricted", 0.5, 0.0),
    (127, 256, "relaxed", 0.5, 0.0), (129, 255, "relaxed", 0.3, 0.0), (300, 225, "restricted", 0.0, 0.0),
    (5000, 65, "restricted", 0.5, 0.0), (17000, 64, "relaxed", 0.5, 0.0),
    (1, 177, "strict", 0.5, 0.0), (130, 256, "strict", 0.3, 0.0),
    (200, 192, "strict", 0.0, 400.0),   # strict accepts all columns: the tail eliminates most
    (260, 256, "single_row", 0.2, 300.0)]


def _matrix(m, p, zero, boost):
    A = inputs.supernode(p + m, p, seed=p + m, zero_diag_frac=zero, diag_boost=boost, scale_cols=p // 40, scale=1e-6)
    A[:, 5] = 0.0
    A[5, :] = 0.0
    # strongly coupled neighbours with small diagonals: 2x2 pivots at odd positions
    for j in range(7, p - 1, 2):
        A[j, j] = A[j + 1, j + 1] = 1e-3
        A[j + 1, j] = A[j, j + 1] = boost + 60.0
    return A


@pytest.mark.parametrize("m,p,pivot,zero,boost", CASES)
def test_blocked_solve(ctx, m, p, pivot, zero, boost):
    A = _matrix(m, p, zero, boost)
    compare(O.factor(A, p, pivot, log_cap=400000), run_gpu(ctx, A, p, pivot), p, A)


def test_blocked_solve_wide_rows(ctx):
    """Rows of A21 whose entries scatter over 2^60 are as good as the oracle's."""
    m, p = 300, 160
    A = _matrix(m, p, 0.3, 0.0)
    rng = np.random.default_rng(1)
    A[p + 40:p + 120] *= 2.0 ** rng.uniform(-60, 0, (80, p))
    compare(O.factor(A, p, "restricted", log_cap=400000), run_gpu(ctx, A, p, "restricted"), p, A)

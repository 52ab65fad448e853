"""Full-column threshold pivoting at the edges of the kernel's layouts: the rows of
A21 held in shared memory (200 KiB a CTA) or streamed, one CTA or many, warps with
a full, a part-filled and no 32-row group, no A21 rows at all; pivots of every
kind.  Against the oracle, with the parity bars of test_gpu_supernode.compare."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1305_2353_gb300 import inputs
from test_gpu_supernode import compare, ctx, run_gpu  # noqa: F401  (ctx is a fixture)

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (2, 2), (64, 64), (256, 256),   # no A21 rows
         (9, 8), (33, 1), (96, 64), (161, 129),  # one row, one CTA, part-filled groups
         (2300, 256),                            # fewer 32-row CTAs than SMs
         (256 + 100 * 152, 256),                 # exactly 200 KiB of rows per CTA on 152 SMs
         (256 + 100 * 152 + 1, 256),             # one row more: streamed
         (25000, 255), (150001, 33)]               # streamed rows end inside a group


def _matrix(n, p):
    # tiny rows and columns (delays, zero pivots below `small`), zero diagonals (2x2 pivots)
    A = inputs.supernode(n, p, seed=31 * p + n % 97, scale_cols=p // 16, scale=1e-7, zero_diag_frac=0.1)
    if p >= 8:
        A[:, 3] = 0.0
        A[3, :] = 0.0
    return A


@pytest.mark.parametrize("n,p", SIZES)
def test_tpp_layout(ctx, n, p):
    A = _matrix(n, p)
    compare(O.factor(A, p, "tpp", log_cap=400000), run_gpu(ctx, A, p, "tpp"), p, A)

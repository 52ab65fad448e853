"""Full-column threshold pivoting where its look-ahead on the next candidate can go
wrong: candidates accepted as 1x1 or 2x2, rejected, or zero when looked ahead, sweeps
that wrap, and the grid sizes at which the exchange of maxima changes its reads
(32, 64 and more CTAs).  Against the oracle, with the parity bars of
test_gpu_supernode.compare."""
import numpy as np
import pytest

from oracle import oracle as O
from test_gpu_supernode import compare, ctx, run_gpu  # noqa: F401  (ctx is a fixture)

pytestmark = pytest.mark.gpu


def _matrix(kind, n, p):
    rng = np.random.default_rng(1000 * p + n)
    A = rng.uniform(-1, 1, (n, p))
    A[:p] = (A[:p] + A[:p].T) / 2
    k = np.arange(p)
    if kind == "accept":      # every candidate passes as it comes
        A[k, k] = 4.0 * p * rng.choice([-1, 1], p)
    elif kind == "pairs":     # a rejection, then a 2x2 pivot with the column before
        A[k, k] = 0.0
        o = k[1::2]
        A[o, o - 1] = A[o - 1, o] = 4.0 * p
    elif kind == "late":      # every third column passes only once the others are gone
        A[k, k] = 8.0 * p
        s = k[::3]
        A[s, s] = 1e-4
        A[p:, s] *= 1e-2
        A[np.ix_(s, s)] *= 1e-4
        A[s, s] = 1e-4
    elif kind == "zeros":     # zero columns between accepted ones, single and in runs
        A[k, k] = 4.0 * p
        z = k[(k % 7 == 3) | ((k // 8) % 4 == 2)]
        A[:, z] = 0.0
        A[z, :] = 0.0
    elif kind == "delay":     # the second half never passes: a last sweep without a pivot
        h = k[p // 2:]
        A[k, k] = 4.0 * p
        A[np.ix_(h, h)] = 0.0
        A[np.ix_(h, k[:p // 2])] = A[np.ix_(k[:p // 2], h)] = 0.0
        if n > p:
            A[p:, h] = 1.0
    return A


@pytest.mark.parametrize("kind", ["accept", "pairs", "late", "zeros", "delay"])
@pytest.mark.parametrize("n,p", [(40, 8), (300, 31), (700, 64), (64 + 33 * 32, 64), (64 + 64 * 32 + 1, 64),
                                 (256 + 99 * 152, 256), (1999, 256), (20000, 256)])
def test_lookahead(ctx, kind, n, p):
    A = _matrix(kind, n, p)
    compare(O.factor(A, p, "tpp", log_cap=400000), run_gpu(ctx, A, p, "tpp"), p, A)

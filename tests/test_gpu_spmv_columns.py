"""The sparse residual over column lengths from one entry to a full column and matrices of few
and of many columns (how many lanes share a column depends on both).

With B = A X rounded, every row of the residual is at most a few roundings of its own
row of |A||X|, so the backward errors vanish against any row left out or counted twice.
"""
import ctypes

import numpy as np
import pytest
import scipy.sparse as sp

from test_gpu_supernode import ctx  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _matrix(N, per, long, seed):
    """Lower triangle in compressed columns: about `per` entries a column, and columns of the lengths
    in `long` (as many as there are rows below)."""
    rng = np.random.default_rng(seed)
    count = rng.integers(1, max(2, 2 * per), N)
    count[rng.choice(N, len(long), replace=False)] = long
    cols = []
    for j in range(N):
        k = min(int(count[j]), N - j)
        cols.append(np.unique(np.r_[j, j + rng.choice(N - j, k - 1, replace=False)]) if k > 1 else np.array([j]))
    colptr = np.r_[0, np.cumsum([len(c) for c in cols])].astype(np.int64)
    return colptr, np.concatenate(cols).astype(np.int32), rng.standard_normal(int(colptr[-1]))


@pytest.mark.parametrize("N,per,long", [(1, 1, []), (33, 3, [1, 20]), (700, 20, [63, 64, 65, 500]), (3000, 2, [129, 3000]),
                                        (3000, 40, [2048, 2049]), (20000, 6, [64, 65, 128, 257, 9000]),
                                        (80000, 4, [64, 65, 66, 20000]), (80000, 24, [129, 130])])
@pytest.mark.parametrize("nrhs", [1, 9])
def test_residual_of_any_column_length(ctx, N, per, long, nrhs):
    colptr, rowind, val = _matrix(N, per, long, N + per)
    L = sp.csc_matrix((val, rowind, colptr), shape=(N, N))
    A = L + sp.tril(L, -1).T if N > 1 else L
    X = np.random.default_rng(3).standard_normal((nrhs, N))
    B = (A @ X.T).T.copy()
    d = [torch.from_numpy(x).cuda() for x in (colptr, rowind, val, B, X)]
    berr = torch.empty(nrhs, dtype=torch.float64, device="cuda")
    ws = torch.empty(8 * (N * nrhs + N + 8 * nrhs) + 8192, dtype=torch.uint8, device="cuda")
    P = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    rc = ctx.lib.ctp_backward_error_csc(ctx.handle, N, P(d[0]), P(d[1]), P(d[2]), nrhs, P(d[3]), N, P(d[4]), N, P(berr),
                                        P(ws), ws.numel(), None)
    assert rc == 0
    # both products round each of a row's entries once: the row's count times 2^-52 of |A||X|
    rows = np.diff((abs(A) > 0).tocsr().indptr).max()
    absx = (abs(A) @ np.abs(X).T).max(0)
    den = abs(A).sum(1).max() * np.abs(X).max(1) + np.abs(B).max(1)
    assert np.all(berr.cpu().numpy() <= (rows + 2) * 2.0 ** -52 * absx / den)
    # and the row sums and norms are the matrix's
    B[:, 0] += 1.0
    d[3].copy_(torch.from_numpy(B))
    assert ctx.lib.ctp_backward_error_csc(ctx.handle, N, P(d[0]), P(d[1]), P(d[2]), nrhs, P(d[3]), N, P(d[4]), N, P(berr),
                                          P(ws), ws.numel(), None) == 0
    den = abs(A).sum(1).max() * np.abs(X).max(1) + np.abs(B).max(1)
    assert np.allclose(berr.cpu().numpy(), 1.0 / den, rtol=1e-6)

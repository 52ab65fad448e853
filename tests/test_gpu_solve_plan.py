"""The repacked multifrontal solve at the edges of its groups (64 pivots), chunks (32
rows) and right-hand-side passes (1, 2, 4, 8, 16), against the front-list solve with
the same factors; and the sparse residual's long columns."""
import numpy as np
import pytest

from paper_1305_2353_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1305_2353_gb300 import build, ctp
    build.build()
    return ctp.Context(0)


# leaf boxes of 200 points and root planes of 81 to 196 columns: groups of 64 that end
# inside a panel (relaxed and TPP accept up to 256 columns a panel) or span many
# (strict accepts a dozen); plane fronts with and without rows below
@pytest.mark.parametrize("k,pivot,leaf", [(9, "relaxed", 200), (14, "strict", 64), (13, "tpp", 200), (4, "strict", 64)])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 7, 16, 33])
def test_repacked_solve(ctx, k, pivot, leaf, nrhs):
    from paper_1305_2353_gb300 import ctp
    cp, ri, v = inputs.laplacian_3d(k, 3.1)
    perm, blocks = inputs.nested_dissection_3d(k, leaf)
    mf = ctp.Multifrontal(ctx, cp, ri, v, perm, blocks)
    mf.factor(ctp.options(pivot=pivot))
    N = mf.N
    B = np.random.default_rng(nrhs).standard_normal((N, nrhs))
    X1, X2 = ctp.colmajor(B), ctp.colmajor(B)
    mf.solve(X1, mf.refine_workspace(nrhs))
    ctp.solve(ctx, mf.fronts, mf.nf, N, nrhs, X2, N,
              ctp.solve_workspace(ctx, int(mf.info()["n"].max()), nrhs))
    x1, x2 = ctp.to_numpy(X1), ctp.to_numpy(X2)
    # both solves carry the factors' error amplified by the matrix (condition below 1e4)
    assert np.abs(x1 - x2).max() <= 1e-10 * np.abs(x2).max()


@pytest.mark.parametrize("nrhs", [1, 9])
def test_residual_with_long_columns(ctx, nrhs):
    """Columns with more entries than a lane walks alone (64) and short ones in one matrix."""
    from paper_1305_2353_gb300 import ctp
    N = 333
    rng = np.random.default_rng(3)
    M = np.diag(rng.uniform(2.0, 3.0, N))
    M[1:, 0] = M[0, 1:] = rng.standard_normal(N - 1) * 0.1
    M[71:200, 70] = rng.standard_normal(129) * 0.1
    M[70, 71:200] = M[71:200, 70]
    r, c = np.nonzero(np.tril(M).T)  # column by column
    colptr = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=N))])
    perm = np.array([j for j in range(N) if j not in (0, 70)] + [70, 0], np.int32)
    blocks = np.array(list(range(0, N - 2, 50)) + [N - 2, N], np.int64)
    mf = ctp.Multifrontal(ctx, colptr, c.astype(np.int32), M[c, r], perm, blocks)
    mf.factor(ctp.options())
    B = rng.standard_normal((N, nrhs))
    dB, X = ctp.colmajor(B), ctp.colmajor(np.zeros_like(B))
    hist, _ = mf.refine(dB, X, mf.refine_workspace(nrhs))
    want = np.linalg.solve(M, B)
    assert hist[-1].max() <= 1e-14
    assert np.abs(ctp.to_numpy(X) - want).max() <= 1e-12 * np.abs(want).max()
    # a wrong solution has the backward error numpy computes for it
    Y = B * 0.5
    dY, berr = ctp.colmajor(Y), torch.zeros(nrhs, dtype=torch.float64, device="cuda")
    import ctypes
    ws = mf.refine_workspace(nrhs)
    assert ctx.lib.ctp_backward_error_csc(
        ctx.handle, N, *(ctypes.c_void_p(t.data_ptr()) for t in (mf.d_colptr, mf.d_rowind, mf.d_val)), nrhs,
        ctypes.c_void_p(dB.data_ptr()), N, ctypes.c_void_p(dY.data_ptr()), N, ctypes.c_void_p(berr.data_ptr()),
        ctypes.c_void_p(ws.data_ptr()), ws.numel(), None) == ctp.CTP_OK
    res = np.abs(B - M @ Y).max(0)
    den = np.abs(M).sum(1).max() * np.abs(Y).max(0) + np.abs(B).max(0)
    assert np.allclose(berr.cpu().numpy(), res / den, rtol=1e-12)

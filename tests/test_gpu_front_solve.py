"""The front-list solve at the edges of its steps (8 pivots), warps (32), row tiles and
right-hand-side groups, on fronts made up here: 2x2 blocks across every such edge,
delayed columns, unread slots filled with NaN."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1305_2353_gb300 import build, ctp
    build.build()
    return ctp.Context(0)


def _front(n, p, e, seed):
    """L (n x e, unit lower) and D (e x e) of one front, their storage and the variables."""
    rng = np.random.default_rng(seed)
    L = np.tril(rng.uniform(-1, 1, (n, e)) / max(e, 1) ** 0.5, -1) + np.eye(n, e)
    D = np.diag(rng.choice([-1.0, 1.0], e) * rng.uniform(1, 2, e)) if e else np.zeros((0, 0))
    piv = np.ones(p, np.int32)
    piv[e:] = 3
    # pairs that straddle the edges of steps and warps, and pairs inside them
    for a in [k for k in (7, 15, 31, 63, 95, 127, 191, 223, 3, 40, 100, 252) if k + 1 < e]:
        d = rng.uniform(-0.5, 0.5)
        D[a:a + 2, a:a + 2] = [[d, 1.0], [1.0, -d]]
        piv[a], piv[a + 1] = 2, 0
        L[a + 1, a] = 0.0
    A = np.full((n, p), np.nan)
    A[:, :e] = np.where(np.arange(n)[:, None] > np.arange(e), L, np.nan)
    Dp = np.zeros(2 * p)
    for q in range(e):
        Dp[2 * q] = D[q, q]
        if piv[q] == 2:
            Dp[2 * q + 1] = A[q + 1, q] = D[q + 1, q]
    return L, D, A, Dp, piv, rng.permutation(p).astype(np.int32), rng.permutation(n).astype(np.int32)


@pytest.mark.parametrize("e,delayed", [(0, 5), (1, 0), (2, 1), (7, 0), (8, 0), (9, 3), (31, 0), (32, 0), (33, 0),
                                       (64, 0), (130, 7), (255, 0), (255, 1), (256, 0)])
@pytest.mark.parametrize("below", [0, 1, 32, 45, 700])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 9])
def test_one_front(ctx, e, delayed, below, nrhs):
    from paper_1305_2353_gb300 import ctp
    p, n = e + delayed, e + delayed + below
    L, D, A, Dp, piv, perm, rows = _front(n, p, e, 7 * e + below)
    dev = [ctp.colmajor(A), torch.tensor(perm, device="cuda"), torch.tensor(piv, device="cuda"),
           torch.tensor(Dp, device="cuda"), torch.tensor([e], dtype=torch.int32, device="cuda"),
           torch.tensor(rows, device="cuda")]
    f = (ctp.SFront * 1)()
    f[0].n, f[0].p, f[0].ldl = n, p, n
    f[0].L, f[0].perm, f[0].piv, f[0].D, f[0].nelim, f[0].rows = [t.data_ptr() for t in dev]
    B = np.random.default_rng(nrhs).standard_normal((n, nrhs))
    X = ctp.colmajor(B)
    ctp.solve(ctx, f, 1, n, nrhs, X, n, ctp.solve_workspace(ctx, n, nrhs))
    var = np.concatenate([rows[perm], rows[p:]])  # variable of front row q after pivoting
    x, b = ctp.to_numpy(X)[var], B[var]
    F = np.eye(n)
    F[:, :e] = L
    T = np.eye(n)
    T[:e, :e] = D
    # substitution is backward stable: |b - F T F' x| <= gamma_3n |F||T||F'||x|
    # (Higham, Accuracy and Stability, Theorems 8.5 and 9.4); the explicit 2x2
    # solve of blocks with condition below 2 adds a few roundings to its 3n
    aF = np.abs(F)
    bound = (3 * n + 40) * np.finfo(float).eps * (aF @ (np.abs(T) @ (aF.T @ np.abs(x))) + np.abs(b))
    assert (np.abs(b - F @ (T @ (F.T @ x))) <= bound).all()

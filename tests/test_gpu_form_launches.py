"""An FP64 Form of more tiles than one launch takes: every launch's tiles are there, also
those whose entries digits do not serve, and the workspace does not grow with S.

Tolerance, entry by entry: (2 e + 8) 2^-53 |W21||L21|^T, as in test_gpu_form_fp64.
"""
import pytest

from test_gpu_supernode import ctx  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_form_of_several_launches(ctx):
    from paper_1305_2353_gb300 import ctp
    p, m = 8, 65601
    n = p + m
    g = torch.Generator(device="cuda").manual_seed(3)
    B = torch.randn((p, m), dtype=torch.float64, device="cuda", generator=g)
    # rows large in the first or in the last half of the pivots only
    tiny = torch.zeros((p, m), dtype=torch.bool, device="cuda")
    for rows in (range(0, 200), range(m - 300, m), range(1000, m, 997)):
        r = torch.tensor(list(rows), device="cuda")
        tiny[:p // 2, r[0::2]] = True
        tiny[p // 2:, r[1::2]] = True
    B[tiny] *= 2.0 ** -50
    A = torch.zeros((p, n), dtype=torch.float64, device="cuda")
    A[:, p:] = B
    d = torch.linspace(1.0, 2.0, p, dtype=torch.float64, device="cuda")
    A[:, :p] = torch.diag(d)
    i32 = lambda k: torch.zeros(k, dtype=torch.int32, device="cuda")  # noqa: E731
    perm, piv, D, ne = i32(p), i32(p), torch.zeros(2 * p, dtype=torch.float64, device="cuda"), i32(1)
    S = torch.full((m, m), 7.0, dtype=torch.float64, device="cuda")  # column-major: S[j, i]
    opt = ctp.options(pivot="restricted", smode="fp64")
    ws = ctx.factor_supernode(A, n, p, n, opt, perm, piv, D, ne, S, m)
    torch.cuda.synchronize()
    assert ctx.read_info(ws) == 0 and int(ne[0]) == p
    Dm = torch.diag(D[0::2])
    for k in range(p - 1):
        if int(piv[k]) == 2:  # the first column of a 2x2 pivot
            Dm[k, k + 1] = Dm[k + 1, k] = D[2 * k + 1]
    L = A[:, p:].t().contiguous()  # m x p
    W = L @ Dm
    bound_w = (2 * p + 8) * 2.0 ** -53 * (L.abs() @ Dm.abs())
    for j in range(0, m, 2048):
        k = min(2048, m - j)
        want, bound = L[j:j + k] @ W[j:].t(), L[j:j + k].abs() @ bound_w[j:].t()
        got = S[j:j + k, j:]
        low = torch.ones((k, m - j), dtype=torch.bool, device="cuda").triu()
        assert bool(((got - want).abs() <= bound)[low].all()), j
        if j + k <= m:
            assert bool((got[~low] == 7.0).all())


@pytest.mark.parametrize("smode", ["fp64_packed", "fp32_packed"])
def test_workspace_of_a_large_form(ctx, smode):
    """Slices of two operands of m x p entries, 16.5 bytes each, one block of Y's columns
    within them, L11's and the compressed matrix (less than 64 MB), and 1040 bytes for each of at most
    2^18 tiles: not for each tile of S."""
    from paper_1305_2353_gb300 import ctp
    n, p = 400000, 256
    got = ctx.workspace_size(n, p, ctp.options(pivot="strict", smode=smode))
    assert got <= 2 * 16.5 * (n - p + 8) * p + 8 * n + 1040 * 2 ** 18 + (64 << 20)

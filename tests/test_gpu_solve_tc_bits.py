"""The tensor-core Solve's operands bit for bit, seen through supernodes whose product
x_e Z is exact: the BF16 pieces of x_e (each the rounding, through FP32, of what the
earlier ones left exactly), and Z's recurrence, which is the FP64 Solve's own."""
import numpy as np
import pytest

from test_gpu_supernode import ctx  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _run(ctx, A, p, solve):
    from paper_1305_2353_gb300 import ctp
    sn = ctp.Supernode(ctx, A, p, ctp.options(pivot="restricted", prec="bf16x6", smode="fp32", solve=solve))
    sn.run()
    torch.cuda.synchronize()
    return sn.result()


def _pieces(v):
    out, r = [], v.copy()
    for _ in range(3):
        b = torch.from_numpy(r.astype(np.float32)).to(torch.bfloat16).to(torch.float64).numpy()
        out.append(b)
        r = r - b
    return out


def _values(rng):
    n = 3000
    v = rng.standard_normal(n) * 2.0 ** rng.uniform(-60, 60, n)
    # third pieces next to a rounding boundary: what is below 2^-48 of the value decides
    one = 1.0 + rng.integers(0, 128, n) * 2.0 ** -7
    two = rng.integers(65, 127, n) * 2.0 ** -15 * rng.choice([-1, 1], n)
    three = (rng.integers(128, 255, n) + 0.5) * 2.0 ** -25 * rng.choice([-1, 1], n)
    tie = (one + two + three + rng.choice([-1, 0, 1], n) * 2.0 ** -rng.integers(49, 53, n))
    tie *= 2.0 ** rng.integers(-50, 50, n) * rng.choice([-1, 1], n)
    return np.concatenate([v, tie, [0.0, 1.0, -3.0, 2.0 ** -70, -1.7 * 2.0 ** -66, 1.3 * 2.0 ** 70, 255.5, 511.75]])


def test_pieces_of_x(ctx):
    """A11 = [[2, 1], [1, 1]] is eliminated column 1 first, both pivots 1: the second
    column of L21 is x_0 - x_1, and with x_1 the first piece of x_0 what is left is the sum of
    the other two.  Of values for which FP32 holds that sum exactly (all but those whose
    remainder happens to be far smaller than the second piece's last place)."""
    v = _values(np.random.default_rng(4))
    p0, p1, p2 = _pieces(v)
    exact = (p1 + p2).astype(np.float32).astype(np.float64) == p1 + p2
    assert exact.mean() > 0.98
    v, p0, p1, p2 = v[exact], p0[exact], p1[exact], p2[exact]
    A = np.zeros((2 + len(v), 2), order="F")
    A[:2] = [[2.0, 1.0], [1.0, 1.0]]
    A[2:, 0], A[2:, 1] = v, p0
    res = _run(ctx, A, 2, "tc")
    assert res["nelim"] == 2 and list(res["perm"]) == [1, 0] and np.all(res["piv"] == 1)
    assert np.array_equal(res["A"][2:, 1], p1 + p2)


@pytest.mark.parametrize("seed", range(6))
def test_z_recurrence_of_2x2_pivots(ctx, seed):
    """Two 2x2 pivots and a last column whose entry of Z is what two cancelling products
    leave: only the FP64 Solve's association gives the FP64 Solve's value."""
    rng = np.random.default_rng(seed)
    t, s = rng.uniform(1, 2, 2)
    A = np.zeros((5 + 40, 5), order="F")
    A[1, 0] = A[0, 1] = A[3, 2] = A[2, 3] = 1.0
    A[2, 1] = A[1, 2] = t
    A[3, 1] = A[1, 3] = -t
    A[4, 2] = A[2, 4] = A[4, 3] = A[3, 4] = s
    A[4, 4] = 16.0
    A[5:, 0] = 2.0 ** rng.integers(-3, 4, 40)
    want, got = _run(ctx, A, 5, "fp64"), _run(ctx, A, 5, "tc")
    assert want["nelim"] == 5 and np.array_equal(want["perm"], np.arange(5))
    w = want["A"][5:, 4]
    assert np.all(np.abs(w) < 1e-14) and np.any(w != 0.0)
    assert np.all(np.abs(got["A"][5:, 4] - w) <= 2.0 ** -15 * np.abs(w))

"""The FP64 Solve in tiles of 8, 16 and 32 rows, at the sizes where the tile changes (as many
32-row tiles as 152 SMs and twice as many; half that when the Solve is blocked) and
at the edges of the tiles; with the Form that reads its operands; single and
batched.  Against the oracle, with the parity bars of test_gpu_supernode.compare and its
1e-11 on an FP64 S."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1305_2353_gb300 import inputs
from test_gpu_supernode import compare, ctx, run_gpu  # noqa: F401  (ctx is a fixture)

pytestmark = pytest.mark.gpu


def _check_s(ref, S, p):
    e = ref["nelim"]
    want = np.tril(O.form(ref["A"][p:, :e], ref["piv"][:e], ref["D"]))
    assert np.allclose(np.tril(S), want, rtol=1e-11, atol=1e-11 * max(np.abs(want).max(), 1))


KINDS = [(1, "strict"), (31, "relaxed"), (64, "strict"), (96, "relaxed"),
         (160, "relaxed"), (200, "strict")]  # the last two blocked: their tile changes below 5000 rows only
SIZES = [1, 7, 8, 9, 16, 17, 33, 2432, 2433, 4864, 4865]


@pytest.mark.parametrize("m,p,pivot", [(m, *k) for k in KINDS for m in SIZES] +
                         [(m, *k) for k in KINDS[1:3] for m in (9728, 9729)])
def test_rows_per_tile(ctx, m, p, pivot):
    A = inputs.supernode(m + p, p, seed=m + p, scale_cols=p // 16, scale=1e-7, zero_diag_frac=0.2 if p > 1 else 0.0)
    ref = O.factor(A, p, pivot, log_cap=200000)
    got = run_gpu(ctx, A, p, pivot, smode="fp64")
    compare(ref, got, p, A)
    _check_s(ref, got["S"], p)


# classes of few tiles (8 rows), of some (16) and of many (32), whole and blocked
@pytest.mark.parametrize("shapes", [[(90, 40), (77, 33), (41, 40)], [(3000, 250), (2000, 200)],
                                    [(900, 70)] * 9 + [(5000, 256)], [(1500, 64)] * 220])
@pytest.mark.parametrize("pivot", ["strict", "restricted"])
def test_rows_per_tile_batch(ctx, shapes, pivot):
    from paper_1305_2353_gb300 import ctp
    import torch
    fr = [inputs.supernode(n, p, seed=13 * k + p, zero_diag_frac=0.05) for k, (n, p) in enumerate(shapes)]
    b = ctp.Batch(ctx, fr, [a.shape[1] for a in fr], ctp.options(pivot=pivot))
    b.run()
    torch.cuda.synchronize()
    assert np.all(b.flags() == 0)
    for k in range(0, len(fr), 7 if len(fr) > 50 else 1):
        p = fr[k].shape[1]
        compare(O.factor(fr[k], p, pivot, log_cap=200000), b.result(k), p, fr[k])

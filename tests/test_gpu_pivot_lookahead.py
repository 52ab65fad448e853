"""The compressed pivot search where its look-ahead on the next candidate applies and
where it does not (accepted, rejected, zero, with a partner, a wrapped sweep), on every
cluster width and at the sizes at which columns begin to be split between warps;
and batches of few fronts, whose searches move to wider clusters.  Against the oracle,
with the parity bars of test_gpu_supernode.compare."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1305_2353_gb300 import inputs
from test_gpu_supernode import compare, ctx, run_gpu  # noqa: F401  (ctx is a fixture)
from test_gpu_tpp_lookahead import _matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["accept", "pairs", "late", "zeros", "delay"])
@pytest.mark.parametrize("pivot", ["relaxed", "strict"])
@pytest.mark.parametrize("n,p,G", [(40, 8, 1), (90, 40, 1), (90, 40, 2), (400, 64, 4), (400, 65, 8),
                                   (700, 130, 16), (1000, 256, 8), (1000, 256, 16)])
def test_pivot_lookahead(ctx, kind, pivot, n, p, G):
    from paper_1305_2353_gb300 import ctp
    A = _matrix(kind, n, p)
    ctx.tune_set(ctp.TUNE_FACTOR_G, G)
    try:
        got = run_gpu(ctx, A, p, pivot)
    finally:
        ctx.tune_set(ctp.TUNE_FACTOR_G, 0)
    compare(O.factor(A, p, pivot, log_cap=400000), got, p, A)


@pytest.mark.parametrize("pivot", ["strict", "restricted"])
@pytest.mark.parametrize("shapes", [
    [(700, 256)], [(300, 33)], [(300, 64), (400, 65), (90, 32)],          # each class moves as far as it wants
    [(500, 129)] * 7, [(500, 129)] * 8,                                  # 112 CTAs on 16 each, and one front more
    [(200, 40)] * 28 + [(600, 200)], [(200, 40)] * 113])                 # some classes move, none does
def test_few_fronts(ctx, pivot, shapes):
    from paper_1305_2353_gb300 import ctp
    import torch
    fr = [inputs.supernode(n, p, seed=11 * k + p, zero_diag_frac=0.05) for k, (n, p) in enumerate(shapes)]
    b = ctp.Batch(ctx, fr, [a.shape[1] for a in fr], ctp.options(pivot=pivot))
    b.run()
    torch.cuda.synchronize()
    assert np.all(b.flags() == 0)
    for k, A in enumerate(fr):
        p = A.shape[1]
        compare(O.factor(A, p, pivot, log_cap=200000), b.result(k), p, A)

"""The multifrontal factorization with two batches of fronts in flight, against one
batch at a time (as a profiled call runs): the same pivots, the same solution; on
streams other than the default one, and again with the same object (its staging kept)."""
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


# trees with one front on a level (k = 2), a few, and hundreds; pivoting that delays
@pytest.mark.parametrize("k,leaf,pivot,prec", [(2, 4, "strict", "fp64"), (5, 20, "strict", "fp64"),
                                               (9, 30, "restricted", "fp64"), (14, 64, "strict", "bf16x6"),
                                               (20, 64, "strict", "fp64")])
def test_two_groups(ctx, k, leaf, pivot, prec):
    from paper_1305_2353_gb300 import ctp
    cp, ri, v = inputs.laplacian_3d(k, 3.1)
    perm, blocks = inputs.nested_dissection_3d(k, leaf)
    opt = ctp.options(pivot=pivot, prec=prec)
    N = len(cp) - 1
    B = np.random.default_rng(k).standard_normal((N, 2))
    res = []
    mf = ctp.Multifrontal(ctx, cp, ri, v, perm, blocks)
    for mode in ("profiled", "plain", "stream", "plain"):
        s = torch.cuda.Stream() if mode == "stream" else None
        if mode == "profiled":
            ctx.profile_begin()
        mf.factor(opt, stream=s)
        torch.cuda.synchronize()
        if mode == "profiled":
            ctx.profile_end()
        X = ctp.colmajor(B)
        mf.solve(X, mf.refine_workspace(2))
        res.append((mf.info(), mf.panel_perms(), ctp.to_numpy(X)))
    # mixed factors are good to about 2^-19, FP64 ones to the rounding of the Solve's two
    # forms, both amplified by the matrix (condition below 1e4)
    tol = 1e-9 if prec == "fp64" else 2.0 ** -19 * 1e4
    for info, perms, X in res[1:]:
        for key in ("n", "p", "nelim", "delayed"):
            assert np.array_equal(info[key], res[0][0][key])
        assert len(perms) == len(res[0][1]) and all(np.array_equal(a, b) for a, b in zip(perms, res[0][1]))
        assert np.abs(X - res[0][2]).max() <= tol * np.abs(res[0][2]).max()


def test_two_threads_one_context(ctx):
    """Two factorizations at once, from two threads and on two streams, share the
    context's side streams."""
    import threading
    from paper_1305_2353_gb300 import ctp
    k = 14
    perm, blocks = inputs.nested_dissection_3d(k, 64)
    jobs = []
    for shift in (3.1, 2.7):
        cp, ri, v = inputs.laplacian_3d(k, shift)
        jobs.append((ctp.Multifrontal(ctx, cp, ri, v, perm, blocks), torch.cuda.Stream()))
    opt = ctp.options(pivot="strict")
    want = []
    for mf, _ in jobs:
        mf.factor(opt)
        want.append((mf.info(), mf.panel_perms()))
    errors = []

    def run(mf, s):
        try:
            torch.cuda.set_device(ctx.device)
            for _ in range(5):
                mf.factor(opt, stream=s)
        except Exception as e:  # noqa: BLE001  (reported by the assertion below)
            errors.append(e)

    ts = [threading.Thread(target=run, args=j) for j in jobs]
    [t.start() for t in ts]
    [t.join() for t in ts]
    torch.cuda.synchronize()
    assert not errors
    for (mf, _), (info, perms) in zip(jobs, want):
        got = mf.info()
        for key in ("n", "p", "nelim", "delayed"):
            assert np.array_equal(got[key], info[key])
        assert all(np.array_equal(a, b) for a, b in zip(mf.panel_perms(), perms))

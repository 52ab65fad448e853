"""Batches from several threads at once, on one context and on two (each context orders the
work that goes through its own side streams): results bit for bit those of a single thread."""
import threading

import numpy as np
import pytest

from paper_1305_2353_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("contexts", [1, 2])
def test_batches_from_several_threads(contexts):
    from paper_1305_2353_gb300 import build, ctp
    build.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    ctxs = [ctp.Context(0) for _ in range(contexts)]
    fronts, ps = inputs.batch(count=60, seed=4), [int(p) for p in inputs.batch_shapes(count=60, seed=4)[:, 1]]
    opt = ctp.options(smode="fp64_packed")
    batches = [ctp.Batch(ctxs[k % contexts], fronts, ps, opt) for k in range(4)]
    batches[0].run()
    torch.cuda.synchronize()
    want = [batches[0].A.cpu().numpy(), batches[0].S.cpu().numpy(), batches[0].piv.cpu().numpy()]
    bad = []

    def work(b):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for _ in range(10):
                b.A.copy_(b.A0)
                b.run(stream=s)
                s.synchronize()
                got = [b.A.cpu().numpy(), b.S.cpu().numpy(), b.piv.cpu().numpy()]
                if not all(np.array_equal(x, y) for x, y in zip(got, want)):
                    bad.append(1)

    threads = [threading.Thread(target=work, args=(b,)) for b in batches]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad

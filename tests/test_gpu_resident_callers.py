"""Several host threads, each with a matrix on a stream of its own, solving small
and mid-sized stencil systems at once with the register-resident solver: every
solve ends with the bits of the same solve alone, whatever runs beside it."""
import threading

import numpy as np
import pytest

from paper_1905_06850_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    from paper_1905_06850_gb300 import build as B
    from paper_1905_06850_gb300 import plcg
    B.build()
    plcg.load()
    torch.cuda.set_device(0)
    return plcg


def test_eight_callers(P):
    import torch
    sizes = [(32, 32), (100, 100), (32, 32), (100, 100), (100, 100), (27, 27, 27), (300, 300), (60, 60, 60)]
    jobs = []
    for k, size in enumerate(sizes):
        op = W.stencil2d(*size, shift=0.1) if len(size) == 2 else W.stencil3d(*size, shift=0.1)
        b = torch.tensor(W.rhs(op, np.random.default_rng(k).standard_normal(W.op_size(op))), device="cuda")
        kw = dict(l=1 + k % 3, interval=W.shift_interval(op), rtol=1e-8, prec="fp32" if k in (4, 6) else "fp64")
        A = P.Matrix(op, stream=torch.cuda.Stream())
        alone = torch.zeros_like(b)
        torch.cuda.synchronize()
        r = A.solve(b, alone, **kw)
        assert r.ok
        jobs.append((A, b, kw, alone, r.iters))
    bad = []

    def work(job, xs):
        A, b, kw, alone, iters = job
        results = [A.solve(b, x, check=False, **kw) for x in xs]
        for x, r in zip(xs, results):
            if not (r.ok and r.iters == iters and torch.equal(x, alone)):
                bad.append((A.n, r))

    xs = [[torch.zeros_like(j[1]) for _ in range(12)] for j in jobs]
    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(j, x)) for j, x in zip(jobs, xs)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for j in jobs:
        j[0].close()
    assert not bad

"""A solve's workspace when what its layout depends on changes around it: the
cluster limit moved between a request's submission and its launch."""
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


def case(*size):
    import torch
    op = W.stencil3d(*size, shift=0.5)
    xs = np.random.default_rng(6).standard_normal(W.op_size(op))
    return op, torch.tensor(W.rhs(op, xs), device="cuda"), torch.tensor(xs, device="cuda")


def test_cluster_limit_moved_after_submission(P):
    """Requests sized while the cluster limit is high (lines as they are) start
    after it is back at its default, which pads their lines."""
    import torch
    op, b, xs = case(43, 47, 41)
    first, fb, fx = case(150, 150, 150)   # occupies the one slot while the limit moves
    A, F = P.Matrix(op), P.Matrix(first)
    kw = dict(l=2, interval=(0.5, 12.5), rtol=1e-8, prec="fp32")
    S = P.Server(max_inflight=1)
    x = [torch.zeros_like(b) for _ in range(3)]
    f = torch.zeros_like(fb)
    torch.cuda.synchronize()
    try:
        P.set_cluster_rows(1 << 20)
        t0 = S.submit(F, fb, f, **kw)
        ts = [S.submit(A, b, v, **kw) for v in x]
    finally:
        P.set_cluster_rows()
    assert S.wait(t0).ok
    rs = [S.wait(t) for t in ts]
    S.close()
    A.close()
    F.close()
    assert float((f - fx).norm() / fx.norm()) <= 1e-6
    for r, v in zip(rs, x):
        assert r.ok and float((v - xs).norm() / xs.norm()) <= 1e-6

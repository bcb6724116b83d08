"""A solve's workspace when what its layout depends on changes around it: the
cluster limit moved between a request's submission and its launch, and a device
that does not hold the padded lines."""
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


def test_padding_that_the_device_refuses(P):
    """The solve runs without padded lines; the refusal leaves no pending error
    for the next launch, and the handle does not ask again."""
    import torch
    op, b, xs = case(17, 181, 183)
    n = W.op_size(op)
    kw = dict(l=1, interval=(0.5, 12.5), rtol=1e-8)
    A, B = P.Matrix(op), P.Matrix(op)
    lib = P.load()

    def solve(M, **more):
        x = torch.zeros_like(b)
        r = M.solve(b, x, **{**kw, **more})
        assert r.ok and float((x - xs).norm() / xs.norm()) <= 1e-6
        return P.last_launch()["kernel"]

    padded = solve(B)
    try:
        lib.plcg_debug_limit_workspace(9 * 8 * n + 600_000)   # nine vectors as they are; padded ones are 6 % longer
        plain = solve(A)
        assert plain != padded
        v = W.hetero27_var27(9, 8, 7)   # its set-up and solve launch kernels
        V = P.Matrix(v)
        y = torch.zeros(V.n, dtype=torch.float64, device="cuda")
        assert V.solve(torch.ones_like(y), y, l=1, interval=W.jacobi_shift_interval(v), rtol=1e-8, precond="jacobi").ok
        V.close()
        assert solve(A) == plain and solve(B) == padded   # B holds its padded workspace
        with pytest.raises(P.PlcgError) as e:             # more vectors, and none of them padded
            solve(A, l=4)
        assert e.value.status == P.PLCG_ERR_NOMEM
        S = P.Server()
        x = torch.zeros_like(b)
        torch.cuda.synchronize()
        assert S.wait(S.submit(A, b, x, **kw)).ok
        S.close()
        assert float((x - xs).norm() / xs.norm()) <= 1e-6
    finally:
        lib.plcg_debug_limit_workspace(0)
    assert solve(A) == plain
    solve(A, l=4)             # holds the padded lines too
    assert solve(A) == padded
    A.close()
    B.close()

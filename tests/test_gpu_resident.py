"""The register-resident solver of small and mid-sized stencil systems
(csrc/resident.cuh) at its edges: one warp, a partly filled last warp and CTA,
the step from one to two and four rows per thread, the largest system it takes
and the first it does not.  Against the grid path on the same system: the same
iteration count, FP64 solutions to 1e-10 or, where the solve is sensitive to
the order of the sums, 4 times what the grid path itself moves by between launch
shapes (p(3)-CG on 1 x 2049, shifts on an interval twice its spectrum: 1e-10 to
1.7e-10), FP32 to 1e-5; and both end below the tolerance."""
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


SM = 152
EDGES = [W.stencil2d(31, 1), W.stencil2d(8, 4), W.stencil2d(11, 3), W.stencil3d(5, 3, 9), W.stencil2d(64, 32),
         W.stencil2d(1, 2049), W.stencil2d(101, 97, shift=0.1), W.stencil2d(SM * 448, 1, shift=0.5),
         W.stencil2d(SM * 448 + 1, 1, shift=0.5), W.stencil2d(2, SM * 448 + 1, shift=0.5),
         W.stencil3d(57, 59, 37, shift=0.2), W.stencil2d(4, SM * 448, shift=0.5),
         W.stencil2d(4, SM * 448 + 1, shift=0.5), W.stencil3d(71, 67, 53, shift=0.2)]


@pytest.mark.parametrize("op", EDGES, ids=lambda o: f"{o['nx']}x{o['ny']}x{o['nz']}")
@pytest.mark.parametrize("prec,l", [("fp64", 1), ("fp64", 2), ("fp64", 3), ("fp32", 1), ("fp32", 3)])
def test_resident_edges_match_the_grid_path(P, op, prec, l):
    import torch
    b = torch.tensor(W.rhs(op, np.random.default_rng(5).standard_normal(W.op_size(op))), device="cuda")
    A = P.Matrix(op)
    kw = dict(l=l, interval=W.shift_interval(op), rtol=1e-8, prec=prec)
    x, y = torch.zeros_like(b), torch.zeros_like(b)
    r = A.solve(b, x, **kw)
    resident = P.last_launch()
    g = A.solve(b, y, grid_ctas=1 << 20, **kw)
    assert resident["cluster"] == 0
    if W.op_size(op) <= 4 * SM * 448:
        assert resident["kernel"] != P.last_launch()["kernel"]
    own = 0.0
    if prec == "fp64":
        for ctas in (1, 5):
            z = torch.zeros_like(b)
            A.solve(b, z, grid_ctas=ctas, **kw)
            own = max(own, float((z - y).norm() / y.norm()))
    A.close()
    assert r.ok and g.ok and r.true_relres < 1e-8
    assert abs(r.iters - g.iters) <= (0 if prec == "fp64" else 1)
    assert float((x - y).norm() / y.norm()) <= (max(1e-10, 4 * own) if prec == "fp64" else 1e-5)


@pytest.mark.parametrize("l", [1, 2, 3])
def test_resident_restarts_and_budget(P, l):
    """Poor shifts (square-root breakdowns and restarts), a budget that ends a
    segment at every k, and x0 other than zero, against the grid path."""
    import torch
    c = W.config_2d(nx=40)
    b = torch.tensor(c["b"], device="cuda")
    A = P.Matrix(c["op"])
    x = torch.zeros_like(b)
    r = A.solve(b, x, l=l, interval=(0, 1), rtol=1e-8, max_restarts=200)
    assert r.ok and r.true_relres < 1e-8 and (l == 1 or r.restarts > 0)
    for k in range(0, 9):
        u = torch.linspace(-1, 1, b.numel(), dtype=torch.float64, device="cuda")
        v = u.clone()
        s = A.solve(b, u, l=l, interval=(0, 8), rtol=1e-12, maxit=k, check=False)
        t = A.solve(b, v, l=l, interval=(0, 8), rtol=1e-12, maxit=k, check=False, grid_ctas=1 << 20)
        assert s.status == t.status == P.PLCG_ERR_MAXIT and s.iters == t.iters == k and s.spmvs == t.spmvs
        assert float((u - v).norm() / v.norm()) <= 1e-12
    A.close()

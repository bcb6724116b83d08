"""Classic CG on the whole grid, FP64: x takes a step one sweep late (csrc/solver.cuh,
kLateX), so every way out of a segment has to apply the step that is owed.  A
budget that ends the solve at each k, and an indefinite operator whose (p, A p)
turns negative, against the oracle from a guess that is not zero: one and two rows
per thread, padded lines, one unit of rows a block and several, and the
structured 27-point operator."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1905_06850_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# (grid_ctas: past every launch's own, or few blocks with several units each)
CASES = [(W.stencil2d(40, 40), 1 << 20), (W.stencil2d(200, 200), 1 << 20), (W.stencil2d(202, 131), 3),
         (W.stencil3d(43, 47, 41), 1 << 20), (W.stencil3d(43, 47, 41), 5)]


@pytest.fixture(scope="module")
def P():
    import torch
    from paper_1905_06850_gb300 import build as B
    from paper_1905_06850_gb300 import plcg
    B.build()
    plcg.load()
    torch.cuda.set_device(0)
    return plcg


def compare(P, op, ctas, maxit, status, tol, precond=None):
    import torch
    rng = np.random.default_rng(8)
    n = W.op_size(op)
    b, x0 = W.rhs(op, rng.standard_normal(n)), rng.standard_normal(n)
    ref = O.cg(op, b, x0=x0, rtol=1e-10, maxit=maxit, max_restarts=0, precond=precond)
    x = torch.tensor(x0, device="cuda")
    A = P.Matrix(op)
    r = A.solve(torch.tensor(b, device="cuda"), x, check=False, method="cg", rtol=1e-10, maxit=maxit, max_restarts=0,
                grid_ctas=ctas, precond=precond)
    A.close()
    assert P.last_launch()["cluster"] == 0
    assert r.status == status and r.iters == ref.iters, (r, ref.status, ref.iters)
    d = x.cpu().numpy() - ref.x
    assert np.linalg.norm(d) / np.linalg.norm(ref.x) <= tol
    return ref


@pytest.mark.parametrize("op,ctas", CASES, ids=lambda v: str(v) if isinstance(v, int) else f"{v['nx']}x{v['ny']}x{v['nz']}")
def test_budget_ends_at_each_step(P, op, ctas):
    for k in range(0, 8):   # eight steps' rounding: far below 1e-12
        assert compare(P, op, ctas, k, P.PLCG_ERR_MAXIT, 1e-12).status == O.ORC_ERR_MAXIT


def test_budget_structured_27_point(P):
    op = W.hetero27_var27(19, 17, 23)
    for k in range(0, 6):
        for precond in (None, "jacobi"):
            assert compare(P, op, 1 << 20, k, P.PLCG_ERR_MAXIT, 1e-12, precond).status == O.ORC_ERR_MAXIT


@pytest.mark.parametrize("op,ctas", CASES, ids=lambda v: str(v) if isinstance(v, int) else f"{v['nx']}x{v['ny']}x{v['nz']}")
def test_indefinite_operator_breaks_down(P, op, ctas):
    """Eigenvalues of both signs: (p, A p) turns negative after a step or two; x is
    the last iterate."""
    shifted = dict(op, center=op["center"] * 0.4)
    ref = compare(P, shifted, ctas, 10000, P.PLCG_ERR_BREAKDOWN, 1e-12)
    assert ref.iters >= 1

"""FP32 dots at the ends of the FP32 range in the register-resident solver
(csrc/resident.cuh): an overflowed dot ends the solve as non-finite with x as it
was, and subnormal dots keep their values -- as on the grid path, at one, two and
four rows per thread."""
import numpy as np
import pytest

from paper_1905_06850_gb300 import workloads as W

pytestmark = pytest.mark.gpu
SIZES = [(100, 100), (300, 300), (400, 400)]


@pytest.fixture(scope="module")
def P():
    import torch
    from paper_1905_06850_gb300 import build as B
    from paper_1905_06850_gb300 import plcg
    B.build()
    plcg.load()
    torch.cuda.set_device(0)
    return plcg


def solve(P, op, scale, l, grid_ctas):
    """From x0 = 1: (x, the result, the kernel)."""
    import torch
    b = torch.tensor(W.rhs(op, np.random.default_rng(3).standard_normal(W.op_size(op))), device="cuda")
    x = torch.ones_like(b)
    A = P.Matrix(op)
    r = A.solve(b, x, l=l, interval=(0.5 * scale, 8.5 * scale), rtol=1e-8, prec="fp32", check=False,
                grid_ctas=grid_ctas)
    A.close()
    return x, r, P.last_launch()["kernel"]


@pytest.mark.parametrize("size", SIZES, ids=str)
@pytest.mark.parametrize("l", [1, 2, 3])
def test_overflowed_dots_are_non_finite(P, size, l):
    scale = 1e22   # |A z| of a unit vector z of 1.6e5 entries: products of about 1e39 and more
    op = W.stencil2d(*size, center=4.5 * scale, off=-scale)
    x, r, kernel = solve(P, op, scale, l, 0)
    y, g, other = solve(P, op, scale, l, 1 << 20)
    assert kernel != other
    assert r.status == g.status == P.PLCG_ERR_NONFINITE
    assert bool((x == 1.0).all()) and bool((y == 1.0).all())


@pytest.mark.parametrize("size", SIZES, ids=str)
def test_subnormal_dots_keep_their_values(P, size):
    scale = 2.0 ** -60   # (A z)_g^2 of 1e-39 to 1e-40: subnormal, with a relative rounding of 1e-5 at most each
    op = W.stencil2d(*size, center=4.5 * scale, off=-scale)
    x, r, kernel = solve(P, op, scale, 1, 0)
    y, g, other = solve(P, op, scale, 1, 1 << 20)
    assert kernel != other
    assert g.ok and g.true_relres < 1e-8
    assert r.ok and r.true_relres < 1e-8 and r.restarts == g.restarts and r.iters <= g.iters + 2

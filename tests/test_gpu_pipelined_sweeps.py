"""The sweeps whose operands are copied a unit ahead (StencilPipe in
csrc/solver.cuh), at the sizes where they can go wrong: few blocks, so that each
sweeps many units forwards and backwards, with a ragged last one; lines of one
vector, of a warp's rows and around them; and lines at a padded pitch.  Against the x that b was made from:
the operator is a Laplacian with shift 1/2 (every entry exact in FP32), so a
solve that ends at rtol leaves at most rtol times the condition number, which is
at most (2 * 2 * dim + 1/2) / (1/2)."""
import numpy as np
import pytest

from paper_1905_06850_gb300 import workloads as W

pytestmark = pytest.mark.gpu
RTOL = 1e-8


@pytest.fixture(scope="module")
def P():
    import torch
    from paper_1905_06850_gb300 import build as B
    from paper_1905_06850_gb300 import plcg
    B.build()
    plcg.load()
    torch.cuda.set_device(0)
    return plcg


def grid(nx, ny, nz=1):
    return W.stencil2d(nx, ny, shift=0.5) if nz == 1 else W.stencil3d(nx, ny, nz, shift=0.5)


def interval(nz):
    return 0.5, 8.5 if nz == 1 else 12.5


def check(x, xs, nz, r):
    assert r.ok and r.true_relres < RTOL
    assert float((x - xs).norm() / xs.norm()) <= 1.001 * RTOL * 2 * interval(nz)[1]


@pytest.mark.parametrize("size", [(4, 2311), (64, 147), (128, 65), (132, 71), (260, 37), (4, 7, 331), (36, 20, 17)],
                         ids=str)
@pytest.mark.parametrize("prec,l", [("fp64", 1), ("fp64", 2), ("fp32", 1), ("fp32", 2)])
@pytest.mark.parametrize("ctas", [1, 3])
def test_few_blocks(P, size, prec, l, ctas):
    import torch
    op, nz = grid(*size), (size + (1,))[2]
    xs = np.random.default_rng(2).standard_normal(W.op_size(op))
    b = torch.tensor(W.rhs(op, xs), device="cuda")
    x = torch.zeros_like(b)
    A = P.Matrix(op)
    r = A.solve(b, x, l=l, interval=interval(nz), rtol=RTOL, prec=prec, grid_ctas=ctas)
    A.close()
    check(x, torch.tensor(xs, device="cuda"), nz, r)


@pytest.mark.parametrize("size", [(17, 30941), (30, 97, 183), (31, 131, 137), (65, 97, 91), (1025, 513)], ids=str)
@pytest.mark.parametrize("prec,l", [(p, l) for p in ("fp64", "fp32") for l in (0, 1, 2, 3)])
@pytest.mark.parametrize("ctas", [0, 5])
def test_padded_lines(P, size, prec, l, ctas):
    """Lines that are not whole vectors, held at a padded pitch; from a guess that is not zero (l = 0: classic CG)."""
    import torch
    op, nz = grid(*size), (size + (1,))[2]
    rng = np.random.default_rng(3)
    xs = rng.standard_normal(W.op_size(op))
    b = torch.tensor(W.rhs(op, xs), device="cuda")
    x = torch.tensor(rng.standard_normal(W.op_size(op)), device="cuda")
    A = P.Matrix(op)
    kw = dict(l=l, interval=interval(nz)) if l else dict(method="cg")
    r = A.solve(b, x, rtol=RTOL, prec=prec, grid_ctas=ctas, **kw)
    A.close()
    check(x, torch.tensor(xs, device="cuda"), nz, r)

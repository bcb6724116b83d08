"""The FP64 sweeps whose operands are copied a unit ahead (StencilPipe in
csrc/solver.cuh; l = 1 and 2, lines of whole vectors, 1310720 rows or more) with a
ragged last unit of rows, on few blocks and on the whole grid, lines of one
vector, of a warp's rows and just past it -- and padded ones.  What ran is checked by
the launch's dynamic shared memory, the slots of those copies.  Against the x
that b was made from, as in test_gpu_pipelined_sweeps.py."""
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


def slots(l):
    """Two stages of 8 + 2 l operands, 16 bytes for each of 256 threads, and each warp's edge slots."""
    return 2 * ((8 + 2 * l) * 256 * 16 + 8 * 16)


@pytest.mark.parametrize("size", [(2, 655411), (64, 20483), (130, 10087), (62, 23, 931), (66, 41, 487), (29, 97, 187)],
                         ids=str)
@pytest.mark.parametrize("l", [1, 2])
@pytest.mark.parametrize("ctas", [0, 5])
def test_fp64_copies_ahead(P, size, l, ctas):
    import torch
    dim3 = len(size) == 3
    op = W.stencil3d(*size, shift=0.5) if dim3 else W.stencil2d(*size, shift=0.5)
    top = 12.5 if dim3 else 8.5
    rng = np.random.default_rng(2)
    xs = rng.standard_normal(W.op_size(op))
    b, want = torch.tensor(W.rhs(op, xs), device="cuda"), torch.tensor(xs, device="cuda")
    x = torch.tensor(rng.standard_normal(W.op_size(op)), device="cuda")
    A = P.Matrix(op)
    r = A.solve(b, x, l=l, interval=(0.5, top), rtol=RTOL, grid_ctas=ctas)
    A.close()
    assert P.last_launch()["dyn_smem"] == slots(l)
    assert r.ok and r.true_relres < RTOL
    assert float((x - want).norm() / want.norm()) <= 1.001 * RTOL * 2 * top

"""Every bounded wait of a single solve, made to run out on the host's say (a
target that is never reached, a short poll limit): the barrier of the whole-grid
kernels, and in the register-resident solver (csrc/resident.cuh) the waits for
the other blocks' dots and for neighbours' values, in the first exchange, in the
fill phase and in the recurrences, at every l and number of rows per thread.  Each
solve returns PLCG_ERR_TIMEOUT with all its blocks gone, and the next one on the
same handle succeeds."""
import ctypes as C

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


def run_out(P, on, solve):
    lib = P.load()
    try:
        lib.plcg_debug_set_poll_limit(20000)
        lib.plcg_debug_force_barrier_timeout(on)
        return solve()
    finally:
        lib.plcg_debug_force_barrier_timeout(0)
        lib.plcg_debug_set_poll_limit(0)


def case(size, seed=4):
    import torch
    op = W.stencil2d(*size, shift=0.1) if len(size) == 2 else W.stencil3d(*size, shift=0.1)
    xs = np.random.default_rng(seed).standard_normal(W.op_size(op))
    return op, torch.tensor(W.rhs(op, xs), device="cuda"), torch.tensor(xs, device="cuda")


# (20, 1): one block; 64 x 64: blocks of one row a thread; the others: two and four
@pytest.mark.parametrize("size", [(20, 1), (64, 64), (300, 300), (60, 60, 60)], ids=str)
@pytest.mark.parametrize("l", [1, 2, 3])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_resident_waits(P, size, l, prec):
    import torch
    op, b, xs = case(size)
    A = P.Matrix(op)
    kw = dict(l=l, interval=W.shift_interval(op), rtol=1e-8, prec=prec)
    for on in (1, 2, 3, 4, 5, 8, -1, -2, -3, -4, -7):
        x = torch.zeros_like(b)
        r = run_out(P, on, lambda: A.solve(b, x, check=False, **kw))
        assert r.status == P.PLCG_ERR_TIMEOUT, on
        x.zero_()
        r = A.solve(b, x, **kw)
        assert r.ok and float((x - xs).norm() / xs.norm()) <= 1e-6, on
    resident = P.last_launch()["kernel"]
    A.solve(b, torch.zeros_like(b), grid_ctas=1 << 20, **kw)
    assert P.last_launch()["kernel"] != resident
    A.close()


@pytest.mark.parametrize("l", [0, 1, 2, 3])   # 0: classic CG
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_grid_barrier(P, l, prec):
    import torch
    op, b, xs = case((64, 64))
    A = P.Matrix(op)
    kw = dict(interval=W.shift_interval(op), rtol=1e-8, prec=prec, grid_ctas=1 << 20,
              **(dict(l=l) if l else dict(method="cg")))
    x = torch.zeros_like(b)
    r = run_out(P, 1, lambda: A.solve(b, x, check=False, **kw))
    assert r.status == P.PLCG_ERR_TIMEOUT and P.last_launch()["cluster"] == 0
    x.zero_()
    r = A.solve(b, x, **kw)
    A.close()
    assert r.ok and float((x - xs).norm() / xs.norm()) <= 1e-6


def test_grid_barrier_without_allocation(P):
    import torch
    op, b, xs = case((64, 64))
    d = P.plcg_stencil_desc(dim=2, points=5, nx=64, ny=64, nz=1, center=op["center"], off=op["off"], diag_shift=0.0)
    p, keep = P.make_params(l=1, interval=W.shift_interval(op), rtol=1e-8, grid_ctas=1 << 20)
    x, r = torch.zeros_like(b), P.plcg_result()

    def solve():
        return P.load().plcg_solve_stencil_noalloc(C.byref(d), b.data_ptr(), x.data_ptr(), C.byref(p), C.byref(r),
                                                   C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert run_out(P, 1, solve) == P.PLCG_ERR_TIMEOUT and r.status == P.PLCG_ERR_TIMEOUT
    x.zero_()
    assert solve() == P.PLCG_OK and float((x - xs).norm() / xs.norm()) <= 1e-6
    del keep

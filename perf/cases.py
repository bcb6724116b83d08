"""What is measured: solves of A x = b through the public entry points of the package.

Every case is a whole solve as a program runs it: the operator handle (and, for request streams, the
server) is made once by ``prepare``; ``run`` sets x0 = 0, solves to the case's relative tolerance and
returns the solution. The right-hand sides are b = A x* with a seeded x* (b itself is random in the
batch of shifted Poisson systems), so ``exact`` is x*, or the direct solution in the sine basis.

Kinds of cases:

* ``stencil``: constant-coefficient 5-/7-point operators (``Matrix.solve``), FP64 vectors or FP32
  vectors with FP64 dots and refinement, p(l)-CG or classic CG.
* ``host``: the same, called on host arrays (``Matrix.solve_host``), copies included.
* ``hetero27``: the heterogeneous 27-point diffusion operator with the Jacobi preconditioner, as a
  CSR matrix or in the structured layout.
* ``spd``: CSR matrices of random sparsity, strictly diagonally dominant.
* ``batch``: many shifted 2D Poisson systems in one ``solve_batched`` call.
* ``serve``: a burst of requests of mixed sizes and operators through ``Server``.
"""
import math

import numpy as np
import torch

from paper_1905_06850_gb300 import plcg
from paper_1905_06850_gb300 import workloads as W


def listed():
    return [
        # the smallest requests of a request stream (10^3 unknowns): launch and iteration latency
        {"name": "poisson2d_32_fp64_l1", "kind": "stencil", "dim": 2, "nx": 32, "ny": 32, "nz": 1,
         "shift": 0.0, "prec": "fp64", "l": 1, "rtol": 1e-8},
        # the 100 x 100 Laplacian of the 2D configuration, p(2)-CG, its tolerance
        {"name": "poisson2d_100_fp64_l2", "kind": "stencil", "dim": 2, "nx": 100, "ny": 100, "nz": 1,
         "shift": 0.0, "prec": "fp64", "l": 2, "rtol": 1e-6},
        # a mid-sized ragged grid (odd x extent), three bases
        {"name": "poisson3d_75x61x57_fp64_l3", "kind": "stencil", "dim": 3, "nx": 75, "ny": 61, "nz": 57,
         "shift": 0.0, "prec": "fp64", "l": 3, "rtol": 1e-8},
        # the headline system: the 256^3 Laplacian in FP64, p(1)-CG
        {"name": "poisson3d_256_fp64_l1", "kind": "stencil", "dim": 3, "nx": 256, "ny": 256, "nz": 256,
         "shift": 0.0, "prec": "fp64", "l": 1, "rtol": 1e-8},
        # the same system on the mixed-precision path
        {"name": "poisson3d_256_fp32_l1", "kind": "stencil", "dim": 3, "nx": 256, "ny": 256, "nz": 256,
         "shift": 0.0, "prec": "fp32", "l": 1, "rtol": 1e-8},
        # classic CG, the method a user compares with, at 160^3
        {"name": "poisson3d_160_fp64_cg", "kind": "stencil", "dim": 3, "nx": 160, "ny": 160, "nz": 160,
         "shift": 0.0, "prec": "fp64", "l": 0, "rtol": 1e-8},
        # one implicit time step on host arrays: a shifted 3D operator, copies in and out included
        {"name": "host3d_128_fp64_l2", "kind": "host", "dim": 3, "nx": 128, "ny": 128, "nz": 128,
         "shift": 0.05, "prec": "fp64", "l": 2, "rtol": 1e-8},
        # the heterogeneous 27-point configuration as a general CSR matrix, Jacobi
        {"name": "hetero27_csr_128_fp32_l1", "kind": "hetero27", "layout": "csr", "nx": 128, "ny": 128,
         "nz": 128, "prec": "fp32", "l": 1, "rtol": 1e-8},
        # the same operator in the structured layout
        {"name": "hetero27_var_128_fp32_l1", "kind": "hetero27", "layout": "var27", "nx": 128, "ny": 128,
         "nz": 128, "prec": "fp32", "l": 1, "rtol": 1e-8},
        # an unstructured sparse matrix in FP64
        {"name": "spd_csr_300001_fp64_l1", "kind": "spd", "n": 300001, "prec": "fp64", "l": 1,
         "rtol": 1e-8},
        # the batched configuration: 4096 shifted 2D systems, sides 16 .. 256
        {"name": "batch_4096_fp32_l1", "kind": "batch", "count": 4096, "s_lo": 16, "s_hi": 256,
         "prec": "fp32", "l": 1, "rtol": 1e-8},
        # a burst of serving requests, n from 10^3 to 3*10^5
        {"name": "serve_24_fp32_l1", "kind": "serve", "count": 24, "n_lo": 1000, "n_hi": 300000,
         "prec": "fp32", "l": 1, "rtol": 1e-8},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["stencil", "stencil", "stencil", "host", "hetero27", "hetero27", "spd", "batch", "serve"])
    prec = rng.choice(["fp64", "fp32"])
    if kind in ("stencil", "host"):
        dim = rng.choice([2, 3])
        c = {"kind": kind, "dim": dim, "prec": prec, "rtol": rng.choice([1e-6, 1e-8])}
        if dim == 2:
            s = _log_int(rng, 32, 1024 if kind == "stencil" else 512)
            c["nx"], c["ny"], c["nz"] = s, max(8, int(s * rng.uniform(0.7, 1.4))), 1
        else:
            s = _log_int(rng, 10, 240 if kind == "stencil" else 128)
            c["nx"], c["ny"] = s, max(4, int(s * rng.uniform(0.8, 1.2)))
            c["nz"] = max(4, int(s * rng.uniform(0.8, 1.1)))
        # implicit time steps (a shift) or the pure Laplacian; the large 2D ones are time steps
        c["shift"] = 0.0 if (dim == 3 or s < 256) and rng.random() < 0.6 else round(rng.uniform(0.01, 1.0), 4)
        c["l"] = rng.choice([1, 1, 2, 3, 0])
        return c
    if kind == "hetero27":
        s = _log_int(rng, 24, 120)
        return {"kind": kind, "layout": rng.choice(["csr", "var27"]), "nx": s, "ny": max(8, int(s * rng.uniform(0.8, 1.2))),
                "nz": max(8, int(s * rng.uniform(0.8, 1.2))), "prec": "fp32", "l": rng.choice([1, 1, 2, 0]), "rtol": 1e-8}
    if kind == "spd":
        return {"kind": kind, "n": _log_int(rng, 1000, 1000000), "prec": prec, "l": rng.choice([1, 1, 0]), "rtol": 1e-8}
    if kind == "batch":
        lo = rng.randint(8, 64)
        return {"kind": kind, "count": _log_int(rng, 64, 4096), "s_lo": lo, "s_hi": rng.randint(lo + 1, 256),
                "prec": rng.choice(["fp32", "fp32", "fp64"]), "l": rng.choice([1, 1, 2, 3, 0]), "rtol": 1e-8}
    return {"kind": kind, "count": rng.randint(4, 32), "n_lo": 1000, "n_hi": _log_int(rng, 10000, 300000), "prec": prec,
            "l": rng.choice([1, 1, 0]), "rtol": 1e-8}


# ------------------------------------------------------------------ inputs


def _gen(*seeds):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(np.random.SeedSequence([int(s) for s in seeds]).generate_state(1, np.uint64)[0] >> np.uint64(1)))
    return g


def _normal(n, *seeds):
    return torch.randn(n, dtype=torch.float64, device="cuda", generator=_gen(*seeds))


def _stencil_op(c):
    make = W.stencil2d(c["nx"], c["ny"], shift=c["shift"]) if c["dim"] == 2 else \
        W.stencil3d(c["nx"], c["ny"], c["nz"], shift=c["shift"])
    return W.fp32_rounded(make)   # the coefficients of either precision are the same


def _stencil_rhs(op, x):
    """b = A x by shifted slices."""
    dims = (op["nz"], op["ny"], op["nx"]) if op["dim"] == 3 else (op["ny"], op["nx"])
    X = x.view(dims)
    nb = torch.zeros_like(X)
    for ax, d in enumerate(dims):
        nb.narrow(ax, 0, d - 1).add_(X.narrow(ax, 1, d - 1))
        nb.narrow(ax, 1, d - 1).add_(X.narrow(ax, 0, d - 1))
    return (op["center"] * X + op["off"] * nb).reshape(-1)


def _csr_rhs(op, x):
    """b = A x of a CSR operator without empty rows."""
    return torch.from_numpy(np.add.reduceat(op["val"] * x.cpu().numpy()[op["col"]], op["rowptr"][:-1])).cuda()


def _hetero27(c, seed):
    """The heterogeneous 27-point operator (harmonic means of exp(N(0,1)) cell coefficients, weights
    1, 1/2, 1/3), FP32-rounded where the path stores FP32: the operator and A x as a function."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    n = nx * ny * nz
    k3 = torch.exp(_normal(n, seed, 1)).view(nz, ny, nx)
    iz, iy, ix = (torch.arange(d, device="cuda").view([-1 if a == b else 1 for b in range(3)]) for a, d in enumerate((nz, ny, nx)))
    offsets = [(dz, dy, dx) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]
    vals = torch.zeros(27, nz, ny, nx, dtype=torch.float64, device="cuda")
    mask = torch.ones(27, nz, ny, nx, dtype=torch.bool, device="cuda")
    diag = torch.zeros_like(k3)
    for j, (dz, dy, dx) in enumerate(offsets):
        if j == 13:
            continue
        ok = (iz + dz >= 0) & (iz + dz < nz) & (iy + dy >= 0) & (iy + dy < ny) & (ix + dx >= 0) & (ix + dx < nx)
        kd = torch.where(ok, torch.roll(k3, (-dz, -dy, -dx), (0, 1, 2)), k3)
        w = 2.0 / (abs(dz) + abs(dy) + abs(dx)) * (k3 * kd) / (k3 + kd)
        diag += w
        vals[j], mask[j] = -w, ok
    vals[13] = diag
    if c["prec"] != "fp64":
        vals = vals.float().double()

    def apply(x):
        X = torch.nn.functional.pad(x.view(nz, ny, nx), (1, 1, 1, 1, 1, 1))
        b = torch.zeros_like(k3)
        for j, (dz, dy, dx) in enumerate(offsets):
            b += torch.where(mask[j], vals[j], 0.0) * X[1 + dz:1 + dz + nz, 1 + dy:1 + dy + ny, 1 + dx:1 + dx + nx]
        return b.reshape(-1)

    if c["layout"] == "var27":
        coef = torch.empty(14, n, dtype=torch.float64, device="cuda")
        coef[0] = vals[13].reshape(-1)
        for k, o in enumerate(W.VAR27_FORWARD):
            j = offsets.index(o)
            coef[1 + k] = torch.where(mask[j], vals[j], 0.0).reshape(-1)
        op = {"kind": "var27", "nx": nx, "ny": ny, "nz": nz, "coef": coef.cpu().numpy()}
    else:
        m = mask.view(27, n).t()
        lin = torch.arange(n, device="cuda")
        step = torch.tensor([(dz * ny + dy) * nx + dx for dz, dy, dx in offsets], device="cuda")
        rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        rowptr[1:] = torch.cumsum(m.sum(1), 0)
        op = {"kind": "csr", "n": n, "rowptr": rowptr.cpu().numpy(),
              "col": (lin[:, None] + step)[m].int().cpu().numpy(), "val": vals.view(27, n).t()[m].cpu().numpy()}
    return op, apply


def _random_spd(n, seed, prec):
    """A CSR matrix of random sparsity, 5 .. 30 entries a row on average, strictly diagonally dominant."""
    r = np.random.default_rng([seed, 2])
    per = (r.integers(5, 31, size=n) - 1) // 2
    i = torch.from_numpy(np.repeat(np.arange(n, dtype=np.int64), per)).cuda()
    j = torch.from_numpy(r.integers(0, n, size=i.numel())).cuda()
    key = torch.unique(torch.minimum(i, j) * n + torch.maximum(i, j))
    i, j = key // n, key % n
    i, j = i[i != j], j[i != j]
    v = -torch.rand(i.numel(), dtype=torch.float64, device="cuda", generator=_gen(seed, 3))
    row, col = torch.cat([i, j]), torch.cat([j, i])
    order = torch.argsort(row * n + col)
    row, col, v = row[order], col[order], torch.cat([v, v])[order]
    # the diagonal: the row's absolute sum times 1.05 .. 1.5 (summed on the host, in order)
    count = torch.bincount(row, minlength=n).cpu().numpy()
    start = np.cumsum(count) - count
    total = np.zeros(n)
    total[count > 0] = np.add.reduceat(np.abs(v.cpu().numpy()), start[count > 0])
    d = np.where(count > 0, total * (1.0 + r.uniform(0.05, 0.5, size=n)), 1.0)
    lin = torch.arange(n, device="cuda")
    row, col, v = torch.cat([row, lin]), torch.cat([col, lin]), torch.cat([v, torch.from_numpy(d).cuda()])
    order = torch.argsort(row * n + col)
    rowptr = np.concatenate([[0], np.cumsum(count + 1)])
    v = v[order]
    if prec != "fp64":
        v = v.float().double()
    return {"kind": "csr", "n": n, "rowptr": rowptr, "col": col[order].int().cpu().numpy(), "val": v.cpu().numpy()}


def _batch_sizes(c, seed):
    """The sides are the case's, the diagonal shifts the seed's."""
    sides = np.random.default_rng([c["count"], c["s_lo"], c["s_hi"]]).integers(c["s_lo"], c["s_hi"] + 1, size=c["count"])
    shifts = np.random.default_rng([seed, 5]).uniform(0.0, 1.0, size=c["count"]).astype(np.float32).astype(np.float64)
    pad = (sides.astype(np.int64) ** 2 + 1) // 2 * 2   # every system starts on a 16-byte boundary
    return sides, shifts, np.concatenate([[0], np.cumsum(pad)])


def _serve_requests(c, seed):
    """Sizes log-uniform (the case's), operators in turn 2D, 3D and random CSR (as a mixed stream has
    them), diagonal shifts by the seed."""
    r, q = np.random.default_rng([c["count"], c["n_lo"], c["n_hi"]]), np.random.default_rng([seed, 6])
    got = []
    for k in range(c["count"]):
        n = math.exp(r.uniform(math.log(c["n_lo"]), math.log(c["n_hi"])))
        got.append((("2d", "3d", "csr")[k % 3], n, round(float(q.uniform(0.01, 1.0)), 4)))
    return got


def _solver(c, lo, hi):
    kw = {"rtol": c["rtol"], "prec": c["prec"], "maxit": 100000}
    return dict(kw, method="cg") if c["l"] == 0 else dict(kw, l=c["l"], interval=(lo, hi))


def prepare(case, seed):
    c = case
    if c["kind"] in ("stencil", "host"):
        op = _stencil_op(c)
        b = _stencil_rhs(op, _normal(W.op_size(op), seed, 0))
        s = {"A": plcg.Matrix(op, prec=c["prec"]), "b": b, "kw": _solver(c, *W.shift_interval(op)), "kind": c["kind"]}
        if c["kind"] == "host":
            s["b"] = b.cpu().numpy()
            s["x"] = np.empty_like(s["b"])
        else:
            s["x"] = torch.empty_like(b)
        return s
    if c["kind"] == "hetero27":
        op, apply = _hetero27(c, seed)
        b = apply(_normal(W.op_size(op), seed, 0))
        # M^{-1} A of this operator: a Gershgorin bound of 2, Ritz values below 1.6
        return {"A": plcg.Matrix(op, prec=c["prec"]), "b": b, "x": torch.empty_like(b), "kind": "stencil",
                "kw": dict(_solver(c, 0.0, 1.62), precond="jacobi")}
    if c["kind"] == "spd":
        op = _random_spd(c["n"], seed, c["prec"])
        b = _csr_rhs(op, _normal(c["n"], seed, 0))
        return {"A": plcg.Matrix(op, prec=c["prec"]), "b": b, "x": torch.empty_like(b), "kind": "stencil",
                "kw": _solver(c, *W.shift_interval(op))}
    if c["kind"] == "batch":
        sides, shifts, at = _batch_sizes(c, seed)
        b = _normal(int(at[-1]), seed, 0)
        x = torch.zeros_like(b)
        ops = [W.fp32_rounded(W.stencil2d(int(m), int(m), shift=float(h))) for m, h in zip(sides, shifts)]
        cut = [(int(at[k]), int(at[k]) + int(sides[k]) ** 2) for k in range(c["count"])]
        return {"kind": "batch", "A": [plcg.Matrix(op, prec=c["prec"]) for op in ops], "x": x, "b": b,
                "bs": [b[p:q] for p, q in cut], "xs": [x[p:q] for p, q in cut],
                "lo": [op["center"] - 4.0 for op in ops], "hi": [op["center"] + 4.0 for op in ops],
                "kw": {k: v for k, v in _solver(c, 0.0, 8.0).items() if k != "interval"}}
    reqs, flat = [], []
    for k, (what, n, shift) in enumerate(_serve_requests(c, seed)):
        if what == "csr":
            op = _random_spd(int(round(n)), seed * 1000 + k, c["prec"])
            b = _csr_rhs(op, _normal(op["n"], seed, 0, k))
        else:
            m = int(round(n ** (0.5 if what == "2d" else 1.0 / 3.0)))
            op = _stencil_op({"dim": 2 if what == "2d" else 3, "nx": m, "ny": m, "nz": m, "shift": shift})
            b = _stencil_rhs(op, _normal(W.op_size(op), seed, 0, k))
        reqs.append((plcg.Matrix(op, prec=c["prec"]), b, _solver(c, *W.shift_interval(op))))
        flat.append((b.numel() + 1) // 2 * 2)
    at = np.concatenate([[0], np.cumsum(flat)])
    x = torch.zeros(int(at[-1]), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()   # the server's streams are its own
    return {"kind": "serve", "server": plcg.Server(mem_budget_bytes=8 << 30), "x": x,
            "reqs": [(A, b, x[int(p):int(p) + b.numel()], kw) for (A, b, kw), p in zip(reqs, at)]}


def run(state):
    s = state
    if s["kind"] == "host":
        s["x"].fill(0.0)
        s["A"].solve_host(s["b"], s["x"], **s["kw"])
        return s["x"]
    s["x"].zero_()
    if s["kind"] == "stencil":
        s["A"].solve(s["b"], s["x"], **s["kw"])
    elif s["kind"] == "batch":
        plcg.solve_batched(s["A"], s["bs"], s["xs"], s["lo"], s["hi"], **s["kw"])
    else:
        torch.cuda.current_stream().synchronize()   # x0 is set before the server's streams read it
        tickets = [s["server"].submit(A, b, x, **kw) for A, b, x, kw in s["reqs"]]
        for t in tickets:
            s["server"].wait(t)
    return s["x"]


# ------------------------------------------------------------------ expectations


def exact(case, seed):
    c = case
    if c["kind"] == "serve":
        parts = []
        for k, (what, n, _) in enumerate(_serve_requests(c, seed)):
            m = int(round(n ** (0.5 if what == "2d" else 1.0 / 3.0))) if what != "csr" else 0
            size = int(round(n)) if what == "csr" else m ** (2 if what == "2d" else 3)
            parts += [_normal(size, seed, 0, k)] + ([torch.zeros(1, dtype=torch.float64, device="cuda")] if size % 2 else [])
        return torch.cat(parts)
    if c["kind"] == "batch":
        # A = S (x) S diag(lambda_i + lambda_j + shift) S (x) S with the sine matrices S of the sides
        sides, shifts, at = _batch_sizes(c, seed)
        b = _normal(int(at[-1]), seed, 0)
        x = torch.zeros_like(b)
        sine = {}
        for k in range(c["count"]):
            m = int(sides[k])
            if m not in sine:
                j = torch.arange(1, m + 1, dtype=torch.float64, device="cuda") * (math.pi / (m + 1))
                sine[m] = (math.sqrt(2.0 / (m + 1)) * torch.sin(j[:, None] * torch.arange(1, m + 1, dtype=torch.float64, device="cuda")),
                           2.0 - 2.0 * torch.cos(j))
            S, lam = sine[m]
            center = float(np.float32(4.0 + float(shifts[k])))
            B = S @ b[int(at[k]):int(at[k]) + m * m].view(m, m) @ S
            x[int(at[k]):int(at[k]) + m * m] = (S @ (B / (lam[:, None] + lam[None, :] + (center - 4.0))) @ S).reshape(-1)
        return x
    n = c["n"] if c["kind"] == "spd" else c["nx"] * c["ny"] * c["nz"]
    x = _normal(n, seed, 0)
    return x.cpu().numpy() if c["kind"] == "host" else x


def _passes(c, n, iters, entry_bytes):
    """(bytes, flops) of one solve. An iteration of p(l)-CG reads the current and the previous vector
    of its l + 1 bases and writes the next (the direction and the iterate need not pass through memory
    every time); one of classic CG reads r, p and q and writes them, r and q once more for the second
    inner product, and the iterate's update reads p; the matrix is read once."""
    word = 8 if c["prec"] == "fp64" else 4
    vectors = 8 if c["l"] == 0 else 3 * (c["l"] + 1) + 1
    flops = 20 if c["l"] == 0 else 6 * c["l"] + 18
    return iters * n * (vectors * word + entry_bytes), iters * n * flops


def _iterations(c, dim, sides, shift):
    """About how many iterations a stencil solve takes (fitted to right-hand sides A x*, x* white)."""
    kappa = (4.0 * dim + shift) / (shift + sum(2.0 - 2.0 * math.cos(math.pi / (m + 1)) for m in sides))
    return max(5.0, 0.45 * kappa ** 0.4 * math.log(2.0 / c["rtol"]))


def work(case):
    c = case
    word = 8 if c["prec"] == "fp64" else 4
    total = [0.0, 0.0]

    def add(n, iters, entry_bytes):
        b, f = _passes(c, n, iters, entry_bytes)
        total[0] += b
        total[1] += f

    if c["kind"] in ("stencil", "host"):
        sides = [c["nx"], c["ny"]] + ([c["nz"]] if c["dim"] == 3 else [])
        add(math.prod(sides), _iterations(c, c["dim"], sides, c["shift"]), 0)
    elif c["kind"] == "hetero27":
        n = c["nx"] * c["ny"] * c["nz"]
        iters = 1.75 * (n ** (1.0 / 3.0))
        add(n, iters, 14 * word if c["layout"] == "var27" else 26.6 * (4 + word) + 8 + 2 * word)
    elif c["kind"] == "spd":
        add(c["n"], 45, 17 * (4 + word) + 8)
    elif c["kind"] == "batch":
        for m in range(c["s_lo"], c["s_hi"] + 1):
            add(m * m * c["count"] / (c["s_hi"] - c["s_lo"] + 1), 51, 0)
    else:
        mean = (c["n_hi"] - c["n_lo"]) / math.log(c["n_hi"] / c["n_lo"])
        add(mean * c["count"], 45, 6 * (4 + word))
    return {"bytes": total[0], "flops": total[1]}

"""1/sqrt(x) and 1/x from an FP32 seed (csrc/fastroot.h), compiled for the host
with g++ and checked against 60-digit decimals (no GPU).  The bound: half an
ulp of the last operation (2^-53 relative) and, before it, a correction of at
most 2^-18 with a handful of roundings and terms below 2^-72 left out -- within
2^-53 (1 + 2^-12) for every seed whose relative error is below 2^-20.  Arguments
outside the stated range take the plain operation."""
import math
import os
import shutil
import struct
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
getcontext().prec = 60
BOUND = Decimal(2) ** -53 * (1 + Decimal(2) ** -12)


@pytest.fixture(scope="module")
def roots(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("roots")
    src = d / "roots.cpp"
    src.write_text(r'''
#include <cstdio>
#include <cstring>
#include "fastroot.h"
using namespace plcg;
static double rd() { unsigned long long u; if (scanf("%llx", &u) != 1) return 0; double x; memcpy(&x, &u, 8); return x; }
int main() {
    char op;
    while (scanf(" %c", &op) == 1) {
        const double x = rd(), y = rd();
        const double r = op == 'r' ? fast_rsqrt(x) : op == 'd' ? fast_rcp(x) : op == 'R' ? rsqrt_from_seed(x, y) : rcp_from_seed(x, y);
        unsigned long long u; memcpy(&u, &r, 8); printf("%016llx\n", u);
    }
    return 0;
}
''')
    exe = d / "roots"
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_1905_06850_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)

    def run(cases):
        h = lambda v: struct.pack(">d", float(v)).hex()   # noqa: E731
        inp = "".join(f"{op} {h(x)} {h(y)}\n" for op, x, y in cases)
        out = subprocess.run([str(exe)], input=inp, capture_output=True, text=True, check=True).stdout
        return [struct.unpack(">d", bytes.fromhex(t))[0] for t in out.split()]
    return run


def values():
    rng = np.random.default_rng(11)
    v = list(np.exp2(rng.uniform(-1021, 1022, 1500)) * rng.uniform(1, 2, 1500))
    v += list(rng.uniform(1, 4, 1500)) + [1.0, 2.0, 4.0, 3.0, np.nextafter(1, 2), np.nextafter(2, 1), np.nextafter(4, 1)]
    return [float(x) for x in v if math.isfinite(x)]


def test_reciprocal_square_root(roots):
    xs = values() + [2.0 ** -1022, 1.7e308]
    for x, r in zip(xs, roots([("r", x, 0) for x in xs])):
        assert abs(Decimal(r) * Decimal(x).sqrt() - 1) <= BOUND, x


def test_reciprocal(roots):
    xs = [x for x in values() if 2.0 ** -1021 <= x < 2.0 ** 1021]
    xs += [-x for x in xs[:500]]
    for x, r in zip(xs, roots([("d", x, 0) for x in xs])):
        assert abs(Decimal(r) * Decimal(x) - 1) <= BOUND, x


@pytest.mark.parametrize("op,power", [("R", Decimal("0.5")), ("D", Decimal(1))])
def test_every_seed_within_2_to_the_minus_20(roots, op, power):
    rng = np.random.default_rng(12)
    m = rng.uniform(1, 4 if op == "R" else 2, 2000)
    exact = m ** (-0.5 if op == "R" else -1.0)
    y = (exact * (1 + rng.choice([-1, 1], 2000) * 2.0 ** -20.1)).astype(np.float32).astype(np.float64)
    for x, r in zip(m, roots([(op, a, b) for a, b in zip(m, y)])):
        ref = Decimal(float(x)).sqrt() if op == "R" else Decimal(float(x))
        assert abs(Decimal(r) * ref - 1) <= BOUND, x


def test_other_arguments_take_the_plain_operation(roots):
    r = roots([("r", v, 0) for v in (-1.0, float("nan"), float("inf"), 0.0)])
    assert math.isnan(r[0]) and math.isnan(r[1]) and r[2] == 0.0 and r[3] == math.inf
    xs = [0.0, -0.0, math.inf, -math.inf, 2.0 ** -1040, 1.5 * 2.0 ** 1023]
    got = roots([("d", v, 0) for v in xs])
    assert got[0] == math.inf and got[1] == -math.inf and got[2] == 0 and got[3] == 0 and math.isinf(got[4])
    assert got[5] == 1.0 / xs[5]
    assert math.isnan(roots([("d", float("nan"), 0)])[0])

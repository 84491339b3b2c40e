"""Indices of the 2D solver's stacked vectors at the limits of what creation accepts (compiled from
csrc/rows2d.h for the host, no GPU): every pair row fits 32 bits, the rho row is formed in 64."""
import ctypes
import os
import random
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1811_05579_gb300", "csrc")


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    d = tmp_path_factory.mktemp("rows2d")
    src, so = str(d / "rows.cpp"), str(d / "rows.so")
    with open(src, "w") as f:
        f.write('#include "rows2d.h"\nextern "C" {\n'
                "int fit(int64_t p, int64_t x, int64_t y) { return grte2::rows_fit(p, x, y); }\n"
                # as the operator pass forms it: K, nc and the cell are int
                "int64_t last(int K, int nc) { const int c = nc - 1; return grte2::rho_row(K, nc) + c; }\n}\n")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", so, src], check=True)
    lib = ctypes.CDLL(so)
    lib.fit.argtypes = [ctypes.c_int64] * 3
    lib.last.argtypes, lib.last.restype = [ctypes.c_int] * 2, ctypes.c_int64
    return lib


def test_rho_row_past_32_bits(rows):
    assert rows.fit(20, 10113, 10113) and 21 * 10113 ** 2 > 1 << 31
    assert rows.last(20, 10113 ** 2) == 21 * 10113 ** 2 - 1


def test_accepted_sizes(rows):
    rng = random.Random(7)
    accepted = 0
    for _ in range(20000):
        K, nx = rng.randint(1, 64), int(2 ** rng.uniform(1, 15))
        ny = min(max(2, (1 << 31) // (max(K, 20) * (nx + 1)) + rng.randint(-3, 3)), 32768)
        n = max(K, 20) * (nx + 1) * (ny + 1)
        assert bool(rows.fit(K, nx, ny)) == (n < 1 << 31)
        if n < 1 << 31:
            accepted += 1
            assert K * nx * ny < 1 << 31
            assert rows.last(K, nx * ny) == (K + 1) * nx * ny - 1
    assert accepted > 1000


def test_operator_takes_the_row_from_there():
    """No index of the Krylov kernels reaches the rho row by a 32-bit K nc."""
    src = open(os.path.join(CSRC, "krylov2d.cuh")).read()
    code = re.sub(r"//[^\n]*", "", src)
    assert not re.search(r"\bK\s*\*\s*nc\b", code)
    assert re.search(r"int64_t\s+rrow\s*=\s*rho_row\(K, nc\)", code)
    for name in ("z", "b", "out"):   # z[rrow + ...], b[orho], out[orho]
        assert re.search(r"\b%s\[(rrow|orho)" % name, code)
    assert re.search(r"const int64_t orho = rrow \+ c;", code)

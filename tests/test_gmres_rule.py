"""The cluster size of the 1D Krylov kernels: the residency of sixteen CTAs is asked for with the
shared memory that the launches then take (csrc/gmres_rule.h on the host, the device's answer
replaced), and on the GPU the largest slices in shared memory and the first in global memory give
what clusters of eight give."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1811_05579_gb300", "csrc")
LIMIT = 200000      # a device's limit of dynamic shared memory per CTA


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("gmres_rule")
    src, so = str(d / "rule.cpp"), str(d / "rule.so")
    with open(src, "w") as f:
        f.write('#include "gmres_rule.h"\nextern "C" {\n'
                # room: what the device can hold per CTA of such a cluster; asked: what it was asked
                "int cluster(const int64_t* nx, int n, int mixed, int64_t limit, int64_t room, int64_t* asked) {\n"
                "  return grte::gmres_cluster(nx, n, mixed != 0, limit, [&](int64_t b) { *asked = b; return b <= room; });\n}\n"
                "int64_t launch_bytes(const int64_t* nx, int n, int ncl, int64_t limit) {\n"
                "  return grte::gmres_dyn_bytes(grte::largest_slice(nx, n, ncl), limit);\n}\n}\n")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", so, src], check=True)
    lib = ctypes.CDLL(so)
    p64 = ctypes.POINTER(ctypes.c_int64)
    lib.cluster.argtypes = [p64, ctypes.c_int, ctypes.c_int, ctypes.c_int64, ctypes.c_int64, p64]
    lib.launch_bytes.argtypes, lib.launch_bytes.restype = [p64, ctypes.c_int, ctypes.c_int, ctypes.c_int64], ctypes.c_int64

    def call(sizes, mixed=False, room=1 << 40):
        nx, asked = (ctypes.c_int64 * len(sizes))(*sizes), ctypes.c_int64(-1)
        ncl = lib.cluster(nx, len(sizes), int(mixed), LIMIT, room, ctypes.byref(asked))
        return ncl, asked.value, lib.launch_bytes(nx, len(sizes), 16, LIMIT)
    return call


@pytest.mark.parametrize("sizes", [[2048], [8192], [2049, 256, 2], [300000], [388000], [500000], [4096] * 7])
def test_residency_is_asked_for_the_launch(rule, sizes):
    ncl, asked, launch = rule(sizes)
    assert ncl == 16 and asked == launch
    if launch > 0:      # a device that holds such clusters, but not with this much shared memory
        assert rule(sizes, room=launch - 1)[0] == 8
        assert rule(sizes, room=launch)[0] == 16
    big = max(n // 16 + 1 if n > 256 else n + 1 for n in sizes)
    need = (big + big // 32 + 1) * 8
    assert launch == (0 if need > LIMIT else (need + 15) // 16 * 16)


def test_small_many_and_mixed_take_eight(rule):
    for sizes, mixed in (([2047], False), ([4096] * 8, False), ([8192], True)):
        assert rule(sizes, mixed)[:2] == (8, -1)


# Both solve to 1e-13 of every cell or the residual's rounding floor; T sees at most 1e2 times
# that.  A slice cut or factored wrongly is off by parts of the solution.
@pytest.mark.gpu
@pytest.mark.parametrize("N", [300000, 450000])   # 16 slices: 155 KB of shared memory; global memory
def test_largest_slices(N):
    from paper_1811_05579_gb300 import grte as G
    rng = np.random.default_rng(N)
    spec = dict(nx=N, n_angle=2, v=np.array([0.2113, 0.7887]), w=np.array([0.5, 0.5]), sigma=0.5 + 2.0 * rng.random(N),
                kind=G.SIGMA_T3, bc=G.BC_INFLOW, bL=np.ones(2), bR=np.full(2, 0.1), dt=0.1 / N, eps=1e-2)
    T0 = 0.6 + 0.4 * np.sin(np.arange(N) * (20.0 / N))
    out = []
    for n in (1, 8):
        h = G.Grte([spec] * n)
        for i in range(n):
            h.set_state(i, T0)
        h.step(1)
        out.append(h.T(n - 1))
        h.close()
    assert np.max(np.abs(out[0] - out[1]) / out[1]) < 1e-9

"""The one-kernel diffusion steps (up to 8192 cells, clusters of 512-cell CTAs, four cells per
thread) and the three-launch path above, at the edges of threads, CTAs and clusters, in one
handle with both opacity forms; more steps than one launch holds; U* outside the binary32
range, where U*^{3/4} is the library's.  Bound: 1e-12 relative per step, the bound of the
solver's other tests."""
import numpy as np
import pytest

from oracle import diffusion1d as dif
from paper_1811_05579_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1811_05579_gb300 import grte
    return grte


def _check(G, sizes, steps, scale=1.0):
    rng = wl.SplitMix64(4711)
    insts = []
    for i, N in enumerate(sizes):
        kind = "t3" if i % 2 else "const"
        x = (np.arange(N) + 0.5) / N
        T0 = scale * (0.05 + np.maximum(np.sin(2 * np.pi * (x - 0.1)), 0.0) + 0.2 * rng.uniform(N))
        insts.append(dict(nx=N, sigma=0.2 + 2.0 * rng.uniform(N), dt=0.05 / N, T0=T0, okind=kind,
                          kind=G.SIGMA_T3 if i % 2 else G.SIGMA_CONST))
    h = G.Diffusion(insts)
    for rep in range(2):                       # the second set replaces the first before any step
        for i, p in enumerate(insts):
            h.set_T(i, p["T0"] * (2.0 - rep))
    h.step(steps)
    for i, p in enumerate(insts):
        T = p["T0"].copy()
        for _ in range(steps):
            T, Us = dif.three_stage_step(T, p["sigma"], 1.0 / p["nx"], p["dt"], kind=p["okind"])
        eT = np.max(np.abs(h.T(i) - T)) / np.max(np.abs(T))
        eU = np.max(np.abs(h.Ustar(i) - Us)) / np.max(np.abs(Us))
        assert eT < 1e-12 * steps and eU < 1e-12 * steps, (p["nx"], p["okind"], eT, eU)
    h.close()


@pytest.mark.parametrize("shift", [0, 1])     # swaps the opacity forms
def test_sizes_around_thread_cta_and_cluster_edges(G, shift):
    _check(G, [2] * shift + [2, 3, 4, 5, 127, 129, 511, 512, 513, 1024, 1025, 1541, 7680, 7681, 8191, 8192, 8193], 3)


def test_more_steps_than_one_launch(G):
    _check(G, [64, 65, 513, 514], 66)


def test_outside_the_binary32_range(G):
    _check(G, [100, 700, 701], 2, scale=1e-9)

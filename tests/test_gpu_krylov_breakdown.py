"""The FP64 Krylov kernels where the new vector lies in the basis: N cells have an N-dimensional Krylov
space, and a cycle started far below the solution (E = 1e-20 of it) goes on past it, on vectors made
of rounding.  The restart's true residual decides: one cycle, the oracle's T to 1e-11 (the prediction
is solved to 1e-13 of every cell, T sees at most 1e2 times that)."""
import numpy as np
import pytest

from oracle import grte1d as og
from oracle.quadrature import gauss_legendre_half

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1811_05579_gb300 import grte
    return grte


@pytest.mark.parametrize("kind", ["const", "t3"])
@pytest.mark.parametrize("N", [2, 3, 4])
def test_past_the_whole_space(G, N, kind):
    v, w = gauss_legendre_half(8)
    M = v.size
    rng = np.random.default_rng(N)
    beyond = 0
    for _ in range(40):
        P = og.Problem(N=N, v=v, w=w, sig=0.5 + rng.random(N), eps=1e-2, dt=1.0, kind=kind, bc="reflect",
                       bL=np.zeros(M), bR=np.zeros(M))
        T0 = 0.5 + rng.random(N)
        S = og.State(E=np.full((N, M), 1e-20), O=np.zeros((N + 1, M)), U=T0 ** 4, T=T0)
        h = G.Grte([dict(nx=N, n_angle=M, v=v, w=w, sigma=P.sig, kind=1 if kind == "t3" else 0, bc=1, bL=P.bL,
                         bR=P.bR, dt=P.dt, eps=P.eps)])
        h.set_state(0, S.T, S.E, S.O)
        h.step(1)
        T = og.step(P, S).T
        assert np.max(np.abs(h.T(0) - T) / T) < 1e-11
        st = h.stats()
        assert st["krylov_cycles"] == 1
        beyond += st["krylov_iters"] > N
        h.close()
    assert beyond > 0     # the case is met

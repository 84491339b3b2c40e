"""The operator pass's larger tilings (32 x 4 from 152 tiles, 32 x 8 from 608) against the oracle with inflow
on both axes: wall and corner vertices of every side, and partial tiles at the upper walls (97 = 3
32 + 1, 203 = 50 4 + 3; 33 = 32 + 1, 2425 = 303 8 + 1).  T and every intensity of one step; FP64 stops
at 1e-13 of the scaled residual, mixed precision at its binary32 tolerance: 1e-9 and 1e-5, the
bounds of the other comparison across tilings."""
import numpy as np
import pytest

from oracle import grte2d as o2

pytestmark = pytest.mark.gpu
CASES = {"32x4": (97, 203, 3), "32x8": (33, 2425, 2)}


@pytest.fixture(scope="module", params=sorted(CASES))
def problem(request):
    nx, ny, K = CASES[request.param]
    tiles = [-(-nx // 32) * -(-ny // t) for t in (8, 4)]
    assert tiles[0] >= 4 * 152 if request.param == "32x8" else tiles[0] < 4 * 152 and tiles[1] >= 152
    rng = np.random.default_rng(3)
    P = o2.Problem2D(Nx=nx, Ny=ny, mu=[0.35, 0.86, -0.6][:K], eta=[0.86, -0.35, 0.3][:K], w=np.full(K, 1.0 / K),
                     sig=0.5 + rng.random((ny, nx)), eps=1e-1, dt=0.2 / nx, kind="t3", bx0=1.0, bx1=0.3, by0=0.1,
                     by1=0.6, Ly=ny / nx)
    T0 = 0.5 + 0.5 * rng.random(ny * nx)
    return P, T0, o2.step(P, o2.equilibrium_state(P, T0))


@pytest.mark.parametrize("mixed", [False, True])
def test_larger_tilings_with_walls_on_both_axes(problem, mixed):
    from paper_1811_05579_gb300 import grte as G
    P, T0, S = problem
    h = G.Grte2D(P.Nx, P.Ny, P.sig, P.dt, P.eps, kind=G.SIGMA_T3, b_x0=P.bx0, b_x1=P.bx1, b_y0=P.by0, b_y1=P.by1,
                 mu=P.mu, eta=P.eta, w=P.w, ly=P.Ly, precision=G.MIXED if mixed else G.FP64)
    h.set_state(T0)
    h.step(1)
    tol = 1e-5 if mixed else 1e-9
    assert np.max(np.abs(h.T() - S.T) / S.T) < tol
    assert np.max(np.abs(h.E() - S.E)) < tol * np.max(np.abs(S.E))
    h.close()

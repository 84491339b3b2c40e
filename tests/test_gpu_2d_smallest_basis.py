"""The 2D state's arrays pass through the Krylov basis, which on the smallest grid with the shortest
restart holds fewer values ((m+1)(K+1) 4 = 168 for 20 pairs) than O (9 K = 180): E and O come
back as they were set, also beside a second handle, and after a sigma_0/T^3 step, which keeps the
prediction's vertex values there."""
import numpy as np
import pytest

from oracle.quadrature import s8_pairs_2d

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1811_05579_gb300 import grte
    return grte


@pytest.mark.parametrize("shape", [(2, 2), (2, 3), (3, 2)])
@pytest.mark.parametrize("K", [1, 8, 9, 20, 63])
def test_state_round_trip_shortest_restart(G, K, shape):
    nx, ny = shape
    rng = np.random.default_rng(K)
    mu, eta, _ = s8_pairs_2d()
    pairs = dict(mu=np.resize(mu, K), eta=np.resize(eta, K), w=np.ones(K))
    hs = [G.Grte2D(nx, ny, 1.0, 0.01, 1e-1, kind=G.SIGMA_T3, b_x0=1.0, krylov_restart=1, **pairs) for _ in range(2)]
    state = [(0.5 + rng.random(nx * ny), rng.random((nx * ny, K)), rng.random(((nx + 1) * (ny + 1), K))) for _ in hs]
    for h, (T, E, O) in zip(hs, state):
        h.set_state(T, E, O)
    for h, (T, E, O) in zip(hs, state):
        assert np.array_equal(h.T().ravel(), T)
        assert np.array_equal(np.reshape(h.E(), E.shape), E)
        assert np.array_equal(np.reshape(h.O(), O.shape), O)
    hs[0].step(1, allow=(4, 5))
    assert np.all(np.isfinite(hs[0].O(allow=(4, 5))))
    assert np.array_equal(np.reshape(hs[1].O(), state[1][2].shape), state[1][2])
    for h in hs:
        h.close()

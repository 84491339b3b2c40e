"""A temperature whose fourth power is not finite is accepted by grte_diff_set_T and gives a NaN right-hand
side in every cell: the diffusion solver reports GRTE_ENAN (a NaN R is neither > 0 nor <= 0), on
the one-kernel path (one CTA and a cluster) and on the three-launch path; R < 0 stays GRTE_ENEGATIVE."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1811_05579_gb300 import grte
    return grte


@pytest.mark.parametrize("kind", ["SIGMA_CONST", "SIGMA_T3"])
@pytest.mark.parametrize("N", [2, 100, 700, 8193])
def test_nan_is_reported(G, N, kind):
    h = G.Diffusion([dict(nx=N, sigma=1.0, dt=1e-3, kind=getattr(G, kind))])
    h.set_T(0, np.full(N, 1e80))
    h.step(1)
    with pytest.raises(G.GrteError) as e:
        h.T(0)
    assert e.value.status == G.GRTE_ENAN
    h.close()


@pytest.mark.parametrize("N", [100, 700, 8193])
def test_negative_right_hand_side(G, N):
    rng = np.random.default_rng(97)     # rough data and a long step: min R = -2.6, -16, -76
    T, sig = 0.5 + rng.random(N), 0.2 + 2.0 * rng.random(N)
    h = G.Diffusion([dict(nx=N, sigma=sig, dt=0.5 / N, kind=G.SIGMA_T3)])
    h.set_T(0, T)
    h.step(1)
    with pytest.raises(G.GrteError) as e:
        h.T(0)
    assert e.value.status == G.GRTE_ENEGATIVE
    assert np.min(h.T(0, allow=(G.GRTE_ENEGATIVE,))) == 0.0
    h.close()

"""U*^{3/4} and the correction's root outside the binary32 range, at inputs where they decide the result:
runs at T ~ 2^27 (U* and R above 1e30) and T ~ 2^-30 (below 1e-30) with sigma and C_v scaled so that
diffusion and heat capacity keep their weight, in which case the exact result is the scaled unit
run.  Compared per cell.  Bound: a flux is G = max dt a c kappa*/(D sigma dx^2) times the
difference of two U*, each good to four ulps of max U*; in T that is 4 eps (1 + 4 G) max U*/(T (4 T^3 + 1))
a step.  Planted in the oracle on the CPU, V = 0, V = U* and the root's start in place of the root
are all far outside it."""
import numpy as np
import pytest

from oracle import diffusion1d as dif
from oracle import scalar

SIZES = (100, 700, 8200)


def _run(N, step=dif.three_stage_step):
    rng = np.random.default_rng(N)
    x = (np.arange(N) + 0.5) / N
    T0 = 1.0 + 0.4 * np.sin(2 * np.pi * x) + 0.2 * np.sin(14 * np.pi * x + 1.0)
    sig, dt = 0.2 + 2.0 * rng.random(N), 0.05 / N
    T, Us = step(T0, sig, 1.0 / N, dt, kind="t3")
    G = dt * N * N / (3.0 * sig.min()) * np.max(Us) ** 0.75
    return T0, sig, dt, T, 4 * 2.2e-16 * (1 + 4 * G) * np.max(Us) / (T * (4 * T ** 3 + 1))


@pytest.mark.parametrize("N", SIZES)
def test_planted_mistakes_are_outside_the_bound(N, monkeypatch):
    T0, sig, dt, T, bound = _run(N)

    def planted(power):     # kappa* from another power of U* (None: 0)
        sn = 2 * sig[:-1] * sig[1:] / (sig[:-1] + sig[1:])
        _, Us = dif.three_stage_step(T0, sig, 1.0 / N, dt, kind="t3")
        V = np.zeros(N) if power is None else Us ** power
        f = 0.5 * (V[:-1] + V[1:]) / (3.0 * sn) * N * N * np.diff(Us)
        R = T0 ** 4 + T0 + dt * (np.append(f, 0.0) - np.append(0.0, f))
        return scalar.quartic_root(1.0, 1.0, R)[0], np.minimum(R ** 0.25, R)

    good, start = planted(0.75)
    assert np.all(np.abs(good - T) <= bound * T)
    for bad in (planted(None)[0], planted(1.0)[0], start):
        assert np.median(np.abs(bad - T) / (bound * T)) > 1e4


@pytest.mark.gpu
@pytest.mark.parametrize("e", [27, -30])
@pytest.mark.parametrize("N", SIZES)
def test_outside_the_binary32_range_per_cell(N, e):
    from paper_1811_05579_gb300 import grte as G
    T0, sig, dt, T, bound = _run(N)
    s = 2.0 ** e
    U = T ** 4 * s ** 4
    assert U.min() > 1e30 if e > 0 else U.max() < 1e-30
    h = G.Diffusion([dict(nx=N, sigma=sig * s ** 3, dt=dt, Cv=s ** 3, kind=G.SIGMA_T3)])
    h.set_T(0, T0 * s)
    h.step(1)
    assert np.all(np.abs(h.T(0) / s - T) <= bound * T)
    h.close()

"""The diffusion solver at the ends of the binary64 range, on the one-kernel path (one CTA and a cluster)
and the three-launch path.  The equations are invariant under T -> s T, U -> s^4 U with C_v -> s^3
C_v and, for sigma_0/T^3, sigma -> s^3 sigma; with s a power of two the scaled run is the unit run
bit for bit up to the rounding of its range-dependent starts.  Bounds against the oracle's unit run:
U* 1e-12 of the largest value and step; T the rounding of the correction's flux, two terms of
G = max dt a c kappa*/(D sigma dx^2) times the difference of two U*, each good to four ulps:
4 eps (1 + 4 G) a step."""
import numpy as np
import pytest

from oracle import diffusion1d as dif

pytestmark = pytest.mark.gpu
SIZES = (100, 700, 8200)
STEPS = 2


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1811_05579_gb300 import grte
    return grte


@pytest.fixture(scope="module")
def unit():
    """(N, form, T^0, sigma, dt, T, U*) at unit scale, from the oracle."""
    rng = np.random.default_rng(97)
    out = []
    for N in SIZES:
        for kind in ("const", "t3"):
            x = (np.arange(N) + 0.5) / N   # smooth: no cell empties (T >= 0.4 throughout)
            T0 = 1.0 + 0.4 * np.sin(2 * np.pi * x) + 0.2 * np.sin(14 * np.pi * x + 1.0)
            sig, dt = 0.2 + 2.0 * rng.random(N), 0.05 / N
            T = T0
            for _ in range(STEPS):
                T, Us = dif.three_stage_step(T, sig, 1.0 / N, dt, kind=kind)
            assert T.min() > 0.4
            out.append((N, kind, T0, sig, dt, T, Us))
    return out


def check(G, unit, exps, sizes=SIZES):
    """Each form scaled by 2^exps[form]."""
    runs = [(2.0 ** exps[u[1]], u) for u in unit if u[1] in exps and u[0] in sizes]
    h = G.Diffusion([dict(nx=N, sigma=sig * (s ** 3 if kind == "t3" else 1.0), dt=dt, Cv=s ** 3,
                          kind=G.SIGMA_T3 if kind == "t3" else G.SIGMA_CONST) for s, (N, kind, _, sig, dt, _, _) in runs])
    for i, (s, u) in enumerate(runs):
        h.set_T(i, u[2] * s)
    h.step(STEPS)
    for i, (s, (N, kind, _, sig, dt, T, Us)) in enumerate(runs):
        G_ = dt * N * N / (3.0 * sig.min()) * (np.max(Us) ** 0.75 if kind == "t3" else 1.0)
        eT = np.max(np.abs(h.T(i) / s - T)) / np.max(T)
        eU = np.max(np.abs(h.Ustar(i) / s / s / s / s - Us)) / np.max(Us)
        assert eT < 4 * 2.2e-16 * (1 + 4 * G_) * STEPS and eU < 1e-12 * STEPS, (N, kind, eT, eU)
    h.close()


# T^7, the size of the stage-1 rows times a T^3 + C_v/4, leaves binary64 at 2^146, T^4 at 2^256; the
# flux of sigma_0/T^3 is itself of the size of T^7.
@pytest.mark.parametrize("exps", [dict(const=0, t3=0), dict(const=150, t3=140), dict(const=-150, t3=-90),
                                  dict(const=230), dict(const=-230)])
def test_far_from_one(G, unit, exps):
    check(G, unit, exps)


# (three launches solve for U*/dt rows, which leave the range earlier)
def test_up_to_the_end_of_the_range(G, unit):
    check(G, unit, dict(const=250), sizes=(100, 700))


# sigma -> s sigma, dt -> s dt leaves a step as it is: the node factor's sigma_l sigma_r stays in the
# binary64 range at s = 2^-510 (sigma >= 1), times dx^2 it would have 28 bits left.
def test_small_sigma(G):
    rng = np.random.default_rng(98)
    N, s = 8192, 2.0 ** -510
    x = (np.arange(N) + 0.5) / N
    T0, sig, dt = 1.0 + 0.4 * np.sin(2 * np.pi * x), 1.0 + rng.random(N), 0.05 / N
    for kind, okind in ((G.SIGMA_CONST, "const"), (G.SIGMA_T3, "t3")):
        T, Us = dif.three_stage_step(T0, sig, 1.0 / N, dt, kind=okind)
        h = G.Diffusion([dict(nx=N, sigma=sig * s, dt=dt * s, kind=kind)])
        h.set_T(0, T0)
        h.step(1)
        G_ = dt * N * N / 3.0 * (np.max(Us) ** 0.75 if okind == "t3" else 1.0)
        assert np.max(np.abs(h.T(0) - T)) / np.max(T) < 4 * 2.2e-16 * (1 + 4 * G_)
        assert np.max(np.abs(h.Ustar(0) - Us)) / np.max(Us) < 1e-13
        h.close()


# Rows are scaled from T = 2^128 on: cells on both sides of it in every CTA (a = C_v = 1, the oracle on
# the same inputs; T^7 = 2^901 is in its range).
def test_cells_on_both_sides_of_the_scaled_range(G, unit):
    s = 2.0 ** 128
    for N, kind, T0, sig, dt, _, _ in unit:
        assert np.any(T0 < 0.9) and np.any(T0 > 1.1)
        sg = sig * (s ** 3 if kind == "t3" else 1.0)
        T, Us = dif.three_stage_step(T0 * s, sg, 1.0 / N, dt, kind=kind)
        h = G.Diffusion([dict(nx=N, sigma=sg, dt=dt, kind=G.SIGMA_T3 if kind == "t3" else G.SIGMA_CONST)])
        h.set_T(0, T0 * s)
        h.step(1)
        G_ = dt * N * N / (3.0 * sg.min()) * (np.max(Us) ** 0.75 if kind == "t3" else 1.0)
        assert np.max(np.abs(h.T(0) - T)) / np.max(T) < 4 * 2.2e-16 * (1 + 4 * G_)
        assert np.max(np.abs(h.Ustar(0) - Us)) / np.max(Us) < 1e-12
        h.close()

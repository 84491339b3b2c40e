"""Kernels at the edges of their tiles, slices and size rules: the network's inference, the
state's layout changes, the FP64 Krylov kernels (one CTA up to 256 cells, clusters of 8, of 16
from 2048 cells for up to seven instances), the one-kernel solve's exact cluster sizes and the
three tilings of the 2D operator pass."""
import numpy as np
import pytest

from oracle import grte1d as og
from oracle.quadrature import gauss_legendre_half
from paper_1811_05579_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1811_05579_gb300 import grte
    return grte


def make(N, nv, eps, kind="t3", bc="inflow", cfl=0.1, lo=0.3, seed=0):
    v, w = gauss_legendre_half(nv)
    rng = wl.SplitMix64(9000 + seed)
    P = og.Problem(N=N, v=v, w=w, sig=0.5 + 2.0 * rng.uniform(N), eps=eps, dt=cfl / N, kind=kind, bc=bc,
                   bL=np.full(v.size, 1.0), bR=np.full(v.size, 0.1))
    spec = dict(nx=N, n_angle=v.size, v=v, w=w, sigma=P.sig, kind=1 if kind == "t3" else 0,
                bc=0 if bc == "inflow" else 1, bL=P.bL, bR=P.bR, dt=P.dt, eps=eps)
    T, E, O = wl.random_state_1d(rng, N, P.M, (lo, 1.0))
    if bc == "reflect":
        O[0] = O[-1] = 0.0
    return P, spec, og.State(E=E, O=O, U=T ** 4, T=T)


# Both tilings work on samples one by one with the same operations: a sample's result does not
# depend on the batch it comes in, so every size agrees bit for bit with the full batch.
@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 33, 127, 129, 4097, 38911, 38912, 38913, 77825])
def test_inference_sizes(G, n):
    rng = np.random.default_rng(11)
    m = G.MLP(seed=2)
    X = rng.standard_normal((80001, 6)).astype(np.float32)
    m.set_norm(np.zeros(6, np.float32), np.ones(6, np.float32), 0.1, 2.0)
    full = m.forward(X)
    for lo in (0, 80001 - n):
        assert np.array_equal(m.forward(X[lo:lo + n]), full[lo:lo + n])
    m.close()


# The device keeps E - a c U and O in its bulk type: FP64 returns O exactly and E to two
# roundings of max(E, a c U); binary32 to its unit roundoff 6e-8 of the same.
@pytest.mark.parametrize("nv", [2, 62, 64, 66])
@pytest.mark.parametrize("N", [2, 31, 32, 33, 65])
def test_state_round_trip(G, N, nv):
    P, spec, S = make(N, nv, 1e-2)
    for prec, u in ((G.FP64, 1.2e-16), (G.MIXED, 6e-8)):
        h = G.Grte([spec], precision=prec)
        h.set_state(0, S.T, S.E, S.O)
        scale = np.maximum(np.abs(S.E), S.U[:, None])
        assert np.array_equal(h.T(0), S.T)
        assert np.all(np.abs(h.E(0) - S.E) <= 2.1 * u * scale)
        assert np.all(np.abs(h.O(0) - S.O) <= (0.0 if prec == G.FP64 else u) * np.abs(S.O))
        h.close()


# The prediction is solved to 1e-13 of every cell; T sees the flux difference over eps dx, here
# at most 1e2 times that: 1e-11 against the oracle.
@pytest.mark.parametrize("kind,bc", [("t3", "inflow"), ("const", "reflect")])
@pytest.mark.parametrize("N", [2, 3, 16, 17, 255, 256, 257, 300, 2047, 2048, 2063])
def test_fp64_krylov_slices(G, N, kind, bc):
    P, spec, S = make(N, 8, 1e-2, kind, bc, seed=N)
    h = G.Grte([spec])
    h.set_state(0, S.T, S.E, S.O)
    h.step(1)
    S1 = og.step(P, S)
    assert np.max(np.abs(h.T(0, allow=(5,)) - S1.T) / np.maximum(np.abs(S1.T), 1e-300)) < 1e-11
    h.close()


def test_fp64_cluster_sizes_agree(G):
    """Seven instances take clusters of sixteen, nine of the same clusters of eight."""
    P, spec, S = make(2100, 8, 1e-2, seed=5)
    out = []
    for n in (7, 9):
        h = G.Grte([spec] * n)
        for i in range(n):
            h.set_state(i, S.T, S.E, S.O)
        h.step(2)
        T = [h.T(i, allow=(5,)) for i in range(n)]
        assert all(np.array_equal(t, T[0]) for t in T)
        out.append(T[0])
        h.close()
    assert np.max(np.abs(out[0] - out[1]) / out[1]) < 2e-11


# A class of every cluster size in one handle, solved side by side: the bits of each run alone.
def test_fused_clusters_side_by_side(G):
    sizes = [64, 511, 512, 513, 1025, 1537, 2561, 3585, 4096, 5633, 6657, 7681]
    runs = [make(N, 8, 10.0 ** (-(i % 3)), seed=i) for i, N in enumerate(sizes)]
    h = G.Grte([r[1] for r in runs], precision=G.MIXED, line_threads=256)
    for i, (_, _, S) in enumerate(runs):
        h.set_state(i, S.T, S.E, S.O)
    h.step(2)
    for i, (_, spec, S) in enumerate(runs):
        one = G.Grte([spec], precision=G.MIXED, line_threads=256)
        one.set_state(0, S.T, S.E, S.O)
        one.step(2)
        assert np.array_equal(h.T(i, allow=(4, 5)), one.T(0, allow=(4, 5))), sizes[i]
        one.close()
    h.close()


# y-periodic data: replicas of a 97 x 24 problem (the smallest tiling, checked against the oracle
# by the other tests) over enough rows for the two wider tilings give every row of the small
# one.  The solves stop at 1e-13 of the residual; 1e-9 leaves four decades for its conditioning.
@pytest.mark.parametrize("copies", [9, 51])
@pytest.mark.parametrize("mixed", [False, True])
def test_2d_operator_tilings(G, copies, mixed):
    rng = np.random.default_rng(31)
    nx, ny = 97, 24
    sig = 0.5 + rng.random((ny, nx))
    T0 = 0.5 + 0.5 * rng.random((ny, nx))
    res = []
    for c in (1, copies):
        h = G.Grte2D(nx, ny * c, np.tile(sig, (c, 1)), 0.2 / nx, 1e-1, kind=G.SIGMA_T3, bc_x=G.BC_INFLOW,
                     bc_y=G.BC_PERIODIC, b_x0=1.0, b_x1=0.3, lx=1.0, ly=ny * c / nx,
                     precision=G.MIXED if mixed else G.FP64)
        h.set_state(np.tile(T0, (c, 1)))
        h.step(1, allow=(5,))
        res.append(h.T(allow=(5,)).reshape(c, ny, nx))
        h.close()
    assert np.max(np.abs(res[1] - res[0]) / res[0]) < (1e-5 if mixed else 1e-9)


@pytest.mark.parametrize("restart", [3, 16, 17, 64])
def test_2d_restart_lengths(G, restart):
    rng = np.random.default_rng(32)
    nx, ny = 33, 9
    sig, T0 = 0.5 + 20.0 * rng.random((ny, nx)), 0.5 + 0.5 * rng.random((ny, nx))
    res = []
    for m in (30, restart):
        h = G.Grte2D(nx, ny, sig, 0.5 / nx, 1e-2, kind=G.SIGMA_T3, bc_x=G.BC_INFLOW, bc_y=G.BC_PERIODIC, b_x0=1.0,
                     krylov_restart=m, krylov_maxcycles=200)
        h.set_state(T0)
        h.step(1, allow=(5,))
        res.append(h.T(allow=(5,)))
        h.close()
    assert np.max(np.abs(res[1] - res[0]) / res[0]) < 1e-9


# The gradient of n samples is the mean of those of its parts (block edges at 64, eight groups of
# blocks in the reduction).  The same products in both: only binary32 sums of up to n terms are
# ordered differently, 1e-5 of the largest entry; the samples' BF16 operands are the same but for
# the 1/n in front, which moves their rounding by up to 2^-8 of single terms: 2e-3.
@pytest.mark.parametrize("n", [1, 63, 64, 65, 448, 512, 513, 577])
def test_gradient_block_edges(G, n):
    rng = np.random.default_rng(12)
    m = G.MLP(seed=4)
    m.set_norm(np.zeros(6, np.float32), np.ones(6, np.float32), 0.0, 1.0)
    X = rng.standard_normal((n, 6)).astype(np.float32)
    Y = rng.standard_normal(n).astype(np.float32)
    loss, g = m.grad(X, Y)
    parts = [(len(X[i:i + 50]), m.grad(X[i:i + 50], Y[i:i + 50])) for i in range(0, n, 50)]
    want_l = sum(k * p[0] for k, p in parts) / n
    want = sum(k * p[1].astype(np.float64) for k, p in parts) / n
    assert abs(loss - want_l) < 1e-5 * want_l
    assert np.max(np.abs(g - want)) < 2e-3 * np.max(np.abs(want))
    m.close()

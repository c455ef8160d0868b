"""Conserved sums of long FP32 runs: what a step's constants are off adds up from step to step."""
import numpy as np
import pytest

from lbe_cases import rel_err, setup_gpu, setup_oracle

pytestmark = pytest.mark.gpu

CX = np.array([0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0])
CY = np.array([0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1])
CZ = np.array([0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1])
W = np.array([12.0] + [2.0] * 6 + [1.0] * 12) / 36.0


@pytest.mark.parametrize("tau", [0.8, 1.0, 0.7])
@pytest.mark.parametrize("M", [1, 2])
def test_fp32_momentum_of_a_periodic_gas(M, tau):
    """Total momentum of an ideal gas in uniform flow over 1000 steps.  One rounding of a node's momentum (2^-24) has no
    preferred sign, so over 4096 nodes a step's sum is off by 2^-24 / 64 at most in the mean: 1e-6 in 1000 steps.  The
    bound is ten times that; a constant off by 3e-8 in each step gives 3e-5."""
    shape, N, u = (16, 16, 16), 4096, np.array([0.04, -0.03, 0.02])
    rng = np.random.default_rng(3)
    n = 0.05 * (1.0 + 0.02 * (rng.random((M, N)) - 0.5))
    arr = dict(solid=np.zeros(N, np.uint8), V=np.zeros((M, N)), phi=np.zeros(N), amp=np.zeros(N), n=n)
    w = dict(shape=shape, periodic=(1, 1, 1), sigma=[0.0] * M, tau=[tau] * M, body=[(0.0, 0.0, 0.0)] * M)
    g = setup_gpu(w, arr, "fp32")
    cu = CX * u[0] + CY * u[1] + CZ * u[2]
    feq = W * (1.0 + 3.0 * cu + 4.5 * cu ** 2 - 1.5 * (u ** 2).sum())
    for a in range(M):
        g.set_populations(a, feq[:, None] * n[a], feq[:, None] * n[a])
    mass0, mom0, _ = g.totals()
    g.step(1000)
    mass, mom, _ = g.totals()
    assert np.abs(mom - mom0).max() <= 1e-5 * np.abs(mom0).max()
    assert np.abs(mass - mass0).max() <= 1e-6 * mass0.max()


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("fp64", 1e-12)])
@pytest.mark.parametrize("M", [1, 2, 3])
def test_nodes_without_density(M, prec, tol):
    """Populations after a collision where f sums to 0 and g does not: velocity and equilibrium are 0 there."""
    shape, N = (9, 5, 4), 180
    rng = np.random.default_rng(8)
    arr = dict(solid=np.zeros(N, np.uint8), V=np.zeros((M, N)), phi=np.zeros(N), amp=np.zeros(N),
               n=np.zeros((M, N)))  # deviations from 0: such a node sums to 0 exactly
    w = dict(shape=shape, periodic=(1, 1, 1), sigma=[0.0] * M, tau=[0.8] * M, body=[(1e-3, 0.0, 0.0)] * M)
    g, o = setup_gpu(w, arr, prec), setup_oracle(w, arr)
    empty = rng.random(N) < 0.3
    for a in range(M):
        f = W[:, None] * 0.05 * (1.0 + 0.1 * rng.random((19, N)))
        q = W[:, None] * 0.05 * (1.0 + 0.1 * rng.random((19, N)))
        f[:, empty] = 0.0
        g.set_populations(a, f, q)
        o.set_populations(a, f, q)
    g.step(1)
    o.step(1)
    for a in range(M):
        for got, ref in zip(g.populations(a), o.get_populations(a)):
            assert rel_err(np.asarray(got).reshape(-1), np.asarray(ref).reshape(-1)) <= tol

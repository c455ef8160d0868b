"""Conserved sums of long FP32 runs: what a step's constants are off adds up from step to step."""
import numpy as np
import pytest

from lbe_cases import setup_gpu

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

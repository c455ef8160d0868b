"""Collision for one to four species in every storage type, against the oracle: a lattice of few nodes (small
CTAs, a last CTA that is mostly empty) and one of enough nodes for the full CTAs, both with odd rows and scattered
solid nodes; the single-distribution ablations at the second size."""
import numpy as np
import pytest

from lbe_cases import rel_err, setup_gpu, setup_oracle

pytestmark = pytest.mark.gpu

SMALL, LARGE = (33, 5, 7), (65, 37, 41)
SIGMA = (2.0, 4.0, 2.0, 4.0)
STEPS = 3
# unit round-off of the stored deviation of a population from w_p n0
ROUND = {"bf16": 2.0 ** -8, "fp16": 2.0 ** -11}


def pair_of_runs(shape, M, prec, scheme="dd_tr"):
    N = int(np.prod(shape))
    rng = np.random.default_rng(97)
    solid = (rng.random(N) < 0.05).astype(np.uint8)
    sig = SIGMA[:M]
    n0 = 6.0 * 0.1 / (np.pi * sum(s ** 3 for s in sig))
    arr = dict(solid=solid, V=np.zeros((M, N)), phi=np.zeros(N), amp=np.zeros(N),
               n=n0 * (1.0 + 0.3 * (rng.random((M, N)) - 0.5)) * (solid == 0)[None, :])
    w = dict(shape=shape, periodic=(1, 0, 1), sigma=list(sig), tau=[0.8, 1.0, 0.9, 1.1][:M],
             body=[(1e-3, 0.0, -1e-3)] * M)
    g = setup_gpu(w, arr, prec, scheme=scheme)
    o = setup_oracle(w, arr, scheme=scheme)
    g.step(STEPS)
    o.step(STEPS)
    return g, o, n0


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16", "fp16"])
@pytest.mark.parametrize("M", [1, 2, 3, 4])
@pytest.mark.parametrize("shape", [SMALL, LARGE])
def test_populations(shape, M, prec):
    """FP64 round-off and FP32 round-off as in the parity tests.  16 bits: each step rounds every stored deviation once
    (ROUND times the largest, D), and the collision spreads the rounding of the populations it sums, over the species
    too: 5 such errors per step."""
    g, o, n0 = pair_of_runs(shape, M, prec)
    scale = np.array([12.0] + [2.0] * 6 + [1.0] * 12)[:, None] / 36.0 * n0
    ref = np.array([o.get_populations(a) for a in range(M)]).reshape(M, 2, 19, -1) / scale
    got = np.array([g.populations(a) for a in range(M)]).reshape(M, 2, 19, -1) / scale
    fluid = np.abs(ref).max((0, 1, 2)) > 0
    dev = np.abs(ref[..., fluid] - 1.0).max()
    tol = {"fp64": 1e-12, "fp32": 1e-5}.get(prec) or 5 * STEPS * ROUND[prec] * dev
    assert np.abs(got - ref).max() <= tol * np.abs(ref).max()


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("scheme", ["sd_tr", "sd_eu", "dd_eu"])
@pytest.mark.parametrize("M", [1, 2])
def test_ablations_full_blocks(M, scheme, prec, tol):
    g, o, _ = pair_of_runs(LARGE, M, prec, scheme)
    for a in range(M):
        for got, ref in zip(g.populations(a), o.get_populations(a)):
            assert rel_err(np.asarray(got), np.asarray(ref)) <= tol


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_auto_takes_the_stencil_on_large_lattices(prec):
    """Which form AUTO takes does not change the force beyond round-off."""
    shape = (32, 26, 20)  # 16640 nodes
    N = int(np.prod(shape))
    rng = np.random.default_rng(5)
    arr = dict(solid=np.zeros(N, np.uint8), V=np.zeros((1, N)), phi=np.zeros(N), amp=np.zeros(N),
               n=2e-3 * (1.0 + 0.3 * (rng.random((1, N)) - 0.5)))
    w = dict(shape=shape, periodic=(1, 1, 1), sigma=[6.0], tau=[1.0], body=[(0.0, 0.0, 0.0)])
    auto, spectral = setup_gpu(w, arr, prec), setup_gpu(w, arr, prec, shell="spectral")
    assert auto.shell_method() == "direct" and spectral.shell_method() == "spectral"
    assert rel_err(auto.force(0), spectral.force(0)) <= (1e-12 if prec == "fp64" else 1e-5)
    # FP32 runs of the single-distribution schemes keep the rule of small lattices
    single = setup_gpu(w, arr, prec, scheme="sd_tr")
    assert single.shell_method() == ("direct" if prec == "fp64" else "spectral")


@pytest.mark.parametrize("scale", [1e-312, 1e-290, 1e-20, 1.0, 1e200])
def test_fp64_moments_of_any_magnitude(scale):
    """Density and momentum of FP64 populations over 30 decades at one node, at both ends of the exponent range, and
    with zeros: a sum of 19 terms is within 18 round-offs of the terms' magnitudes (a subnormal term's last bit)."""
    shape, N = (9, 4, 3), 108
    rng = np.random.default_rng(11)
    arr = dict(solid=np.zeros(N, np.uint8), V=np.zeros((1, N)), phi=np.zeros(N), amp=np.zeros(N), n=np.ones((1, N)))
    w = dict(shape=shape, periodic=(1, 1, 1), sigma=[0.0], tau=[1.0], body=[(0.0, 0.0, 0.0)])
    g = setup_gpu(w, arr, "fp64")
    f = scale * rng.random((19, N)) * 10.0 ** rng.uniform(-20, 3, (19, N)) * (rng.random((19, N)) < 0.8)
    gq = scale * rng.standard_normal((19, N)) * 10.0 ** rng.uniform(-20, 3, (19, N))
    g.set_populations(0, f, gq)
    ulp = 18 * 2.0 ** -53
    assert (np.abs(g.density(0) - f.sum(0)) <= 2 * ulp * f.sum(0) + 19 * 5e-324).all()
    pairs = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]
    J = np.asarray(g.momentum(0)).reshape(3, N)
    for c in range(3):
        ref = sum(p[c] * (gq[1 + 2 * k] - gq[2 + 2 * k]) for k, p in enumerate(pairs))
        assert (np.abs(J[c] - ref) <= 2 * ulp * np.abs(gq).sum(0) + 19 * 5e-324).all()
    back_f, back_g = g.populations(0)
    assert np.array_equal(back_f, f) and np.array_equal(back_g, gq)

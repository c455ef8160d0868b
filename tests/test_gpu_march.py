"""Contact values and shell force of the marching kernels at the edges of their tiles, against the oracle:
lattices of one plane, narrower than a tile or a shell, odd rows (no 8-byte rows), one node more than a tile,
periodic axes shorter than the shell (several images of a node in the halo), and up to four species."""
import numpy as np
import pytest

from lbe_cases import rel_err, setup_gpu, setup_oracle

pytestmark = pytest.mark.gpu

CASES = [
    ((33, 5, 7), (1, 1, 1), (6.0,)),
    ((32, 4, 1), (1, 1, 0), (4.0,)),
    ((7, 3, 2), (1, 1, 1), (5.0,)),
    ((1, 9, 40), (0, 1, 1), (3.0, 5.0)),
    ((65, 6, 13), (1, 0, 0), (4.0, 6.0)),
    ((30, 11, 26), (0, 0, 1), (2.0, 4.0, 6.0)),
    ((18, 17, 15), (1, 1, 1), (1.0, 3.0, 5.0, 7.0)),
    ((34, 9, 18), (0, 0, 0), (8.0,)),
    ((16, 16, 64), (1, 1, 1), (0.0, 4.0)),
]


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("fp64", 1e-12)])
@pytest.mark.parametrize("shape,periodic,sig", CASES)
def test_march_edges(shape, periodic, sig, prec, tol):
    """Tolerances of the stage parity: FP32 sums of up to 762 points, FP64 round-off, of a field's largest value."""
    N, M = int(np.prod(shape)), len(sig)
    rng = np.random.default_rng(31)
    solid = (rng.random(N) < 0.06).astype(np.uint8)
    solid[rng.integers(N)] = 0
    n0 = 6.0 * 0.12 / (np.pi * sum(s ** 3 for s in sig))
    arr = dict(solid=solid, V=np.zeros((M, N)), phi=np.zeros(N), amp=np.zeros(N),
               n=n0 * (1.0 + 0.3 * (rng.random((M, N)) - 0.5)) * (solid == 0)[None, :])
    w = dict(shape=shape, periodic=periodic, sigma=list(sig), tau=[1.0] * M, body=[(0.0, 0.0, 0.0)] * M)
    if prec == "fp64" and max(sig) > 7:
        pytest.skip("no direct FP64 stencil of this diameter")
    g = setup_gpu(w, arr, prec, shell="direct")
    o = setup_oracle(w, arr)
    obs = o.observe()
    for a in range(M):
        for b in range(M):
            if sig[a] + sig[b] > 0:
                assert rel_err(g.contact(a, b), obs["g"][a, b]) <= tol
        scale = np.abs(obs["C"][a]).max()
        if scale > 0:
            assert rel_err(g.force(a), obs["C"][a]) <= tol
        else:
            assert np.abs(g.force(a)).max() <= tol * n0


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("fp64", 1e-12)])
@pytest.mark.parametrize("sig", [(2.0,), (4.0,), (6.0,), (7.0,), (8.0,), (2.0, 4.0, 6.0, 8.0), (6.0, 0.0)])
def test_diameters_a_rounding_off_an_integer(sig, prec, tol):
    """Diameters are integers to 1e-12.  Just below an even one the ball |d| <= sigma/2 ends before the points at sigma/2,
    just above any it is the integer's."""
    if prec == "fp64" and max(sig) > 7:
        pytest.skip("no direct FP64 stencil of this diameter")
    shape, N, M = (19, 10, 9), 1710, len(sig)
    rng = np.random.default_rng(7)
    n0 = 6.0 * 0.1 / (np.pi * sum(s ** 3 for s in sig))
    for off in (-1e-13, 1e-13):
        s = [v * (1.0 + off) for v in sig]
        arr = dict(solid=np.zeros(N, np.uint8), V=np.zeros((M, N)), phi=np.zeros(N), amp=np.zeros(N),
                   n=n0 * (1.0 + 0.3 * (rng.random((M, N)) - 0.5)))
        w = dict(shape=shape, periodic=(1, 1, 1), sigma=s, tau=[1.0] * M, body=[(0.0, 0.0, 0.0)] * M)
        g, o = setup_gpu(w, arr, prec, shell="direct"), setup_oracle(w, arr)
        obs = o.observe()
        for a in range(M):
            for b in range(M):
                if s[a] + s[b] > 0:
                    assert rel_err(g.contact(a, b), obs["g"][a, b]) <= tol
            assert rel_err(g.force(a), obs["C"][a]) <= tol


@pytest.mark.parametrize("prec,tol,shape,sig", [
    ("fp64", 1e-12, (4, 131076, 2), 2.0),  # more rows than 65535 tiles of two hold
    ("fp32", 1e-5, (2, 262148, 1), 3.0),   # of four
    ("fp32", 1e-5, (4, 3, 65540), 1.0),    # more planes than a grid is long, where marches of one plane are cheapest
    ("fp64", 1e-12, (4, 3, 65540), 1.0),
])
def test_long_axes(prec, tol, shape, sig):
    """The same lattice with its long axis along x, where no limit lies, up to round-off."""
    rng = np.random.default_rng(9)
    nx, ny, nz = shape
    n = 6.0 * 0.1 / (np.pi * sig ** 3) * (1.0 + 0.3 * (rng.random((nz, ny, nx)) - 0.5))

    def run(n, shape):
        N = n.size
        arr = dict(solid=np.zeros(N, np.uint8), V=np.zeros((1, N)), phi=np.zeros(N), amp=np.zeros(N),
                   n=np.ascontiguousarray(n).reshape(1, N))
        w = dict(shape=shape, periodic=(1, 1, 1), sigma=[sig], tau=[1.0], body=[(0.0, 0.0, 0.0)])
        g = setup_gpu(w, arr, prec, shell="direct")
        c = g.force(0).reshape((3,) + n.shape)
        g.step(2)
        return g.density(0).reshape(n.shape), c

    swap = 1 if ny > nz else 0  # the long axis of an array [z][y][x]
    d, c = run(n, shape)
    e, f = run(np.swapaxes(n, swap, 2), (ny, nx, nz) if swap else (nz, ny, nx))
    order = [1, 0, 2] if swap else [2, 1, 0]
    assert rel_err(d, np.swapaxes(e, swap, 2)) <= tol
    assert rel_err(c, np.swapaxes(f, swap + 1, 3)[order]) <= tol


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("fp64", 1e-12)])
@pytest.mark.parametrize("shape,periodic,sig", [
    ((37, 97, 1), (1, 1, 1), (6.0,)),            # one node along z: the march goes along y
    ((37, 97, 1), (0, 1, 0), (5.0,)),
    ((66, 301, 2), (1, 0, 1), (4.0, 6.0)),
    ((33, 150, 3), (1, 1, 0), (2.0, 4.0, 6.0)),
    ((5, 1030, 5), (1, 1, 1), (7.0,)),
    ((35, 1, 90), (1, 1, 1), (4.0,)),            # one along y: it stays along z
])
def test_march_along_the_longer_axis(shape, periodic, sig, prec, tol):
    test_march_edges(shape, periodic, sig, prec, tol)
    # the adjoint keeps P of every pair: the transposed and the spectral form on the same lattice
    if prec == "fp64" and len(sig) < 3:
        N, M = int(np.prod(shape)), len(sig)
        rng = np.random.default_rng(2)
        n0 = 6.0 * 0.12 / (np.pi * sum(s ** 3 for s in sig))
        arr = dict(solid=np.zeros(N, np.uint8), V=np.zeros((M, N)), phi=np.zeros(N), amp=np.zeros(N),
                   n=n0 * (1.0 + 0.3 * (rng.random((M, N)) - 0.5)))
        w = dict(shape=shape, periodic=periodic, sigma=list(sig), tau=[1.0] * M, body=[(1e-4, 0.0, 0.0)] * M)
        x, y = (np.asarray(setup_gpu(w, arr, prec, shell=m).adjoint_flux_gradient(2, 1, 0, 3)[2])
                for m in ("direct", "spectral"))
        assert np.abs(x - y).max() <= 1e-10 * np.abs(y).max()

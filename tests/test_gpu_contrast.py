"""FP64 shell forces of fields whose values lie far apart: each node's force against the oracle, to the round-off of the
values on that node's own shells (fixed-point sums in units of the field's largest value would lose them)."""
import numpy as np
import pytest

import oracle
from lbe_cases import setup_gpu, setup_oracle

pytestmark = pytest.mark.gpu


def shell_scale(shape, sig, n, g, a):
    """kT sigma^2 w n_a sum_e (g(r) + g(r + e)) / 2 n_b(r + e): the sum without its signs."""
    nx, ny, nz = shape
    total = np.zeros((nz, ny, nx))
    for b, s in enumerate(sig):
        d = (sig[a] + s) / 2
        e = np.asarray(oracle.shell(d)).reshape(-1, 3)
        w = 4 * np.pi * d / np.sqrt((e * e).sum(1)).sum()
        gab, nb = g[a, b].reshape(nz, ny, nx), n[b].reshape(nz, ny, nx)
        for v in e:
            at = (-v[2], -v[1], -v[0])
            total += d * d * w / 3 * 0.5 * (gab + np.roll(gab, at, (0, 1, 2))) * np.roll(nb, at, (0, 1, 2))
    return (total * n[a].reshape(nz, ny, nx)).reshape(-1)


@pytest.mark.parametrize("kind,sig,shell", [
    ("decades", (3.0,), "auto"), ("decades", (3.0,), "direct"), ("decades", (2.0, 4.0), "direct"),
    ("decades", (6.0,), "direct"), ("decades", (1.0, 3.0, 5.0, 7.0), "direct"), ("spike", (3.0,), "auto"),
    ("sparse", (3.0, 5.0), "direct")])
def test_fp64_force_is_exact_locally(kind, sig, shell):
    """1e-12, the parity of the stages, of the sum of the magnitudes on the node's shells."""
    shape = nx, ny, nz = 37, 11, 19
    N, M = nx * ny * nz, len(sig)
    rng = np.random.default_rng(17)
    n0 = 6.0 * 0.12 / (np.pi * sum(s ** 3 for s in sig))
    n = n0 * (1.0 + 0.3 * (rng.random((M, nz, ny, nx)) - 0.5))
    if kind == "decades":  # twelve decades along z
        n *= 10.0 ** (-12.0 * np.arange(nz) / (nz - 1))[None, :, None, None]
    elif kind == "spike":  # packing 0.99 around one node: contact values of 1e6 there
        balls = 19  # nodes of the ball of diameter 3
        n[0, 9, 5, 18] = balls * (0.99 * 6.0 / (np.pi * sig[0] ** 3) - 1.1 * n0)
    else:  # single nodes of fluid far below the others
        n[rng.random(n.shape) < 0.3] *= 1e-20
    arr = dict(solid=np.zeros(N, np.uint8), V=np.zeros((M, N)), phi=np.zeros(N), amp=np.zeros(N), n=n.reshape(M, N))
    w = dict(shape=shape, periodic=(1, 1, 1), sigma=list(sig), tau=[1.0] * M, body=[(0.0, 0.0, 0.0)] * M)
    g, obs = setup_gpu(w, arr, "fp64", shell=shell), setup_oracle(w, arr).observe()
    for a in range(M):
        scale = shell_scale(shape, sig, n.reshape(M, N), obs["g"], a)
        assert (np.abs(g.force(a) - obs["C"][a]) <= 1e-12 * scale).all()


@pytest.mark.parametrize("short_of", ["images", "scratch"])
@pytest.mark.parametrize("sig", [(3.0,), (2.0, 4.0)])
def test_no_room_for_the_images(sig, short_of, monkeypatch):
    """A device without room for the fixed-point images, or for a getter's scratch beside them: the stencil needs none."""
    from paper_1202_3842_gb300 import lbe
    shape, N, M = (20, 18, 16), 5760, len(sig)
    H = (int(max(sig)) + 3) // 4 * 4
    P = (shape[0] + 2 * H + 7) // 8 * 8 * (shape[1] + 2 * H) * (shape[2] + 2 * H)
    size = {"images": 8 * (M + M * M) * P, "scratch": 8 * (4 * M * N + 4 * N)}[short_of]
    refused = []

    class Full(lbe.TorchAllocator):
        def __init__(self, *args, **kw):
            super().__init__(*args, **kw)
            alloc = self._a

            def _alloc(nbytes, stream, user):
                if nbytes == (size + 255) // 256 * 256 and (short_of == "images" or not refused):
                    refused.append(nbytes)
                    return None
                return alloc(nbytes, stream, user)

            self._full = lbe._ALLOC_FN(_alloc)
            self.struct = lbe.lbe_allocator(self._full, self._f, None)

    rng = np.random.default_rng(4)
    n0 = 6.0 * 0.12 / (np.pi * sum(s ** 3 for s in sig))
    arr = dict(solid=np.zeros(N, np.uint8), V=np.zeros((M, N)), phi=np.zeros(N), amp=np.zeros(N),
               n=n0 * (1.0 + 0.3 * (rng.random((M, N)) - 0.5)))
    w = dict(shape=shape, periodic=(1, 1, 1), sigma=list(sig), tau=[1.0] * M, body=[(0.0, 0.0, 0.0)] * M)
    o = setup_oracle(w, arr)
    monkeypatch.setattr(lbe, "TorchAllocator", Full)
    g = setup_gpu(w, arr, "fp64", shell="direct")
    for _ in range(2):
        obs = o.observe()
        for a in range(M):
            assert np.abs(g.force(a) - obs["C"][a]).max() <= 1e-12 * np.abs(obs["C"][a]).max()
            assert np.abs(g.density(a) - obs["n"][a]).max() <= 1e-12 * n0
            J = obs["J"][a].reshape(-1)
            assert np.abs(np.asarray(g.momentum(a)).reshape(-1) - J).max() <= 1e-12 * np.abs(J).max()
        g.step(3)
        o.step(3)
    assert refused

"""Performance cases of the framework: calls of the public API over the range its users run.

A case is one lattice and what a program does with it between two looks at the result: so many time
steps and the fields it then reads ("fluid"), or one gradient of the averaged flux ("adjoint").  Sizes,
diameters, packings and relaxation times are those of ``inputs.WORKLOADS``, of the studies and of the
tests, and sizes between them, ragged ones among them.

The getters of the API hand every field out in FP64; ``run`` returns it in the type that the lattice
stores its populations in, as a program does that keeps snapshots of a run.

``exact`` is a second statement of the method in 64 bits, in plain torch on whole fields: shell sums and
ball averages as circular convolutions on a grid with zeros beyond closed axes.
"""
import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_1202_3842_gb300 import inputs, lbe

KT = 1.0 / 3.0


def _fluid(name, geometry, shape, sigma, prec, steps, eta=0.2, tau=1.0, depth=1.0, slit=(16, 64), scheme="dd_tr",
           visc=False, read="velocity"):
    c = dict(kind="fluid", geometry=geometry, nx=shape[0], ny=shape[1], nz=shape[2],
             sigma=",".join("%g" % s for s in sigma), prec=prec, steps=steps, eta=eta, tau=tau, depth=depth,
             width=slit[0], length=slit[1], scheme=scheme, visc=visc, read=read)
    return dict(c, name=name) if name else c


def _adjoint(name, shape, sigma, prec, steps, every, slit=(12, 32)):
    c = dict(kind="adjoint", geometry="channel", nx=shape[0], ny=shape[1], nz=shape[2],
             sigma=",".join("%g" % s for s in sigma), prec=prec, steps=steps, every=every, eta=0.25, tau=1.0,
             depth=1.0, width=slit[0], length=slit[1], scheme="dd_tr", visc=False, read="gradient")
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest lattice of the parity tests, looked at after every step: launches and latency
        _fluid("well24_fp64_1step", "well", (24, 24, 24), (3,), "fp64", 1),
        # a point of the spurious-current study: a comparison scheme in FP64 on a (4 xi)^3 box
        _fluid("study48_fp64_sd_tr", "well", (48, 48, 48), (4,), "fp64", 20, depth=0.3, scheme="sd_tr"),
        # the optional viscous force on the smallest well
        _fluid("well24_fp32_visc", "well", (24, 24, 24), (3,), "fp32", 20, visc=True),
        # the small bottleneck channel of the precision and divergence studies
        _fluid("channel128_fp32", "channel", (128, 32, 32), (4, 6), "fp32", 50, eta=0.25),
        # a point of the stability map (diameter and relaxation time of the production well)
        _fluid("well64_fp32", "well", (64, 64, 64), (6,), "fp32", 50, eta=0.25, tau=0.8),
        # a channel whose sides fit no tile, diameters 3 and 5 (pairs 3, 4, 5)
        _fluid("channel_ragged_fp32", "channel", (203, 77, 61), (3, 5), "fp32", 20, slit=(15, 41)),
        # a ternary mixture (pairs 2 to 6), ragged sides
        _fluid("mixture3_fp32", "well", (90, 75, 66), (2, 4, 6), "fp32", 20, depth=0.5),
        # the two-species channel in FP64, with the averaged flux
        _fluid("channel256_fp64", "channel", (256, 64, 64), (4, 6), "fp64", 10, eta=0.25, slit=(12, 32), read="flux"),
        # the production channel with 16-bit storage, the form for lattices that do not fit otherwise
        _fluid("channel512_bf16", "channel", (512, 128, 128), (4, 6), "bf16", 40, eta=0.25),
        # the production channel (the benchmark's workload)
        _fluid("channel512_fp32", "channel", (512, 128, 128), (4, 6), "fp32", 40, eta=0.25),
        # the production-size one-species well, at a depth where it runs on
        _fluid("well256_fp32", "well", (256, 256, 256), (6,), "fp32", 20, eta=0.25, tau=0.8, read="density"),
        # the adjoint channel: gradient of the averaged flux, segments recomputed from checkpoints
        _adjoint("adjoint256_fp32", (256, 64, 64), (4, 6), "fp32", 20, 10),
    ]


SIGMAS = ((0,), (2,), (3,), (4,), (5,), (6,), (7,), (8,), (4, 6), (3, 5), (2, 4), (4, 4), (6, 6), (4, 8), (2, 6),
          (2, 4, 6))


def draw(rng):
    if rng.random() < 0.12:  # a gradient
        nodes = math.exp(rng.uniform(math.log(8e3), math.log(6e5)))
        ny = max(14, round((nodes / 4) ** (1 / 3) * rng.uniform(0.8, 1.25)))
        nz = max(14, round((nodes / 4) ** (1 / 3) * rng.uniform(0.8, 1.25)))
        nx = max(32, round(nodes / (ny * nz)) // 2 * 2)
        steps = rng.randint(6, 20)
        return _adjoint(None, (nx, ny, nz), rng.choice(((4, 6), (4,), (3, 5))), "fp32", steps,
                        rng.randint(3, steps), slit=(max(6, ny // 3), nx // 4))
    geometry = rng.choice(("well", "channel"))
    sigma = rng.choice(SIGMAS)
    prec = rng.choice(("fp32", "fp32", "fp32", "fp32", "fp64", "fp64", "bf16", "fp16"))
    nodes = math.exp(rng.uniform(math.log(1e4), math.log(4e6)))
    side = nodes ** (1 / 3)
    ny, nz = (max(20, round(side * rng.uniform(0.6, 1.2))) for _ in range(2))
    nx = max(20, round(nodes / (ny * nz)))
    if prec == "fp64" or max(sigma) >= 5:
        nx += nx % 2  # the spectral form, which such cases may take, transforms rows of even length
    scheme, visc = "dd_tr", False
    if geometry == "well" and prec in ("fp32", "fp64") and len(sigma) == 1 and sigma[0] > 0:
        scheme = rng.choice(("dd_tr", "dd_tr", "sd_tr", "sd_eu"))
        if scheme == "dd_tr" and sigma[0] <= 3 and nx * ny * nz < 1e5:
            visc = rng.random() < 0.5
    # the studies' chunks of 20 to 100 steps on small lattices, fewer on large ones
    budget = (2e7 if prec == "fp64" else 8e7) / (nx * ny * nz * len(sigma))
    steps = max(2, min(rng.choice((1, 10, 20, 50)), int(budget)))
    eta = 0.0 if sigma == (0,) else round(rng.uniform(0.1, 0.2), 3)
    return _fluid(None, geometry, (nx, ny, nz), sigma, prec, steps, eta=eta, tau=1.0,
                  depth=round(rng.uniform(0.2, 0.5), 3), slit=(max(8, ny // 3), nx // 4), scheme=scheme, visc=visc,
                  read="flux" if prec == "fp64" and geometry == "channel" else rng.choice(("density", "velocity")))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _sigmas(case):
    return [float(s) for s in case["sigma"].split(",")]


def _periodic(case):
    return (1, 0, 0) if case["geometry"] == "channel" else (1, 1, 1)


def _inputs(case, seed):
    """solid [N], V [N] (the same for every species), densities [M][N], body force, wall shape and amplitude."""
    nx, ny, nz = shape = case["nx"], case["ny"], case["nz"]
    sig = _sigmas(case)
    x = np.arange(nx)[None, None, :]
    y = np.arange(ny)[None, :, None]
    z = np.arange(nz)[:, None, None]
    solid = np.zeros((nz, ny, nx), np.uint8)
    V = None
    if case["geometry"] == "channel":
        solid[[0, -1]] = 1
        solid[:, [0, -1]] = 1
        x0 = nx // 2 - case["length"] // 2
        slit = (x >= x0) & (x < x0 + case["length"]) & (np.abs(y - (ny - 1) / 2) > case["width"] / 2)
        solid |= slit.astype(np.uint8)
    else:  # a Gaussian well, minimum-image distance, radius a tenth of the shortest side
        R = 0.1 * min(shape)
        g = 1.0
        for c, n in ((x, nx), (y, ny), (z, nz)):
            d = c - n // 2
            d = d - n * np.round(d / n)
            g = g * np.exp(-(d * d) / (2 * R * R))
        V = np.ascontiguousarray(-case["depth"] * KT * g).reshape(-1)
    # equal mole fractions at the total packing; 1% noise from the seed
    n0 = 6 * case["eta"] / (math.pi * sum(s ** 3 for s in sig)) if case["eta"] > 0 else 0.05
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    rng = torch.Generator(device=dev)
    rng.manual_seed(seed)
    fluid = torch.from_numpy(1.0 - solid.reshape(-1)).to(dev)
    dens = [(n0 * (1 + 0.01 * (2 * torch.rand(nx * ny * nz, generator=rng, dtype=torch.float64, device=dev) - 1))
             * fluid).cpu().numpy() for _ in sig]
    # a body force along the channel; a gradient starts at rest and sees few steps, so it may be the paper's 1e-3
    body = 0.0 if case["geometry"] == "well" else 1e-3 if case["kind"] == "adjoint" else 1e-5
    phi = amp = None
    if case["kind"] == "adjoint":
        phi = inputs.wall_shape(shape, solid.reshape(-1), _periodic(case))
        amp = np.full(nx * ny * nz, KT)
    return solid.reshape(-1), V, dens, (body, 0.0, 0.0), phi, amp


def prepare(case, seed):
    solid, V, dens, body, phi, amp = _inputs(case, seed)
    sig = _sigmas(case)
    sim = lbe.Simulation((case["nx"], case["ny"], case["nz"]), _periodic(case), len(sig), case["prec"],
                         scheme=case["scheme"], visc=case["visc"])
    if solid.any():
        sim.set_geometry(solid)
    for a, s in enumerate(sig):
        sim.set_species(a, s, case["tau"])
        sim.set_body_force(a, body)
        if V is not None:
            sim.set_potential(a, V)
    if phi is not None:
        sim.set_wall_potential(phi, amp)
    for a in range(len(sig)):
        sim.init_density(a, dens[a])
    if case["geometry"] == "channel" and case["kind"] == "fluid":
        sim.set_flux_plane(0, case["nx"] // 2)  # every channel run accumulates its flux
    return dict(case=case, sim=sim)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
STORED = {"fp64": torch.float64, "fp32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16}


def run(state):
    case, sim = state["case"], state["sim"]

    def kept(v):
        return torch.as_tensor(v, dtype=torch.float64).to(STORED[case["prec"]])

    if case["kind"] == "adjoint":
        phi, damp, dg = sim.adjoint_flux_gradient(case["steps"], case["every"], 0, case["nx"] // 2)
        return {"phi": kept(phi), "damp": kept(damp), "dg": kept(dg)}
    sim.step(case["steps"])
    out = {"density": [kept(sim.density(a)) for a in range(sim.M)]}
    if case["read"] == "velocity":
        out["velocity"] = kept(sim.velocity(-1))
    if case["read"] == "flux":  # in 32 and 16 bits the flux of so short a run is a small rest of large terms
        out["flux"] = kept(sim.flux(-1)[1])
    return out


def work(case):
    """Bytes: the populations read and written once per step, the force field and link mask read, the fields
    handed out.  Operations: the collision and the shell sums, each shell point once per field and pair."""
    N = case["nx"] * case["ny"] * case["nz"]
    sig = _sigmas(case)
    M = len(sig)
    size = {"fp64": 8, "fp32": 4, "bf16": 2, "fp16": 2}[case["prec"]]
    real = 8 if size == 8 else 4
    nb = (76 * size + 3 * real) * M + 4
    nf = 400 * M
    for s in sig:
        for t in sig:
            nf += 2 * 2 * len(_shell((s + t) / 2)[0])
    steps = case["steps"]
    if case["kind"] == "adjoint":  # forward, recomputation and the transposed step
        return {"bytes": 3 * steps * N * nb + 8 * N, "flops": 4 * steps * N * nf}
    if case["visc"]:
        nf *= 3
    fields = M + (3 if case["read"] == "velocity" else 0)
    return {"bytes": steps * N * nb + 8 * N * fields, "flops": steps * N * nf}


# ---------------------------------------------------------------------------
# the method in 64 bits
# ---------------------------------------------------------------------------
C19 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
       (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
       (0, -1, 1)]
OPP = [0] + [p + 1 if p % 2 else p - 1 for p in range(1, 19)]
W19 = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


def _shell(s):
    """Integer vectors with s - 1/2 <= |e| < s + 1/2 and the weight 4 pi s / sum |e|."""
    if s <= 0:
        return np.zeros((0, 3), int), 0.0
    r = int(s) + 1
    e = np.stack(np.meshgrid(*[np.arange(-r, r + 1)] * 3, indexing="ij"), -1).reshape(-1, 3)
    d = np.sqrt((e * e).sum(1))
    e = e[(d >= s - 0.5) & (d < s + 0.5)]
    return e, 4 * math.pi * s / np.sqrt((e * e).sum(1)).sum()


def _ball(radius):
    r = int(radius)
    e = np.stack(np.meshgrid(*[np.arange(-r, r + 1)] * 3, indexing="ij"), -1).reshape(-1, 3)
    return e[(e * e).sum(1) <= radius * radius]


class _Method:
    def __init__(self, case, solid, V, body, phi):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.shape = (case["nz"], case["ny"], case["nx"])
        self.per = _periodic(case)[::-1]
        self.sig = _sigmas(case)
        self.M = len(self.sig)
        self.scheme, self.visc = case["scheme"], case["visc"]
        self.om = 1 / case["tau"]
        self.euler = self.scheme in ("sd_eu", "dd_eu")
        self.single = self.scheme in ("sd_tr", "sd_eu")
        self.inv = 1.0 if self.euler else 1 / (1 + 0.5 / (case["tau"] - 0.5))
        self.fluid = torch.from_numpy(solid == 0).reshape(self.shape).to(self.dev)
        self.fl = self.fluid.to(torch.float64)
        self.V = self._field(V)
        self.body = body
        self.phi = self._field(phi)
        # blocked links: the population arriving along c_p comes from a solid node or from outside
        ok = self._pad(self.fl, 1)
        self.blocked = [self._crop(torch.roll(ok, (c[2], c[1], c[0]), (0, 1, 2))) < 0.5 for c in C19]
        # convolution kernels on a grid with room for the widest reach along closed axes
        reach = max([int(max(self.sig))] + [1])
        self.L = [n if p else n + reach for n, p in zip(self.shape, self.per)]
        self.pairs = [(a, b, (self.sig[a] + self.sig[b]) / 2) for a in range(self.M) for b in range(self.M)
                      if self.sig[a] + self.sig[b] > 0]
        self.kernel = {}
        for s in {s for _, _, s in self.pairs}:
            e, w = _shell(s)
            unit = e / np.sqrt((e * e).sum(1, keepdims=True))
            self.kernel[s] = (torch.stack([self._spectrum(e, unit[:, c]) for c in range(3)]), s * s * w, e, unit)
        self.ball = []
        for s in self.sig:
            e = _ball(s / 2)
            self.ball.append(self._spectrum(e, np.full(len(e), 1 / len(e))))

    def _field(self, v):
        if v is None:
            return torch.zeros(self.shape, dtype=torch.float64, device=self.dev)
        return torch.from_numpy(np.asarray(v, dtype=np.float64)).reshape(self.shape).to(self.dev)

    def _pad(self, v, r):
        out = v
        for ax in range(3):
            if not self.per[ax]:
                s = list(out.shape)
                s[ax] = 2 * r
                out = torch.cat([out, out.new_zeros(s)], ax)
        return out

    def _crop(self, v):
        nz, ny, nx = self.shape
        return v[..., :nz, :ny, :nx]

    def _spectrum(self, e, w):
        """Spectrum of the kernel of sum_e w_e v(r + e)."""
        k = torch.zeros(self.L, dtype=torch.float64, device=self.dev)
        idx = tuple(torch.as_tensor(-e[:, 2 - ax] % self.L[ax]).to(self.dev) for ax in range(3))
        k.index_put_(idx, torch.as_tensor(np.asarray(w, dtype=np.float64)).to(self.dev), accumulate=True)
        return torch.fft.rfftn(k)

    def _fft(self, v):
        return torch.fft.rfftn(v, s=self.L, dim=(-3, -2, -1))

    def _ifft(self, v):
        return self._crop(torch.fft.irfftn(v, s=self.L, dim=(-3, -2, -1)))

    def force(self, amp, shift):
        """F = -grad V + g, a neighbour outside a closed axis standing for the node itself."""
        V = self.V if amp is None else self.V + amp * self.phi
        inside = self._pad(torch.ones_like(V), 1)
        Vp = self._pad(V, 1)
        g = [0.0, 0.0, 0.0]
        for c, w in zip(C19[1:], W19[1:]):
            back = (-c[2], -c[1], -c[0])
            nb = self._crop(torch.roll(Vp, back, (0, 1, 2)))
            nb = torch.where(self._crop(torch.roll(inside, back, (0, 1, 2))) > 0.5, nb, V)
            for k in range(3):
                if c[k]:
                    g[k] = g[k] + 3 * w * c[k] * nb
        return torch.stack([self.body[k] + (0 if shift is None else shift[k]) - g[k] for k in range(3)])

    def collide_forces(self, n, ut):
        """C^mf of every species, and C^visc when it is on (else None)."""
        if not self.pairs:
            return torch.zeros((self.M, 3) + self.shape, dtype=torch.float64, device=self.dev), None
        nh = [self._fft(v) for v in n]
        xi2 = xi3 = 0.0
        for b, s in enumerate(self.sig):
            nbar = self._ifft(nh[b] * self.ball[b])
            xi2 = xi2 + math.pi / 6 * s ** 2 * nbar
            xi3 = xi3 + math.pi / 6 * s ** 3 * nbar
        i1 = 1 / (1 - xi3)
        C, Cv = [0.0] * self.M, [0.0] * self.M
        for a, b, s in self.pairs:
            kern, s2w, e, unit = self.kernel[s]
            t = self.sig[a] * self.sig[b] / (self.sig[a] + self.sig[b])
            g = i1 + 3 * t * xi2 * i1 ** 2 + 2 * t * t * xi2 ** 2 * i1 ** 3
            P = self._ifft(nh[b] * kern)
            Qs = self._ifft(self._fft(g * n[b]) * kern)
            C[a] = C[a] - KT * s2w * 0.5 * n[a] * (g * P + Qs)
            if self.visc:  # periodic wells: the shell point by point
                pre = 2 * s2w * math.sqrt(KT / math.pi)
                total = torch.zeros((3,) + self.shape, dtype=torch.float64, device=self.dev)
                for ee, u in zip(e.tolist(), unit.tolist()):
                    at = (-ee[2], -ee[1], -ee[0])
                    du = torch.roll(ut[b], at, (1, 2, 3)) - ut[b]
                    v = (0.5 * (g + torch.roll(g, at, (0, 1, 2))) * torch.roll(n[b], at, (0, 1, 2))
                         * (u[0] * du[0] + u[1] * du[1] + u[2] * du[2]))
                    total += torch.stack([u[0] * v, u[1] * v, u[2] * v])
                Cv[a] = Cv[a] + pre * n[a] * total
        return torch.stack(C), torch.stack(Cv) if self.visc else None

    def moments(self, f, g, F):
        n = f.sum(1) * self.fl
        src = f if self.single else g
        Jt = torch.stack([sum(c[k] * src[:, p] for p, c in enumerate(C19) if c[k]) for k in range(3)], 1)
        safe = torch.where(n > 0, n, torch.ones_like(n))
        ut = torch.where((n > 0)[:, None], Jt / safe[:, None], torch.zeros_like(Jt)) if self.visc else None
        C, Cv = self.collide_forces(n, ut)
        nF = n[:, None] * F
        if Cv is not None:
            nF = nF + Cv
        J = Jt if self.euler else Jt + 0.5 * (C + nF)
        J = J * self.fl
        ua = torch.where((n > 0)[:, None], J / safe[:, None], torch.zeros_like(J))
        if self.single:
            Pi = n
        else:
            Pi = g.sum(1) if self.euler else g.sum(1) - 0.5 * (C * ua).sum(1)
        tot = n.sum(0)
        u = torch.where(tot > 0, J.sum(0) / torch.where(tot > 0, tot, torch.ones_like(tot)), torch.zeros_like(J[0]))
        return n, J, ua, Pi, u, C, nF

    def step(self, f, g, F, plane):
        """Streamed populations [M][19] of one step to the next, and the flux through x = plane."""
        n, J, ua, Pi, u, C, nF = self.moments(f, g, F)
        flux = J[:, 0, :, :, plane].sum()

        def dot(c, v, ax):
            out = 0.0
            for k in range(3):
                if c[k]:
                    out = out + c[k] * v.select(ax, k)
            return out

        X = C + nF
        uau = (ua * u).sum(1)
        iso = 1.5 * n * (2 * uau - (u * u).sum(0))
        s0 = -3 * (X * ua).sum(1)
        post = [[], []]
        for p, c in enumerate(C19):
            if p == 0:
                t1, Sf, Sg = 0.0, s0, s0
            else:
                cua, cu = dot(c, ua, 1), dot(c, u, 0)
                t1 = 3 * n * cua + 4.5 * n * (2 * cua * cu - cu * cu)
                cX, cY, cC = dot(c, X, 1), dot(c, nF, 1), dot(c, C, 1)
                Sf = s0 + 3 * cX + 9 * cX * cua
                Sg = s0 + 3 * cY + 18 * cC * cua + 9 * cY * cua
            fp = f[:, p] + self.om * (W19[p] * (n - iso + t1) - f[:, p]) + self.inv * W19[p] * Sf
            gp = fp if self.single else (g[:, p] + self.om * (W19[p] * (Pi - iso + t1) - g[:, p])
                                         + self.inv * W19[p] * Sg)
            post[0].append(fp * self.fl)
            post[1].append(gp * self.fl)
        out = []
        for q in (post[:1] if self.single else post):
            moved = []
            for p, c in enumerate(C19):
                v = torch.roll(q[p], (c[2], c[1], c[0]), (1, 2, 3))
                moved.append(torch.where(self.blocked[p], q[OPP[p]], v) * self.fl)
            out.append(torch.stack(moved, 1))
        return out[0], out[-1], flux


def _start(m, dens):
    n = torch.stack([m._field(v) for v in dens]) * m.fl
    f = torch.stack([w * n for w in W19], 1)
    return f, f.clone()


def exact(case, seed):
    solid, V, dens, body, phi, amp = _inputs(case, seed)
    m = _Method(case, solid, V, body, phi)
    f, g = _start(m, dens)
    plane = case["nx"] // 2
    if case["kind"] == "adjoint":
        a = m._field(amp).requires_grad_()
        shift = torch.zeros(3, dtype=torch.float64, device=m.dev, requires_grad=True)
        F = m.force(a, shift)
        total = 0.0
        for _ in range(case["steps"]):
            f, g, flux = torch.utils.checkpoint.checkpoint(lambda x, y, F: m.step(x, y, F, plane), f, g, F,
                                                           use_reentrant=False)
            total = total + flux
        phi_avg = total / case["steps"]
        phi_avg.backward()
        return {"phi": phi_avg.detach().cpu(), "damp": a.grad.reshape(-1).cpu(), "dg": shift.grad.cpu()}
    with torch.no_grad():
        F = m.force(None, None)
        total = 0.0
        for _ in range(case["steps"]):
            f, g, flux = m.step(f, g, F, plane)
            total = total + flux
        n, J, _, _, u, _, _ = m.moments(f, g, F)
        out = {"density": [v.reshape(-1).cpu() for v in n]}
        if case["read"] == "velocity":
            out["velocity"] = u.reshape(3, -1).cpu()
        if case["read"] == "flux":
            out["flux"] = (total / case["steps"]).cpu()
    return out

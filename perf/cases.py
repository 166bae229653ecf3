"""What the performance of this framework is measured on: simulation passes through its public entry points.

A pass of most cases is what a driver program does between two outputs of a run: put a state on the
grid (a snapshot with `Grid.upload`, or primitives with `Grid.init_equilibrium`), advance it some
steps (`Grid.step`) and take the state out (`Grid.download`).  The gradient case is one evaluation
of the boundary-outflow objective with its gradient through `autograd.boundary_outflow`.

`exact` restates the method in plain torch at 64 bits (whole-array operations, no code of the
package): the equations are those of include/fx.h and of the paper it cites.
"""
import math

import numpy as np
import torch

DEV = "cuda"
F64 = torch.float64


# ---------------------------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------------------------
def listed():
    return [
        # a 1-d shock tube in full precision: the smallest grid anybody runs, latency is all
        dict(name="tube", kind="tube", nx=512, groups=12, precision="fp64", steps=20),
        # a small 2-d box, as in parameter studies: a few blocks per kernel
        dict(name="shear_small", kind="shear", nx=96, ny=80, groups=8, precision="fp32n64", steps=10),
        # the production shear layer in the form of the benchmark: FP32 with the FP64 Newton
        dict(name="shear", kind="shear", nx=1024, ny=1024, groups=16, precision="fp32n64", steps=2),
        # the same physics in plain FP64
        dict(name="shear_fp64", kind="shear", nx=512, ny=512, groups=16, precision="fp64", steps=1),
        # with the velocity-dependent radiation terms
        dict(name="shear_vterms", kind="shear", nx=768, ny=768, groups=16, precision="fp32n64", steps=2, vterms=1),
        # an odd grid, an odd group count, open boundaries, a beam of radiation through dense blobs
        dict(name="blobs_odd", kind="blobs", nx=515, ny=389, groups=7, precision="fp32", steps=4),
        # the largest: a 3-d cloud
        dict(name="cloud", kind="cloud", nx=256, ny=256, nz=256, groups=12, precision="fp32n64", steps=1),
        # a ragged 3-d box with more groups
        dict(name="cloud_odd", kind="cloud", nx=75, ny=61, nz=50, groups=20, precision="fp32", steps=2),
        # a star on the spherical (r, theta) grid: long runs of steps on a mid-sized grid
        dict(name="atmosphere", kind="atmosphere", nx=640, ny=128, groups=20, precision="fp32", steps=10),
        # three neutrino species and the composition
        dict(name="neutrinos", kind="neutrinos", nx=512, ny=512, groups=8, precision="fp32n64", steps=2),
        # a strong shock against a wall, from the primitives on: boundary layers, carbuncle guard
        dict(name="mach", kind="mach", nx=520, ny=160, groups=1, precision="fp32", steps=10),
        # one objective and gradient evaluation of an optimisation over the initial density
        dict(name="gradient", kind="gradient", nx=128, ny=96, groups=8, precision="fp64", steps=4, every=2),
    ]


def _size(rng, lo, hi):
    """A size between lo and hi, uniform in its logarithm."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["tube", "shear", "shear", "blobs", "cloud", "cloud", "atmosphere", "neutrinos", "mach", "gradient"])
    form = rng.choice(["fp32n64", "fp32n64", "fp32", "fp64"])
    big = 1.0 if form != "fp64" else 0.25  # (FP64 runs are made on smaller grids)
    c = dict(kind=kind, precision=form, groups=rng.randint(3, 24), steps=rng.randint(1, 4))
    if kind == "tube":
        c.update(nx=_size(rng, 100, 4000), steps=rng.randint(5, 20))
    elif kind == "shear":
        c.update(nx=_size(rng, 40, int(1000 * big)), ny=_size(rng, 40, int(1000 * big)), vterms=rng.choice([0, 0, 1]))
    elif kind == "blobs":
        c.update(nx=_size(rng, 40, int(800 * big)), ny=_size(rng, 40, int(800 * big)))
    elif kind == "cloud":
        m = 150 if form != "fp64" else 50
        c.update(nx=_size(rng, 20, m), ny=_size(rng, 20, m), nz=_size(rng, 20, m), steps=rng.randint(1, 2))
    elif kind == "atmosphere":
        c.update(nx=_size(rng, 80, int(800 * big)), ny=_size(rng, 24, 160), steps=rng.randint(1, 6))
    elif kind == "neutrinos":
        c.update(nx=_size(rng, 32, int(500 * big)), ny=_size(rng, 32, int(500 * big)), groups=rng.randint(3, 10))
    elif kind == "mach":
        ny = _size(rng, 40, 200)
        c.update(nx=int(3.25 * ny), ny=ny, groups=rng.randint(1, 2), steps=rng.randint(4, 10))
    else:
        c.update(nx=_size(rng, 32, 140), ny=_size(rng, 24, 110), groups=rng.randint(3, 10), precision="fp64",
                 steps=rng.randint(2, 4), every=rng.randint(1, 2))
    return c


# ---------------------------------------------------------------------------------------------
# Inputs: parameters, primitive fields, and the conserved snapshot they give
# ---------------------------------------------------------------------------------------------
def _pick(where, a, b):
    """a or b, as 64-bit values."""
    return torch.where(where, torch.tensor(a, device=where.device, dtype=F64), torch.tensor(b, device=where.device, dtype=F64))


def _field(gen, shape, slope):
    """Periodic Gaussian random field with power spectrum k^slope, zero mean and unit deviation."""
    white = torch.randn(shape, generator=gen, device=DEV, dtype=F64)
    k2 = 0.0
    for d, m in enumerate(shape):
        k = torch.fft.fftfreq(m, device=DEV, dtype=F64) * m
        k2 = k2 + (k ** 2).reshape([-1 if e == d else 1 for e in range(len(shape))])
    amp = torch.where(k2 > 0, k2.clamp_min(1.0) ** (slope / 4.0), torch.zeros_like(k2))
    f = torch.fft.ifftn(torch.fft.fftn(white) * amp).real
    f = f - f.mean()
    return f / f.std()


def _setup(case, seed):
    """Parameters (the fields of workloads.Problem), primitives [rho, p, v.., T_rad (, Y_e)] and boundary layers."""
    kind, G = case["kind"], case["groups"]
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    n = [case["nx"], case.get("ny", 1), case.get("nz", 1)]
    D = 1 if kind == "tube" else 3 if kind == "cloud" else 2
    q = dict(name=kind, dims=D, n=tuple(n), x_lo=(0.0,) * 3, x_hi=(1.0,) * 3, bc_lo=("periodic",) * 3,
             bc_hi=("periodic",) * 3, ngroups=G, gamma=5.0 / 3.0, kappa0=1.0, kap_rho_exp=1.0, kap_T_exp=-1.5,
             kap_eps_exp=-2.0, precision=case["precision"], vterms=case.get("vterms", 0))
    shape = tuple(reversed(n[:D]))

    def centre(d):
        x = q["x_lo"][d] + (torch.arange(n[d], device=DEV, dtype=F64) + 0.5) * (q["x_hi"][d] - q["x_lo"][d]) / n[d]
        return x.reshape([-1 if e == D - 1 - d else 1 for e in range(D)]).expand(shape)

    def rand(*s):
        return torch.rand(s or shape, generator=gen, device=DEV, dtype=F64) * 2.0 - 1.0

    layers, v, trad, ye = [], [torch.zeros(shape, device=DEV, dtype=F64) for _ in range(D)], None, None
    if kind == "tube":  # Sod's states
        q.update(bc_lo=("outflow",) * 3, bc_hi=("outflow",) * 3)
        left = centre(0) < 0.5
        rho = _pick(left, 1.0, 0.125) * (1.0 + 1e-3 * rand())
        p = _pick(left, 1.0, 0.1)
    elif kind == "shear":  # a periodic Kelvin-Helmholtz layer
        q.update(gamma=1.4, kappa0=10.0)
        band = (centre(1) >= 0.25) & (centre(1) < 0.75)
        rho = _pick(band, 2.0, 1.0)
        v = [_pick(band, 0.5, -0.5), 0.01 * rand()]
        p = torch.full(shape, 2.5, device=DEV, dtype=F64)
    elif kind in ("blobs", "gradient"):  # dense blobs in a uniform medium, radiation leaving through +x
        q.update(bc_lo=("outflow", "periodic", "periodic"), bc_hi=("outflow", "periodic", "periodic"), kap_rho_exp=3.0)
        rho = torch.ones(shape, device=DEV, dtype=F64)
        for bx, by in torch.rand(16, 2, generator=gen, device=DEV, dtype=F64).tolist():
            bx = 0.9 + 0.1 * bx if kind == "gradient" else bx
            rho = rho + 9.0 * torch.exp(-((centre(0) - bx) ** 2 + (centre(1) - by) ** 2) / (2.0 * 0.03 ** 2))
        p = torch.ones_like(rho)
        if kind == "gradient":  # (a generic state: no two cells alike)
            rho, p, v = rho * (1.0 + 0.1 * rand()), p * (1.0 + 0.1 * rand()), [0.1 * rand(), 0.1 * rand()]
    elif kind == "cloud":  # a lognormal density, radiation at twice the gas temperature
        q.update(kap_T_exp=-3.5, kap_eps_exp=-3.0)
        rho = torch.exp(_field(gen, shape, -11.0 / 3.0) - 0.5)
        p = torch.ones_like(rho)
        trad = 2.0 * p / rho
    elif kind == "atmosphere":  # log-r grid over r in [1, 1000], thick core, streaming outer edge
        q.update(x_hi=(math.log(1000.0), math.pi, 1.0), bc_lo=("reflect", "axis", "periodic"),
                 bc_hi=("outflow", "axis", "periodic"), kappa0=1e3, kap_rho_exp=2.0, geom="sph", map1="exp")
        r = torch.exp(centre(0))
        rho = r ** -2.0 * (1.0 + 1e-3 * rand(n[1], 1))
        p = r ** -2.5
    elif kind == "neutrinos":  # three species in a periodic box
        q.update(gamma=4.0 / 3.0, kappa0=3.0, species=3, xi0=0.05)
        rho = torch.exp(0.5 * _field(gen, shape, -3.0))
        p = torch.ones_like(rho)
        s, t = torch.sin(2 * math.pi * centre(0)), torch.sin(2 * math.pi * centre(1))
        v[0], trad, ye = 0.3 * t, 1.5 * p / rho, 0.3 + 0.1 * s * t
    elif kind == "mach":  # double Mach reflection: a Mach-10 shock at 60 degrees to a wall
        nx, ny = n[0], n[1]
        dx, alpha = 1.0 / ny, math.pi / 3.0
        n[0], n[1] = nx + 2, ny + 4
        shape = (n[1], n[0])
        q.update(n=tuple(n), x_lo=(-2 * dx, -2 * dx, 0.0), x_hi=(nx * dx, 1.0 + 2 * dx, 1.0), bc_lo=("outflow",) * 3,
                 bc_hi=("outflow",) * 3, gamma=1.4, kappa0=0.0, kap_rho_exp=0.0, kap_T_exp=0.0, kap_eps_exp=0.0,
                 c_light=20.0, couple=0, shock_guard=0.5)
        pre, post = (1.4, 1.0, 0.0, 0.0), (8.0, 116.5, 8.25 * math.sin(alpha), -8.25 * math.cos(alpha))
        x0, cot, speed = 1.0 / 6.0, 1.0 / math.tan(alpha), 10.0 / math.sin(alpha)
        behind = centre(0) - x0 - centre(1) * cot <= 0.0
        rho, p, v0, v1 = (_pick(behind, post[m], pre[m]) for m in range(4))
        rho, v = rho * (1.0 + 1e-3 * rand()), [v0, v1]
        trad = torch.full(shape, 0.01, device=DEV, dtype=F64)
        first = int(torch.searchsorted(centre(0)[0].contiguous(), torch.tensor(x0, device=DEV, dtype=F64), right=True))
        A, B = post + (0.01,), pre + (0.01,)
        fixed = dict(kind="front", x0=1e30, y0=0.0, cot_alpha=0.0, speed=0.0, A=A, B=A)
        layers = [dict(fixed, lo=(0, 0, 0), hi=(2, n[1], 1)), dict(fixed, lo=(2, 0, 0), hi=(first, 2, 1)),
                  dict(kind="mirror", d=1, m=2, lo=(first, 0, 0), hi=(n[0], 2, 1)),
                  dict(kind="front", lo=(2, n[1] - 2, 0), hi=(n[0], n[1], 1), x0=x0, y0=0.0, cot_alpha=cot,
                       speed=speed, A=A, B=B)]
    trad = p / rho if trad is None else trad
    # the speed of light and the step: c = 10 max(|v| + a), light-crossing limit, CFL 1/2
    a = torch.sqrt(q["gamma"] * p / rho)
    if "c_light" not in q:
        q["c_light"] = float(10.0 * (torch.sqrt(sum(w * w for w in v)) + a).max())
    inv = 0.0
    for d in range(D):
        h = torch.exp(centre(0) - 0.5 * (q["x_hi"][0] - q["x_lo"][0]) / n[0]) if kind == "atmosphere" else 1.0
        inv = inv + torch.clamp_min(v[d].abs() + a, q["c_light"]) * n[d] / ((q["x_hi"][d] - q["x_lo"][d]) * h)
    q["dt"] = float(0.5 / inv.max())
    prim = torch.stack([rho, p, *v, trad] + ([ye] if ye is not None else []))
    return q, prim, layers


def _snapshot(case, seed, q, prim):
    """A conserved state: equilibrium radiation at T_rad carrying a flux of up to a fifth of c E (a beam for the blobs)."""
    M = _Method(q)
    gas, rad, comp = M.equilibrium(prim)
    c, D = q["c_light"], M.D
    kind = case["kind"]
    for d in range(D):
        if kind in ("blobs", "gradient"):
            f = 0.5 if d == 0 else 0.05
        elif kind == "atmosphere":
            f = 0.0  # (the flux builds up from the gradient)
        else:
            ph = (seed % 997) * 0.1 + d
            x = (torch.arange(M.n[d], device=DEV, dtype=F64) + 0.5) / M.n[d]
            f = 0.2 * torch.sin(2 * math.pi * x + ph).reshape([-1 if e == D - 1 - d else 1 for e in range(D)] + [1])
        rad[1 + d] = f * c * rad[0]
    if kind == "gradient":
        gen = torch.Generator(device=DEV)
        gen.manual_seed(seed + 1)
        rad[0] *= 1.0 + 0.1 * torch.rand(rad[0].shape, generator=gen, device=DEV, dtype=F64)
        for d in range(D):
            rad[1 + d] *= 1.0 + 0.1 * torch.rand(rad[0].shape, generator=gen, device=DEV, dtype=F64)
    flat = torch.cat([gas.reshape(-1), rad.reshape(-1)] + ([comp.reshape(-1)] if comp is not None else []))
    return flat if q["precision"] == "fp64" else flat.float()


def _split(q, flat):
    """The state's gas, energy, flux and composition blocks (views)."""
    D, N, K = q["dims"], math.prod(q["n"][:q["dims"]]), q["ngroups"] * q.get("species", 1)
    g, r = (2 + D) * N, (1 + D) * N * K
    out = {"gas": flat[:g].view(2 + D, N), "E": flat[g:g + N * K].view(N, K), "F": flat[g + N * K:g + r].view(D, N, K)}
    if q.get("species", 1) > 1:
        out["rho_ye"] = flat[g + r:].view(N)
    return out


class _State:
    pass


def prepare(case, seed):
    from paper_1806_07390_gb300 import fx
    from paper_1806_07390_gb300.workloads import Problem

    s = _State()
    s.case = case
    q, prim, s.layers = _setup(case, seed)
    s.q = q
    s.grid = fx.Grid(Problem(**q))
    s.prim = prim.reshape(prim.shape[0], -1).contiguous() if case["kind"] == "mach" else None
    s.flat = None if case["kind"] == "mach" else _snapshot(case, seed, q, prim)
    s.out = torch.empty(s.grid.nelem, device=DEV, dtype=F64 if q["precision"] == "fp64" else torch.float32)
    if case["kind"] == "gradient":
        s.rho = s.flat[:math.prod(q["n"][:2])].clone()
        s.kappa = torch.tensor(q["kappa0"], dtype=F64, device=DEV)
    return s


def run(s):
    case, q, g = s.case, s.q, s.grid
    if case["kind"] == "gradient":
        from paper_1806_07390_gb300 import autograd

        rho, kappa = s.rho.detach().requires_grad_(), s.kappa.detach().requires_grad_()
        J = autograd.boundary_outflow(g, s.flat, rho, kappa, q["dt"], case["steps"], case["every"])
        J.backward()
        return {"J": J.detach(), "rho": rho.grad, "kappa": kappa.grad}
    if s.prim is not None:
        g.init_equilibrium(s.prim)
        g.boundary_layers(s.layers, 0.0)
    else:
        g.upload(s.flat)
    g.step(q["dt"], case["steps"])
    g.download(s.out)
    return _split(q, s.out)


def work(case):
    """Bytes: the method needs the whole state of a stage before the next one, so each of the two stages of a step
    reads its input and writes its result, and the second reads the step's start too.  Flops: the arithmetic of
    the reconstructions, closures, fluxes and updates per cell and group, and of the interaction."""
    kind, D = case["kind"], 1 if case["kind"] == "tube" else 3 if case["kind"] == "cloud" else 2
    N = case["nx"] * case.get("ny", 1) * case.get("nz", 1)
    K = case["groups"] * (3 if kind == "neutrinos" else 1)
    b = 8 if case["precision"] == "fp64" else 4
    state = N * (2 + D + K * (1 + D)) * b
    stage = D * ((1 + D) * 10 + 2 * (14 + 3 * D) + 12 + 5 * D) + (1 + D) * (4 * D + 4)  # per cell and group
    stage += 0 if kind == "mach" else 90  # the interaction: two evaluations of the group energies
    stage += (30 + 14 * D * D * (1 + D)) if case.get("vterms") else 0
    if kind == "gradient":  # the steps, their recomputation, and the adjoint at about twice a forward step
        return {"bytes": case["steps"] * 4 * 5 * state, "flops": case["steps"] * 4 * 2 * N * K * stage}
    return {"bytes": case["steps"] * 5 * state, "flops": case["steps"] * 2 * N * K * stage}


# ---------------------------------------------------------------------------------------------
# The method at 64 bits, whole arrays at a time
# ---------------------------------------------------------------------------------------------
_BERN = [1.0 / 6, -1.0 / 30, 1.0 / 42, -1.0 / 30, 5.0 / 66, -691.0 / 2730, 7.0 / 6, -3617.0 / 510]


def _bernoulli(terms):
    """B_2m / (2m)! from the even zeta values."""
    return [2.0 * (-1.0) ** (m + 1) * math.fsum(k ** (-2.0 * m) for k in range(1, 200 if m > 4 else 2)) / (2.0 * math.pi) ** (2 * m)
            if m > 4 else _BERN[m - 1] / math.factorial(2 * m) for m in range(1, terms + 1)]


_SPLIT = 3.0
_B2M = _bernoulli(26)
_TOTAL = math.pi ** 4 / 15.0


def _planck_edge(x):
    """(Q, w) at x = eps/T: Q = Int_0^x below the split and Int_x^inf above it of t^3/(e^t - 1), w = x^4/(e^x - 1)."""
    low = x < _SPLIT
    y = torch.where(low, x, torch.ones_like(x))
    y2 = y * y
    sd, sw = torch.zeros_like(y), torch.zeros_like(y)
    for m in range(26, 0, -1):
        sd = sd * y2 + _B2M[m - 1] / (2 * m + 3)
        sw = sw * y2 + _B2M[m - 1]
    ql = y ** 3 * (1.0 / 3.0 - y / 8.0 + y2 * sd)
    wl = y ** 3 * (1.0 - y / 2.0 + y2 * sw)
    z = torch.where(low, torch.full_like(x, _SPLIT), x)
    e = torch.exp(-z)
    en, qh = e.clone(), torch.zeros_like(z)
    for k in range(1, 16):
        qh = qh + en * (z ** 3 / k + 3.0 * z ** 2 / k ** 2 + 6.0 * z / k ** 3 + 6.0 / k ** 4)
        en = en * e
    return torch.where(low, ql, qh), torch.where(low, wl, z ** 4 * e / (1.0 - e)), low


class _Axis:
    """Cells -2 .. n+1 of one direction: centres, volume moments, and the reconstruction weights of cells -1 .. n."""

    def __init__(self, q, d):
        self.n, lo, hi = q["n"][d], q["x_lo"][d], q["x_hi"][d]
        self.dx = (hi - lo) / self.n
        self.bc = (q["bc_lo"][d], q["bc_hi"][d])
        i = np.arange(-2, self.n + 2)
        self.xl = lo + i * self.dx
        self.xc = self.xl + 0.5 * self.dx
        sph = q.get("geom", "cart") == "sph"
        self.weight = (lambda x: np.exp(3.0 * x)) if sph and d == 0 else (lambda x: np.abs(np.sin(x))) if sph else np.ones_like
        self.vol = self.mean(lambda x: np.ones_like(x), False)
        c = self.xc[:, None]
        self.m1, self.m2 = self.mean(lambda x: x - c), self.mean(lambda x: (x - c) ** 2)
        self.cen = self.xc + self.m1
        # per cell -1 .. n: centroid gaps and the parabola's systems, in coordinates about the cell centre
        k = np.arange(1, self.n + 3)
        M1 = np.stack([self.xc[k + o] - self.xc[k] + self.m1[k + o] for o in (-1, 0, 1)])
        M2 = np.stack([(self.xc[k + o] - self.xc[k]) ** 2 + 2 * (self.xc[k + o] - self.xc[k]) * self.m1[k + o] + self.m2[k + o] for o in (-1, 0, 1)])
        xl, xr = -0.5 * self.dx, 0.5 * self.dx
        one = np.ones_like(M1[0])
        inv1 = np.linalg.inv(np.stack([np.stack([one, M1[o], M2[o]], -1) for o in range(3)], -2))
        inv2 = np.linalg.inv(np.stack([np.stack([one, xl * one, xl * xl * one], -1), np.stack([one, M1[1], M2[1]], -1),
                                       np.stack([one, xr * one, xr * xr * one], -1)], -2))
        row = lambda x: np.array([1.0, x, x * x])  # noqa: E731
        der = lambda x: np.array([0.0, 1.0, 2.0 * x])  # noqa: E731
        self.wa, self.wb = np.einsum("j,kjo->ok", row(xl), inv1), np.einsum("j,kjo->ok", row(xr), inv1)
        self.al, self.ar = np.einsum("j,kjo->ok", der(xl), inv2), np.einsum("j,kjo->ok", der(xr), inv2)
        self.sl, self.sr = (xl - M1[0]) / (M1[1] - M1[0]), (xr - M1[1]) / (M1[2] - M1[1])
        self.rl = self.dx ** 2 / (M2[1] - 2 * xl * M1[1] + xl * xl)
        self.rr = self.dx ** 2 / (M2[1] - 2 * xr * M1[1] + xr * xr)
        self.gl, self.gr, self.gc = M1[1] - M1[0], M1[2] - M1[1], M1[2] - M1[0]
        self.dl, self.dr = xl - M1[1], xr - M1[1]

    def mean(self, f, over=True):
        """Volume mean (or integral) of f over each cell, ghosts mirrored in the weight."""
        x, w = np.polynomial.legendre.leggauss(20)
        t = self.xl[:, None] + 0.5 * self.dx * (x[None, :] + 1.0)
        v = (0.5 * self.dx * w * self.weight(t) * f(t)).sum(1)
        return v / self.vol if over else v


class _Method:
    def __init__(self, q):
        self.q, self.D, self.n = q, q["dims"], q["n"]
        self.G, self.S = q["ngroups"], q.get("species", 1)
        self.K = self.G * self.S
        self.c, self.gam = q["c_light"], q["gamma"]
        self.sph = q.get("geom", "cart") == "sph"
        self.ax = [_Axis(q, d) for d in range(self.D)]
        self.edge = np.array([0.01 * 1000.0 ** (k / self.G) for k in range(self.G + 1)])
        self.eps = np.sqrt(self.edge[1:] * self.edge[:-1])
        self.efac = self.t(np.tile(self.eps ** q["kap_eps_exp"], self.S))
        if self.S > 1:
            self.xi = self.t(np.concatenate([-q["xi0"] / self.eps, q["xi0"] / self.eps, 0 * self.eps]))
            self.dw = self.t(np.repeat([2.0, -2.0, 0.0], self.G))
            self.w0 = self.t(np.repeat([0.0, 2.0, 1.0], self.G))
        self.kappa0 = q["kappa0"]
        if self.sph:
            R, T = self.ax
            r, V = np.exp, R.vol
            self.h = [np.sqrt(R.mean(lambda x: r(2 * x)))] * 2  # dr/dx1 = r: both scale factors are sqrt<r^2>
            self.ra, self.rb, self.rc = (np.array([(np.exp(m * (x + R.dx)) - np.exp(m * x)) / m for x in R.xl]) for m in (2.0, 3.0, 3.0))
            self.g221, self.g122 = np.ones_like(V), -np.ones_like(V)
            self.g111 = (r(3 * (R.xl + R.dx)) - r(3 * R.xl)) / V - 2.0
            self.g332 = T.mean(lambda x: np.cos(x) / np.sin(x))
            self.g222 = (np.abs(np.sin(T.xl + T.dx)) - np.abs(np.sin(T.xl))) / T.vol - self.g332

    @staticmethod
    def t(a):
        return torch.as_tensor(np.ascontiguousarray(a), device=DEV, dtype=F64)

    def along(self, a, d, extra=0):
        """An array over direction d, shaped to broadcast over the cells (and the groups)."""
        return self.t(a).reshape([-1 if e == self.D - 1 - d else 1 for e in range(self.D)] + [1] * extra)

    def pad(self, f, d, sign=1.0):
        ax = self.D - 1 - d
        lo, hi = self.ax[d].bc
        n = f.shape[ax]
        a = f.narrow(ax, n - 2, 2) if lo == "periodic" else torch.cat([f.narrow(ax, 0, 1)] * 2, ax) if lo == "outflow" \
            else f.narrow(ax, 0, 2).flip(ax) * sign
        b = f.narrow(ax, 0, 2) if hi == "periodic" else torch.cat([f.narrow(ax, n - 1, 1)] * 2, ax) if hi == "outflow" \
            else f.narrow(ax, n - 2, 2).flip(ax) * sign
        return torch.cat([a, f, b], ax)

    def cut(self, f, d, lo, hi):
        """Entries lo .. len-hi along direction d."""
        ax = self.D - 1 - d
        return f.narrow(ax, lo, f.shape[ax] - lo - hi)

    # -- state
    def equilibrium(self, prim):
        D = self.D
        rho, p, v, T = prim[0], prim[1], prim[2:2 + D], prim[2 + D]
        h = [1.0] * D
        if self.sph:
            h = [self.along(self.h[d][2:-2], 0) for d in range(2)]
        gas = torch.stack([rho, *[rho * v[d] * h[d] for d in range(D)], p / (self.gam - 1.0) + 0.5 * rho * (v ** 2).sum(0)])
        B = self.planck(T)[0].repeat([1] * D + [self.S])
        if self.S > 1:
            B = B * (self.w0 + self.dw * prim[3 + D].unsqueeze(-1))
        rad = torch.stack([B] + [torch.zeros_like(B)] * D)
        return gas, rad, rho * prim[3 + D] if self.S > 1 else None

    def planck(self, T):
        """B_g(T) and dB_g/dT, groups last."""
        x = self.t(self.edge) / T.unsqueeze(-1)
        Q, w, low = _planck_edge(x)
        ql, qh, ll, lh = Q[..., :-1], Q[..., 1:], low[..., :-1], low[..., 1:]
        band = torch.where(ll & lh, qh - ql, torch.where(ll, _TOTAL - ql - qh, ql - qh))
        a = 0.1 / _TOTAL  # a_R 15 / pi^4
        T3 = (T ** 3).unsqueeze(-1)
        return a * T3 * T.unsqueeze(-1) * band, a * T3 * (4.0 * band + w[..., :-1] - w[..., 1:])

    def kappa(self, rho, T):
        q = self.q
        return (self.kappa0 * rho ** q["kap_rho_exp"] * T ** q["kap_T_exp"]).unsqueeze(-1) * self.efac

    # -- reconstruction along d of cells -1 .. n from padded cells -2 .. n+1
    def parabola(self, f, d):
        A = self.ax[d]
        pm, p0, pp = self.cut(f, d, 0, 2), self.cut(f, d, 1, 1), self.cut(f, d, 2, 0)
        c = lambda a: self.along(a, d)  # noqa: E731
        dl, dr = p0 - pm, pp - p0
        a = c(A.wa[0]) * pm + c(A.wa[1]) * p0 + c(A.wa[2]) * pp
        b = c(A.wb[0]) * pm + c(A.wb[1]) * p0 + c(A.wb[2]) * pp

        def clamp(f, pa, dlt, pb, s):
            u, w = pa + dlt * c(s ** 2), pb - dlt * c((1.0 - s) ** 2)
            lo, hi = torch.where(dlt < 0, w, u), torch.where(dlt < 0, u, w)
            return torch.where(f < lo, lo, torch.where(f > hi, hi, f))

        a, b = clamp(a, pm, dl, p0, A.sl), clamp(b, p0, dr, pp, A.sr)
        sl = c(A.al[0]) * a + c(A.al[1]) * p0 + c(A.al[2]) * b
        sr = c(A.ar[0]) * a + c(A.ar[1]) * p0 + c(A.ar[2]) * b
        inside, flat, lower = sl * sr < 0, sl.abs() == sr.abs(), sl.abs() < sr.abs()
        an = torch.where(inside, torch.where(flat, p0, torch.where(lower, a, b + (p0 - b) * c(A.rr))), a)
        bn = torch.where(inside, torch.where(flat, p0, torch.where(lower, a + (p0 - a) * c(A.rl), b)), b)
        ext = dl * dr <= 0
        return torch.where(ext, p0, an), torch.where(ext, p0, bn)

    def linear(self, f, d):
        A = self.ax[d]
        pm, p0, pp = self.cut(f, d, 0, 2), self.cut(f, d, 1, 1), self.cut(f, d, 2, 0)
        c = lambda a: self.along(a, d, 1)  # noqa: E731
        s = _mc((p0 - pm) / c(A.gl), (pp - p0) / c(A.gr), (pp - pm) / c(A.gc))
        return p0 + s * c(A.dl), p0 + s * c(A.dr)

    def m1(self, E, F, n):
        """Row n of the pressure tensor."""
        pos = E > 0
        Es = torch.where(pos, E, torch.ones_like(E))
        f2 = sum(f * f for f in F) / (self.c * Es) ** 2
        scale = torch.where(f2 > 1, 1.0 / f2.clamp_min(1.0), torch.ones_like(f2))
        f2 = f2.clamp_max(1.0)
        qd = 1.0 / (2.0 + torch.sqrt(4.0 - 3.0 * f2))
        w = 3.0 * qd * scale * F[n] / (self.c ** 2 * Es)
        return [torch.where(pos, w * F[k] + (E * (1.0 / 3.0 - f2 * qd) if k == n else 0.0), E / 3.0 if k == n else torch.zeros_like(E))
                for k in range(self.D)]

    def hllc(self, L, R):
        gam, D = self.gam, self.D
        rl, pl, ul, rr, pr, ur = L[0], L[1], L[2], R[0], R[1], R[2]
        El = pl / (gam - 1) + 0.5 * rl * sum(x * x for x in L[2:2 + D])
        Er = pr / (gam - 1) + 0.5 * rr * sum(x * x for x in R[2:2 + D])
        al, ar, sl, sr = torch.sqrt(gam * pl / rl), torch.sqrt(gam * pr / rr), torch.sqrt(rl), torch.sqrt(rr)
        H = (sl * (El + pl) / rl + sr * (Er + pr) / rr) / (sl + sr)
        vt = [(sl * L[2 + k] + sr * R[2 + k]) / (sl + sr) for k in range(D)]
        at = torch.sqrt(((gam - 1) * (H - 0.5 * sum(x * x for x in vt))).clamp_min(0.0))
        SL, SR = torch.minimum(ul - al, vt[0] - at), torch.maximum(ur + ar, vt[0] + at)
        dl, dr = rl * (SL - ul), rr * (SR - ur)
        Ss = (pr - pl + ul * dl - ur * dr) / (dl - dr)
        U = lambda W, E: [W[0], *[W[0] * W[2 + k] for k in range(D)], E]  # noqa: E731

        def flux(W, E):
            f = [W[0] * W[2] * x for x in (torch.ones_like(W[0]), *W[2:2 + D])] + [(E + W[1]) * W[2]]
            f[1] = f[1] + W[1]
            return f

        def star(W, E, S):
            fac = W[0] * (S - W[2]) / (S - Ss)
            return [fac, fac * Ss, *[fac * x for x in W[3:2 + D]], fac * (E / W[0] + (Ss - W[2]) * (Ss + W[1] / (W[0] * (S - W[2]))))]

        UL, UR, FL, FR = U(L, El), U(R, Er), flux(L, El), flux(R, Er)
        sL, sR = star(L, El, SL), star(R, Er, SR)
        out = [torch.where(SL >= 0, FL[k], torch.where(SR < 0, FR[k], torch.where(
            Ss >= 0, FL[k] + SL * (sL[k] - UL[k]), FR[k] + SR * (sR[k] - UR[k])))) for k in range(2 + D)]
        bl, br = SL.clamp_max(0.0), SR.clamp_min(0.0)
        hlle = lambda: [(br * FL[k] - bl * FR[k] + bl * br * (UR[k] - UL[k])) / (br - bl) for k in range(2 + D)]  # noqa: E731
        return out, Ss, hlle

    def prims(self, gas, h):
        rho, v = gas[0], [gas[1 + k] / (gas[0] * h[k]) for k in range(self.D)]
        return [rho, (self.gam - 1.0) * (gas[-1] - 0.5 * rho * sum(x * x for x in v)), *v]

    def face_geometry(self, d):
        """Areas of the faces 0 .. n of direction d for scalars and for covariant component k, and the normal scale factor."""
        D = self.D
        if not self.sph:
            return 1.0, [1.0] * D, 1.0
        R, T = self.ax
        if d == 0:
            r = self.along(np.exp(R.xl[2:-1]), 0)
            th = self.along(T.vol[2:-2], 1)
            return r ** 2 * th, [r ** 3 * th] * 2, r
        s = self.along(np.abs(np.sin(T.xl[2:-1])), 1)
        ra, rb, rc = (self.along(x[2:-2], 0) for x in (self.ra, self.rb, self.rc))
        return s * ra, [s * rb, s * rc], rc / ra

    def rhs(self, gas, rad, comp):
        """dU/dt of the explicit operator, and the radiation energy leaving through the upper x boundary."""
        D, c, q = self.D, self.c, self.q
        dg, dr, dc, phi = torch.zeros_like(gas), torch.zeros_like(rad), None if comp is None else torch.zeros_like(comp), 0.0
        flags = None
        hc = [self.along(self.h[k][2:-2], 0) for k in range(2)] if self.sph else [1.0] * D
        if q.get("shock_guard", 0.0) > 0:
            p = self.prims(gas, hc)[1]
            flags = []
            for d in range(D):
                pp = self.pad(p, d)
                a, b = self.cut(pp, d, 0, 1), self.cut(pp, d, 1, 0)
                jump = torch.maximum(a, b) > (1.0 + q["shock_guard"]) * torch.minimum(a, b)
                flags.append(self.cut(jump, d, 1, 2) | self.cut(jump, d, 2, 1))
        vface = []
        if self.sph:
            V = self.along(self.ax[0].vol[2:-2], 0) * self.along(self.ax[1].vol[2:-2], 1)
        for d in range(D):
            A = self.ax[d]
            sgn = [-1.0 if k == d else 1.0 for k in range(D)]
            ug = [self.pad(gas[0], d), *[self.pad(gas[1 + k], d, sgn[k]) for k in range(D)], self.pad(gas[-1], d)]
            h = hc if not self.sph else [self.along(self.h[k] if d == 0 else self.h[k][2:-2], 0) for k in range(2)]
            W = self.prims(ug, h)
            rec = [self.parabola(w, d) for w in W]
            L = [self.cut(b, d, 0, 1) for _, b in rec]
            Rr = [self.cut(a, d, 1, 0) for a, _ in rec]
            rot = lambda X: [X[0], X[1], *[X[2 + (d + k) % D] for k in range(D)]]  # noqa: E731
            fl, vs, hlle = self.hllc(rot(L), rot(Rr))
            if flags is not None:
                other = torch.zeros_like(vs, dtype=torch.bool)
                for e in range(D):
                    if e != d:
                        fe = self.pad(flags[e].to(torch.uint8), d)
                        other = other | (self.cut(fe, d, 1, 2) > 0) | (self.cut(fe, d, 2, 1) > 0)
                fl = [torch.where(other, y, x) for x, y in zip(fl, hlle())]
            area, ac, hn = self.face_geometry(d)
            div = lambda f: (self.cut(f, d, 1, 0) - self.cut(f, d, 0, 1)) / (V if self.sph else A.dx)  # noqa: E731, B023
            divr = lambda f: (self.cut(f, d, 1, 0) - self.cut(f, d, 0, 1)) / (V.unsqueeze(-1) if self.sph else A.dx)  # noqa: E731, B023
            dg[0] -= div(fl[0] * area)
            for k in range(D):
                dg[1 + (d + k) % D] -= div(fl[1 + k] * ac[(d + k) % D])
            dg[-1] -= div(fl[-1] * area)
            if comp is not None:
                a, b = self.parabola(self.pad(comp, d) / ug[0], d)
                dc -= div(fl[0] * area * torch.where(vs >= 0, self.cut(b, d, 0, 1), self.cut(a, d, 1, 0)))
            if q.get("vterms", 0):
                up = [torch.where(vs >= 0, L[2 + k], Rr[2 + k]) for k in range(D)]
                up[d] = vs
                vface.append(up)
            # radiation
            T = W[1] / W[0]
            chi = self.kappa(W[0], T.clamp_min(1e-300)) * (T > 0).unsqueeze(-1)
            chi = self.cut(chi, d, 1, 1)
            hr = [1.0] * D if not self.sph else [x.unsqueeze(-1) for x in h]
            Q = [self.pad(rad[0], d)] + [self.pad(rad[1 + k], d, sgn[k]) / hr[k] for k in range(D)]
            rec = [self.linear(x, d) for x in Q]
            QL, QR = [self.cut(b, d, 0, 1) for _, b in rec], [self.cut(a, d, 1, 0) for a, _ in rec]
            del rec, Q
            PL, PR = self.m1(QL[0], QL[1:], d), self.m1(QR[0], QR[1:], d)
            ell = self.along(A.cen[2:-1] - A.cen[1:-2], d)
            ell = (ell * hn).unsqueeze(-1) if self.sph else ell.unsqueeze(-1)
            tau = 0.5 * (self.cut(chi, d, 0, 1) + self.cut(chi, d, 1, 0)) * ell
            eps = 1.0 / tau.clamp_min(1.0)
            v = vs.unsqueeze(-1)
            up = v >= 0
            r1 = (lambda x: x.unsqueeze(-1)) if self.sph else (lambda x: x)
            fE = (0.5 * (QL[1 + d] + QR[1 + d]) - 0.5 * c * eps * (QR[0] - QL[0]) + v * torch.where(up, QL[0], QR[0])) * r1(area)
            dr[0] -= divr(fE)
            if d == 0 and not self.sph:
                others = math.prod(self.ax[e].dx for e in range(1, D)) if D > 1 else 1.0
                phi = fE.narrow(D - 1, fE.shape[D - 1] - 1, 1).sum() * others
            for k in range(D):
                f = 0.5 * c * c * (PL[k] + PR[k]) - 0.5 * c * (QR[1 + k] - QL[1 + k]) + v * torch.where(up, QL[1 + k], QR[1 + k])
                dr[1 + k] -= divr(f * r1(ac[k]))
        if self.sph:
            self.geometric(gas, rad, hc, dg, dr)
        if vface:
            Vg = [[(self.cut(vface[b][a], b, 1, 0) - self.cut(vface[b][a], b, 0, 1)) / self.ax[b].dx for b in range(D)] for a in range(D)]
            self.velocity_terms(rad, Vg, dr)
        return dg, dr, dc, phi

    def geometric(self, gas, rad, h, dg, dr):
        rho, p, v1, v2 = self.prims(gas, h)
        g111, g221, g122 = (self.along(x[2:-2], 0) for x in (self.g111, self.g221, self.g122))
        g222, g332 = (self.along(x[2:-2], 1) for x in (self.g222, self.g332))
        a, b = h[0] / h[1], h[1] / h[0]
        dg[1] += g111 * (rho * v1 * v1 + p) + g221 * (rho * v2 * v2 + p) + g221 * p
        dg[2] += g122 * rho * v1 * v2 * a + g221 * rho * v1 * v2 * b + g222 * (rho * v2 * v2 + p) + g332 * p
        E, F = rad[0], [rad[1] / h[0].unsqueeze(-1), rad[2] / h[1].unsqueeze(-1)]
        c2 = self.c ** 2
        P0, P1 = self.m1(E, F, 0), self.m1(E, F, 1)
        P33 = E - P0[0] - P1[1]
        u = lambda x: x.unsqueeze(-1)  # noqa: E731
        R11, R22 = c2 * P0[0] + u(v1) * F[0], c2 * P1[1] + u(v2) * F[1]
        R21, R12 = (c2 * P0[1] + u(v2) * F[0]) * u(a), (c2 * P0[1] + u(v1) * F[1]) * u(b)
        dr[1] += u(g111) * R11 + u(g221) * R22 + u(g221) * c2 * P33
        dr[2] += u(g122) * R21 + u(g221) * R12 + u(g222) * R22 + u(g332) * c2 * P33

    def velocity_terms(self, rad, V, dr):
        """Work terms and upwind frequency fluxes of nu P and nu Q (Cartesian)."""
        D, G, c = self.D, self.G, self.c
        nu = self.t(self.edge)
        mid, dnu = 0.5 * (nu[1:] + nu[:-1]), nu[1:] - nu[:-1]
        E, F = rad[0], [rad[1 + k] for k in range(D)]
        Fm = torch.sqrt(sum(f * f for f in F))
        ok = (Fm > 0) & (E > 0)
        f = torch.where(ok, Fm / (c * torch.where(ok, E, torch.ones_like(E))), torch.zeros_like(E)).clamp_max(1.0)
        chi = (3 + 4 * f * f) / (5 + 2 * torch.sqrt(4 - 3 * f * f))
        qf = f * (2 + 3 * chi) / 5
        n = [torch.where(ok, x / torch.where(ok, Fm, torch.ones_like(Fm)), torch.zeros_like(x)) for x in F]
        P = lambda i, j: E * ((0.5 * (1 - chi) if i == j else 0.0) + 0.5 * (3 * chi - 1) * n[i] * n[j])  # noqa: E731
        Q = lambda k, j, i: c * E * (0.5 * (f - qf) * ((n[k] if i == j else 0.0) + (n[j] if i == k else 0.0) + (n[i] if j == k else 0.0))  # noqa: E731
                                     + 0.5 * (5 * qf - 3 * f) * n[k] * n[j] * n[i])

        def edge_flux(x, v):
            """v times the upwind value of the density x at the interior edges, times nu."""
            x = x / dnu
            s = torch.zeros_like(x)
            if G > 2:
                m = x[..., 1:-1]
                s[..., 1:-1] = _mc((m - x[..., :-2]) / (mid[1:-1] - mid[:-2]), (x[..., 2:] - m) / (mid[2:] - mid[1:-1]),
                                   (x[..., 2:] - x[..., :-2]) / (mid[2:] - mid[:-2]))
            lo, hi = x - s * (mid - nu[:-1]), x + s * (nu[1:] - mid)
            return v * torch.where(v < 0, hi[..., :-1], lo[..., 1:]) * nu[1:-1]

        zero = torch.zeros_like(E[..., :1])
        net = lambda f: torch.diff(torch.cat([zero, f, zero], -1), dim=-1)  # noqa: E731
        fE = 0.0
        for i in range(D):
            for j in range(D):
                v = V[i][j].unsqueeze(-1)
                fE = fE + edge_flux(P(i, j), v)
                dr[0] -= v * P(i, j)
                dr[1 + j] -= v * F[i]
        dr[0] += net(fE)
        for j in range(D):
            fF = 0.0
            for i in range(D):
                for k in range(D):
                    fF = fF + edge_flux(Q(k, j, i), V[i][k].unsqueeze(-1))
            dr[1 + j] += net(fF)

    # -- the implicit interaction
    def couple(self, gas, rad, comp, dt):
        D, c, q = self.D, self.c, self.q
        cv, b = 1.0 / (self.gam - 1.0), q["kap_T_exp"]
        hc = [self.along(self.h[k][2:-2], 0) for k in range(2)] if self.sph else [1.0] * D
        rho = gas[0]
        ke = 0.5 * rho * sum((gas[1 + k] / (rho * hc[k])) ** 2 for k in range(D))
        um, Em = gas[-1] - ke, rad[0].clamp_min(1e-300 if q["precision"] == "fp64" else 1e-37)  # (positivity floor)
        kr = (self.kappa0 * rho ** q["kap_rho_exp"]).unsqueeze(-1) * self.efac
        Yv = comp / rho if comp is not None else None

        def energies(T, Y):
            B, dB = self.planck(T)
            if self.S > 1:
                B, dB = B.repeat([1] * D + [3]), dB.repeat([1] * D + [3])
            tau = c * dt * kr * (T ** b).unsqueeze(-1)
            w = 1.0 if Y is None else self.w0 + self.dw * Y.unsqueeze(-1)
            E = (Em + tau * w * B) / (1.0 + tau)
            dE = (tau * w * dB + tau * (b / T).unsqueeze(-1) * (w * B - E)) / (1.0 + tau)
            return E, dE, tau, B, dB

        with torch.no_grad():
            T = (um / (rho * cv)).clone()
            if comp is None:
                lo, hi = torch.zeros_like(T), torch.full_like(T, math.inf)
                for _ in range(80):
                    E, dE = energies(T, None)[:2]
                    r, drdT = rho * cv * T - um + (E - Em).sum(-1), rho * cv + dE.sum(-1)
                    lo, hi = torch.where(r < 0, T, lo), torch.where(r > 0, T, hi)
                    new = T - r / drdT
                    bad = ~((new > lo) & (new < hi)) & (r != 0)
                    new = torch.where(bad, torch.where(torch.isinf(hi), 2.0 * T, 0.5 * (lo + hi)), new)
                    done = bool(((new - T).abs() <= 4e-16 * T).all())
                    T = torch.where(r == 0, T, new)
                    if done:
                        break
            else:
                Y = Yv.clone()
                sE, sX = um + Em.sum(-1), comp.abs() + (self.xi.abs() * Em).sum(-1)

                def residual(T, Y):
                    E, dE, tau, B, _ = energies(T, Y)
                    dY = tau * self.dw * B / (1.0 + tau)
                    rE = rho * cv * T - um + (E - Em).sum(-1)
                    rX = rho * (Y - Yv) - (self.xi * (E - Em)).sum(-1)
                    return rE, rX, rho * cv + dE.sum(-1), dY.sum(-1), -(self.xi * dE).sum(-1), rho - (self.xi * dY).sum(-1)

                size = lambda r: (r[0] / sE) ** 2 + (r[1] / sX) ** 2  # noqa: E731
                now = residual(T, Y)
                for _ in range(40):
                    det = now[2] * now[5] - now[3] * now[4]
                    dT, dY = -(now[5] * now[0] - now[3] * now[1]) / det, -(now[2] * now[1] - now[4] * now[0]) / det
                    lam = torch.ones_like(T)
                    for _ in range(30):
                        Tn, Yn = T + lam * dT, Y + lam * dY
                        okay = (Tn > 0) & (Yn >= 0) & (Yn <= 1)
                        new = residual(torch.where(okay, Tn, T), torch.where(okay, Yn, Y))
                        okay &= (size(new) < size(now)) | (size(now) < 1e-29)
                        if bool(okay.all()):
                            break
                        lam = torch.where(okay, lam, 0.5 * lam)
                    T, Y = torch.where(okay, Tn, T), torch.where(okay, Yn, Y)
                    now = residual(T, Y)
                    if bool(((size(now) < 1e-29) & (dT.abs() <= 1e-13 * T)).all()):
                        break
        if comp is None:
            # the converged temperature as a function of the inputs: one Newton step at the root
            with torch.no_grad():
                _, dE, _, B, dB = energies(T, None)
                slope = rho * cv + dE.sum(-1)
            E = energies(T, None)[0]
            Td = T - (rho * cv * T - um + (E - Em).sum(-1)) / slope
            tau = c * dt * kr * (Td ** b).unsqueeze(-1)
            En = (Em + tau * (B + dB * (Td - T).unsqueeze(-1))) / (1.0 + tau)
        else:
            En, _, tau, _, _ = energies(T, Y)
            comp = comp + (self.xi * (En - Em)).sum(-1)
        u = um - (En - Em).sum(-1)
        fac = 1.0 / (1.0 + tau)
        Fn = [rad[1 + k] * fac for k in range(D)]
        dm = [(Fn[k] - rad[1 + k]).sum(-1) for k in range(D)]
        work = sum(gas[1 + k] / (rho * hc[k] ** 2) * dm[k] for k in range(D))
        m = [gas[1 + k] - dm[k] / c ** 2 for k in range(D)]
        return torch.stack([rho, *m, ke + u - work / c ** 2]), torch.stack([En, *Fn]), comp

    def layer(self, gas, rad, layers, t):
        gas, rad, D = gas.clone(), rad.clone(), self.D
        x = self.along(self.ax[0].xc[2:-2], 0).expand(gas[0].shape)
        y = self.along(self.ax[1].xc[2:-2], 1).expand(gas[0].shape)
        for ly in layers:
            (x0, y0, _), (x1, y1, _) = ly["lo"], ly["hi"]
            box = (slice(y0, y1), slice(x0, x1))
            if ly["kind"] == "mirror":
                src = (torch.arange(2 * ly["m"] - 1 - y0, 2 * ly["m"] - 1 - y1, -1, device=DEV), slice(x0, x1))
                for k in range(2 + D):
                    gas[k][box] = gas[k][src] * (-1.0 if k == 1 + ly["d"] else 1.0)
                for k in range(1 + D):
                    rad[k][box] = rad[k][src] * (-1.0 if k == 1 + ly["d"] else 1.0)
                continue
            behind = x[box] - ly["x0"] - (y[box] - ly["y0"]) * ly["cot_alpha"] - ly["speed"] * t <= 0
            prim = torch.stack([_pick(behind, a, b) for a, b in zip(ly["A"], ly["B"])])
            g2, r2, _ = self.equilibrium(prim)
            gas[(slice(None), *box)], rad[(slice(None), *box)] = g2, r2
        return gas, rad

    def step(self, gas, rad, comp, dt, layers=(), t=0.0):
        """One SSP-RK2 step with the interaction after each stage; also the objective's part."""
        on = self.q.get("couple", 1)
        if layers:
            gas, rad = self.layer(gas, rad, layers, t)
        g, r, k, phi0 = self.rhs(gas, rad, comp)
        g, r, k = gas + dt * g, rad + dt * r, None if comp is None else comp + dt * k
        if on:
            g, r, k = self.couple(g, r, k, dt)
        if layers:
            g, r = self.layer(g, r, layers, t + dt)
        g2, r2, k2, phi1 = self.rhs(g, r, k)
        g = 0.5 * gas + 0.5 * (g + dt * g2)
        r = 0.5 * rad + 0.5 * (r + dt * r2)
        k = None if comp is None else 0.5 * comp + 0.5 * (k + dt * k2)
        if on:
            g, r, k = self.couple(g, r, k, 0.5 * dt)
        if layers:
            g, r = self.layer(g, r, layers, t + dt)
        return g, r, k, 0.5 * dt * (phi0 + phi1)


def _mc(sl, sr, sc):
    """The MC limiter's slope."""
    m = torch.minimum(torch.minimum(2.0 * sl.abs(), 2.0 * sr.abs()), sc.abs())
    return torch.where(sl * sr > 0, torch.where(sc > 0, m, -m), torch.zeros_like(m))


def exact(case, seed):
    q, prim, layers = _setup(case, seed)
    M = _Method(q)
    D, N, n = M.D, math.prod(q["n"][:M.D]), tuple(reversed(q["n"][:M.D]))
    if case["kind"] == "mach":
        gas, rad, comp = M.equilibrium(prim)
    else:
        flat = _snapshot(case, seed, q, prim).to(F64)
        g, r = (2 + D) * N, (1 + D) * N * M.K
        gas, rad = flat[:g].view(2 + D, *n), flat[g:g + r].view(1 + D, *n, M.K)
        comp = flat[g + r:].view(n) if M.S > 1 else None
    if case["kind"] == "gradient":
        rho = gas[0].clone().requires_grad_()
        M.kappa0 = torch.tensor(q["kappa0"], dtype=F64, device=DEV, requires_grad=True)
        v = gas[1:1 + D] / gas[0]  # pressure, velocity and radiation held fixed
        u = gas[-1] - 0.5 * gas[0] * (v ** 2).sum(0)
        gas, J = torch.stack([rho, *[rho * v[k] for k in range(D)], u + 0.5 * rho * (v ** 2).sum(0)]), 0.0
        for _ in range(case["steps"]):
            gas, rad, comp, part = M.step(gas, rad, comp, q["dt"])
            J = J + part
        J.backward()
        return {"J": J.detach(), "rho": rho.grad.reshape(-1), "kappa": M.kappa0.grad}
    for k in range(case["steps"]):
        gas, rad, comp, _ = M.step(gas, rad, comp, q["dt"], layers, k * q["dt"])
    out = {"gas": gas.reshape(2 + D, N), "E": rad[0].reshape(N, M.K), "F": rad[1:].reshape(D, N, M.K)}
    if comp is not None:
        out["rho_ye"] = comp.reshape(-1)
    return out

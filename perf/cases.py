"""What is timed of this library: the calls that a user's program makes, at the sizes and with the options it uses.

Every case is one pass through the public entry points (``Plan``, ``Batch``, ``autograd.evolve``): split steps
in 2D and 3D, float32 and float64; the batched 2D runs; a gradient; a ground state; the observables; steps on
host memory. ``exact`` restates each in 64-bit torch from the equations of the scheme alone.
"""
import math
import random

import numpy as np
import torch

import paper_1512_03210_gb300 as fse
from paper_1512_03210_gb300.autograd import evolve, overlap_objective

SQ = 1.0 / math.sqrt(2.0)
SIZES = (8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512)  # per axis
BATCH_SIZES = (128, 192, 256, 384, 512)


def listed():
    return [
        # one step per call with a trap frequency of its own: a control loop on a small grid, all latency
        dict(name="step_2d_64_f32", kind="step", nx=64, ny=64, nz=0, prec="f32", kernel="coulomb", steps=1, control=True),
        # the 2D Coulomb workload in float64, ten steps between looks at the field
        dict(name="step_2d_128_f64", kind="step", nx=128, ny=128, nz=0, prec="f64", kernel="coulomb", steps=10),
        # an oblong 2D grid with radix-3 lengths and the in-plane dipolar kernel
        dict(name="step_2d_384x192_f32", kind="step", nx=384, ny=192, nz=0, prec="f32", kernel="ddi2d", steps=4),
        # the 3D dipolar workload at its middle size
        dict(name="step_3d_128_f32", kind="step", nx=128, ny=128, nz=128, prec="f32", kernel="ddi3d", steps=4),
        # the 3D dipolar workload that the benchmark quotes: the largest call
        dict(name="step_3d_256_f32", kind="step", nx=256, ny=256, nz=256, prec="f32", kernel="ddi3d", steps=4),
        # a ragged 3D grid of a flat cloud, held to its mass
        dict(name="step_3d_ragged_f32", kind="step", nx=192, ny=96, nz=48, prec="f32", kernel="coulomb", steps=4, renormalize=1),
        # the float64 path that accuracy studies compare with
        dict(name="step_3d_128_f64", kind="step", nx=128, ny=128, nz=128, prec="f64", kernel="ddi3d", steps=1),
        # parameter scans: 256 independent 2D runs of mixed sizes advanced together
        dict(name="batch_2d_256", kind="batch", runs=256, mix=2, steps=4),
        # optimal control: gradient of an overlap with respect to the start and the trap frequencies
        dict(name="gradient_2d_256_f32", kind="gradient", nx=256, ny=256, prec="f32", steps=36),
        # the gradient-flow ground state on the paper's grid
        dict(name="ground_2d_512_f64", kind="ground", nx=512, ny=512, nz=0, omega=0.0, s=0.8, dt=1e-3, outer=2),
        # the conserved quantities that a run logs
        dict(name="observables_3d_128_f32", kind="observables", nx=128, ny=128, nz=128, prec="f32", kernel="ddi3d"),
        # a program whose field lives in (page-locked) host memory
        dict(name="host_3d_128_f32", kind="host", nx=128, ny=128, nz=128, prec="f32", kernel="ddi3d", steps=1),
    ]


def _sizes(rng, dim, most):
    """Supported axis lengths, within a factor of 8 of one another, at most `most` points in all."""
    while True:
        n = [rng.choice(SIZES) for _ in range(dim)]
        if max(n) <= 8 * min(n) and 16 ** dim <= math.prod(n) <= most:
            return n


def draw(rng):
    most = _cost(next(c for c in listed() if c["name"] == "step_3d_256_f32"))
    while True:
        c = _draw(rng)
        if _cost(c) <= most:
            return c


def _cost(case):
    """Work of a pass, float64 at its rate (a sixteenth or less of float32's); the lattice's sines count for seven steps."""
    f64 = case["kind"] == "ground" or case.get("prec") == "f64"
    return work(case)["flops"] * (16 if f64 else 1) * (8 if case.get("lattice") else 1)


def _draw(rng):
    kind = rng.choice(("step", "step", "step", "step", "batch", "gradient", "ground", "observables", "host"))
    if kind == "batch":
        return dict(kind=kind, runs=int(round(2 ** rng.uniform(2, 8))), mix=rng.randrange(1 << 20), steps=rng.choice((1, 2, 4)))
    prec = rng.choice(("f32", "f32", "f64"))
    if kind == "gradient":
        n = _sizes(rng, 2, 256 * 256)
        return dict(kind=kind, nx=n[0], ny=n[1], prec=prec, steps=rng.randint(4, 36))
    dim = rng.choice((2, 3))
    if kind == "ground":
        n = _sizes(rng, dim, 512 * 512)
        s = rng.choice((0.8, 1.0))
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2] if dim == 3 else 0, omega=rng.choice((0.0, 0.3)) if s == 1.0 else 0.0, s=s,
                    dt=rng.choice((1e-3, 1e-2)), outer=rng.choice((1, 2)))
    n = _sizes(rng, dim, 512 * 512 if dim == 2 else (256 ** 3 if prec == "f32" and kind == "step" else 128 ** 3))
    c = dict(kind=kind, nx=n[0], ny=n[1], nz=n[2] if dim == 3 else 0, prec=prec, kernel=rng.choice(("coulomb", "coulomb", "ddi%dd" % dim, "ddi%dd" % dim, "none")))
    if kind != "observables":
        c["steps"] = rng.choice((1, 2, 4)) if prec == "f32" else 1
    if kind == "step":
        option = rng.choice(("", "", "renormalize", "control", "order", "lattice"))
        if option in ("renormalize", "control"):
            c[option] = 1
        elif option == "order" and c["steps"] < 4:
            c["order"] = 4
        elif option == "lattice":
            c["lattice"] = 10.0
    return c


# ----- what a program has in hand -----

def _n(case):
    return tuple(case[k] for k in ("nx", "ny", "nz") if case.get(k))


def _params(case, rng):
    """The parameter dict of a plan: the physics of the repository's workloads, strengths drawn from the seed."""
    n = _n(case)
    dim = len(n)
    half = [min(12.0, max(4.0, v / 16.0)) if dim == 3 else min(16.0, max(6.0, v / 16.0)) for v in n]
    kernel = case.get("kernel", "coulomb")
    p = dict(dim=dim, n=n, lo=tuple(-h for h in half), hi=tuple(half), s=0.6 + 0.2 * rng.random(), m=0.0,
             omega=0.5 + 0.4 * rng.random(), beta=100.0 + 400.0 * rng.random(), lam=10.0 if dim == 2 else 60.0,
             dt=1e-3 if dim == 2 else 2.5e-4, kernel=kernel, mu=1.0, gamma=(1.0, 1.2, 2.0)[:dim], prec=case.get("prec", "f64"),
             dip_n={"ddi3d": (SQ, 0.0, SQ), "ddi2d": (0.48, -0.36, 0.8)}.get(kernel, (0.0, 0.0, 1.0)))
    if case.get("renormalize"):
        p["renormalize"] = 1
    if case.get("order"):
        p["order"] = case["order"]
    if case.get("lattice"):
        p.update(lat_amp=case["lattice"], lat_k=(math.pi, 0.8 * math.pi, 0.5 * math.pi)[:dim])
    if case["kind"] == "ground":
        p.update(s=case["s"], omega=case["omega"], beta=10.0 + 30.0 * rng.random(), lam=10.0, gamma=(1.0, 1.1, 1.5)[:dim])
    return p


def _axes(p):
    """x, y[, z] as float64 tensors that broadcast to the field's shape [nz][ny][nx]."""
    ax = []
    for j in range(p["dim"]):
        a = p["lo"][j] + (p["hi"][j] - p["lo"][j]) / p["n"][j] * torch.arange(p["n"][j], device="cuda", dtype=torch.float64)
        ax.append(a.view([-1 if p["dim"] - 1 - j == d else 1 for d in range(p["dim"])]))
    return ax


def _cell(p):
    return math.prod((p["hi"][j] - p["lo"][j]) / p["n"][j] for j in range(p["dim"]))


def _field(p, rng, vortices=4):
    """A displaced, moving cloud of unit mass with a few phase vortices (complex128)."""
    ax = _axes(p)
    psi = torch.ones((), device="cuda", dtype=torch.complex128)
    for j, a in enumerate(ax):
        psi = psi * torch.exp(-0.5 * p["gamma"][j] * (a - rng.uniform(-0.8, 0.8)) ** 2 + 1j * rng.uniform(-0.6, 0.6) * a)
    for _ in range(vortices):
        z = (ax[0] - rng.uniform(-1.5, 1.5)) + 1j * (ax[1] - rng.uniform(-1.5, 1.5))
        psi = psi * (z / torch.sqrt(z.abs() ** 2 + 0.25))
    return psi / torch.sqrt(_cell(p) * (psi.abs() ** 2).sum())


def _type(p):
    return torch.complex64 if p["prec"] == "f32" else torch.complex128


def _gammas(p, steps, rng):
    g = np.ones((steps, p["dim"]))
    for v in range(p["dim"]):
        g[:, v] += 0.2 * np.sin(2 * np.pi * (np.arange(steps) / 200.0 + rng.random()))
    return g


def _batch_sizes(case):
    rng = random.Random(case["mix"])
    return [rng.choice(BATCH_SIZES) for _ in range(case["runs"])]


def _batch_params(case, rng):
    return [dict(dim=2, n=(n, n), lo=(-8.0, -8.0), hi=(8.0, 8.0), s=0.3 + 0.7 * rng.random(), m=0.0, omega=0.95 * rng.random(),
                 beta=50.0 + 450.0 * rng.random(), lam=10.0, dt=1e-3, kernel="coulomb", mu=1.0, gamma=(1.0, 1.0), prec="f32")
            for n in _batch_sizes(case)]


def _inputs(case, seed):
    """Parameters and start data, from the seed alone: what prepare() hands to the library and exact() starts from."""
    rng = random.Random(seed)
    if case["kind"] == "batch":
        ps = _batch_params(case, rng)
        return ps, [_field(p, rng, vortices=1).to(torch.complex64) for p in ps], None
    p = _params(case, rng)
    psi = _field(p, rng, vortices=0 if case["kind"] == "ground" else 4).to(_type(p))
    extra = None
    if case["kind"] == "gradient":
        # trap frequencies as a float32 parameter tensor, and the target of the overlap
        extra = (torch.tensor(_gammas(p, case["steps"], rng), dtype=torch.float32), _field(p, rng, vortices=0).to(_type(p)))
    elif case.get("control"):
        extra = _gammas(p, case["steps"], rng)
    return p, psi, extra


def prepare(case, seed):
    p, psi, extra = _inputs(case, seed)
    st = dict(kind=case["kind"], steps=case.get("steps", 0), t=0.0, extra=extra)
    if case["kind"] == "batch":
        # the runs' fields side by side in one buffer
        flat = torch.empty(sum(x.numel() for x in psi), dtype=torch.complex64, device="cuda")
        views, at = [], 0
        for x in psi:
            v = flat[at:at + x.numel()].view(x.shape)
            v.copy_(x)
            views.append(v)
            at += x.numel()
        st.update(batch=fse.Batch(p), flat=flat, psi=views, dt=p[0]["dt"])
        return st
    st.update(plan=fse.Plan(p), psi=psi, dt=p["dt"])
    if case["kind"] == "host":
        st["psi"] = psi.cpu().pin_memory().numpy()
    elif case["kind"] == "gradient":
        st.update(psi=psi.requires_grad_(True), gam=extra[0].requires_grad_(True), target=extra[1], cell=_cell(p))
    elif case["kind"] == "ground":
        st.update(gs=dict(dt=case["dt"], max_outer=case["outer"], tol=0.0, max_inner=500, inner_tol=1e-12))
    return st


def run(st):
    kind, n = st["kind"], st["steps"]
    if kind == "step":
        st["plan"].step(st["psi"], st["t"], n, st["extra"])
        st["t"] += n * st["dt"]
        return st["psi"]
    if kind == "batch":
        st["batch"].step(st["psi"], st["t"], n)
        st["t"] += n * st["dt"]
        return st["flat"]
    if kind == "host":
        st["plan"].step_host(st["psi"], st["t"], n)
        st["t"] += n * st["dt"]
        return st["psi"]
    if kind == "gradient":
        out = evolve(st["plan"], st["psi"], st["gam"], 0.0)
        J = overlap_objective(out, st["target"], st["cell"])
        g = torch.autograd.grad(J, (st["psi"], st["gam"]))
        return dict(out=out.detach(), objective=J.detach(), psi=g[0], gamma=g[1])
    if kind == "ground":
        psi = st["psi"].clone()
        info = st["plan"].ground_state(psi, **st["gs"])
        return dict(psi=psi, change=info["change"])
    return st["plan"].observables(st["psi"], 0.3)


# ----- what one pass cannot do without -----

def _fft(n):
    return 5.0 * n * math.log2(n)


def _step_flops(n, nonlocal_):
    """Two full transforms of the field and a zero-padded real convolution, 5 N log2 N each, and the pointwise factors."""
    N = math.prod(n)
    f = 2 * _fft(N) + 40.0 * N
    if nonlocal_:
        f += _fft(2 ** len(n) * N) + 6.0 * 2 ** (len(n) - 1) * N
    return f


def work(case):
    kind = case["kind"]
    if kind == "batch":
        sizes = _batch_sizes(case)
        return {"bytes": sum(16.0 * n * n for n in sizes) + sum(4.0 * (n + 1) ** 2 for n in set(sizes)),
                "flops": case["steps"] * sum(_step_flops((n, n), True) for n in sizes)}
    n = _n(case)
    N = math.prod(n)
    nl = case.get("kernel", "coulomb") != "none"
    c = 8.0 if case.get("prec") == "f32" else 16.0
    chat = (c / 2) * math.prod(v + 1 for v in n) if nl else 0.0
    if kind == "observables":
        return {"bytes": c * N + chat, "flops": (_step_flops(n, nl) + 2 * _fft(N))}
    if kind == "ground":
        # a preconditioned solve of at least two iterations of two operator products each
        return {"bytes": 2 * c * N + chat, "flops": case["outer"] * (_step_flops(n, nl) + 4 * 2 * _fft(N))}
    steps = case["steps"] * (3 if case.get("order") == 4 else 1)
    if kind == "gradient":
        # the forward steps and their transpose, about two steps' work each
        return {"bytes": 4 * c * N + chat, "flops": 3 * steps * _step_flops(n, nl)}
    return {"bytes": 2 * c * N + chat, "flops": steps * _step_flops(n, nl)}


# ----- the same in 64 bits, from the equations -----

def _panels(a, b, panels, order=24):
    """Composite Gauss-Legendre nodes and weights on [a, b]."""
    x, w = np.polynomial.legendre.leggauss(order)
    e = np.linspace(a, b, panels + 1)
    h = 0.5 * (e[1:] - e[:-1])
    return ((h[:, None] * x) + 0.5 * (e[1:] + e[:-1])[:, None]).ravel(), (h[:, None] * w).ravel()


def _chat(p):
    """Transform of the cube-truncated kernel 1/(2^{d-1} pi |x|^mu) on |p_j| = 0..n_j: a sum of Gaussians and the near field."""
    d, mu, delta, hq = p["dim"], p["mu"], 1e-3, 0.125
    W = [p["hi"][j] - p["lo"][j] for j in range(d)]
    sc = 0.5 * max(W)
    t0 = -36.0 / mu
    t = t0 + hq * np.arange(int(math.ceil((math.log(7.0 / delta) - t0) / hq)) + 1)
    pref = 1.0 / (2.0 ** (d - 1) * math.pi)
    w = pref * 2.0 * hq / math.gamma(mu / 2) * np.exp(mu * t) / sc ** mu
    tau = np.exp(t) / sc
    g = []
    for j in range(d):
        k = math.pi * np.arange(p["n"][j] + 1) / W[j]
        y, yw = _panels(0.0, W[j], p["n"][j] // 2 + 16)
        wide = tau * W[j] < 8.0
        gj = np.where(wide[:, None], 0.0, math.sqrt(math.pi) / tau[:, None] * np.exp(-np.minimum((k[None, :] / (2 * tau[:, None])) ** 2, 700.0)))
        gj[wide] = 2.0 * (yw * np.exp(-(tau[wide, None] * y) ** 2)) @ np.cos(y[:, None] * k)
        g.append(torch.from_numpy(gj).cuda())
    r, rw = _panels(0.0, delta * sc, 8)
    gauss = (w[:, None] * np.exp(-(tau[:, None] * r) ** 2)).sum(0)
    ball, R = (2.0 if d == 2 else 4.0) * math.pi, delta * sc
    I0 = ball * (pref * R ** (d - mu) / (d - mu) - float((rw * r ** (d - 1) * gauss).sum()))
    I2 = ball * (pref * R ** (d + 2 - mu) / (d + 2 - mu) - float((rw * r ** (d + 1) * gauss).sum()))
    wq = torch.from_numpy(w).cuda()
    k2 = [(math.pi / W[j] * torch.arange(p["n"][j] + 1, device="cuda", dtype=torch.float64)) ** 2 for j in range(d)]
    if d == 2:
        C = (g[1] * wq[:, None]).T @ g[0]
        return C + I0 - I2 / 4.0 * (k2[1][:, None] + k2[0])
    C = torch.empty([v + 1 for v in reversed(p["n"])], device="cuda", dtype=torch.float64)
    for z in range(p["n"][2] + 1):
        C[z] = (g[1] * (wq * g[2][:, z])[:, None]).T @ g[0]
    return C + I0 - I2 / 6.0 * (k2[2][:, None, None] + k2[1][:, None] + k2[0])


class _Exact:
    """The split step on complex128 tensors, differentiable by torch."""

    def __init__(self, p, chat=None):
        self.p, self.d, self.ax = p, p["dim"], _axes(p)
        n, d = p["n"], self.d
        self.W = [p["hi"][j] - p["lo"][j] for j in range(d)]
        self.dims = tuple(range(d))
        self.k = [self._along(2 * math.pi * torch.fft.fftfreq(n[j], self.W[j] / n[j], device="cuda", dtype=torch.float64), j) for j in range(d)]
        k2 = sum(k ** 2 for k in self.k) + p["m"] ** 2
        self.sym = torch.where(k2 > 0, k2, torch.ones_like(k2)) ** p["s"] * (k2 > 0)
        self.nl = p["kernel"] != "none" and p["lam"] != 0.0
        if not self.nl:
            return
        self.chat = _chat(p) if chat is None else chat
        # the padded frequencies: signed along y and z, the half spectrum along x; odd factors vanish at a Nyquist index
        idx = [torch.arange(n[0] + 1, device="cuda")] + [torch.fft.fftfreq(2 * n[j], 0.5 / n[j], device="cuda", dtype=torch.float64).long() for j in range(1, d)]
        self.kp = [self._along(math.pi / self.W[j] * idx[j].double(), j) for j in range(d)]
        self.ko = [self._along(torch.where(idx[j].abs() == n[j], torch.zeros_like(idx[j]), idx[j]).double() * math.pi / self.W[j], j) for j in range(d)]
        for j in range(1, d):
            self.chat = self.chat.index_select(d - 1 - j, idx[j].abs())

    def _along(self, v, j):
        return v.view([-1 if self.d - 1 - j == q else 1 for q in range(self.d)])

    def kinetic(self, u, dt):
        return torch.fft.ifftn(torch.fft.fftn(u, dim=self.dims) * torch.exp(-1j * dt * self.sym), dim=self.dims)

    def kernel(self, ta, tb, axis=None):
        """The time-integrated multiplier over [ta, tb], or that of a fixed axis at one time."""
        p, d = self.p, self.d
        dt = tb - ta if axis is None else 1.0
        if p["kernel"] == "coulomb":
            return dt * self.chat
        M = np.zeros((3, 3))
        if axis is None:
            x, w = np.polynomial.legendre.leggauss(16)
            for xi, wi in zip(x, w):
                a = self.axis(0.5 * (ta + tb) + 0.5 * (tb - ta) * xi)
                M += 0.5 * (tb - ta) * wi * np.outer(a, a)
        else:
            M = np.outer(axis, axis)
        q = sum(M[j, j] * self.kp[j] ** 2 for j in range(d))
        for i in range(d):
            for j in range(i + 1, d):
                q = q + 2 * M[i, j] * self.ko[i] * self.ko[j]
        if d == 3:
            return -dt + 3.0 * q * self.chat
        return 1.5 * (q - M_n3(p) * dt * sum(k ** 2 for k in self.kp)) * self.chat

    def axis(self, t):
        c, s = math.cos(self.p["omega"] * t), math.sin(self.p["omega"] * t)
        a = self.p["dip_n"]
        return np.array([c * a[0] - s * a[1], s * a[0] + c * a[1], a[2]])

    def convolve(self, rho, K):
        n = self.p["n"]
        R = torch.fft.rfftn(rho, s=[2 * v for v in reversed(n)], dim=self.dims)
        out = torch.fft.irfftn(R * K, s=[2 * v for v in reversed(n)], dim=self.dims)
        return out[tuple(slice(0, v) for v in reversed(n))]

    def trap(self, ta, tb, gamma):
        """Time integral of the trap over [ta, tb] at the points of the rotating frame."""
        p, om, d = self.p, self.p["omega"], tb - ta
        X, Y = self.ax[0], self.ax[1]
        x, w = np.polynomial.legendre.leggauss(16)
        P = 0.0
        for xi, wi in zip(x, w):
            t, wt = 0.5 * (ta + tb) + 0.5 * d * xi, 0.5 * d * wi
            c, s = math.cos(om * t), math.sin(om * t)
            xr, yr = c * X + s * Y, -s * X + c * Y
            P = P + wt * 0.5 * (gamma[0] ** 2 * xr ** 2 + gamma[1] ** 2 * yr ** 2)
            if p.get("lat_amp"):
                P = P + wt * p["lat_amp"] * (torch.sin(p["lat_k"][0] * xr) ** 2 + torch.sin(p["lat_k"][1] * yr) ** 2)
        if self.d == 3:
            P = P + d * 0.5 * gamma[2] ** 2 * self.ax[2] ** 2
            if p.get("lat_amp"):
                P = P + d * p["lat_amp"] * torch.sin(p["lat_k"][2] * self.ax[2]) ** 2
        return P

    def step(self, u, ta, tb, gamma):
        p = self.p
        u = self.kinetic(u, (tb - ta) / 4)
        rho = u.real ** 2 + u.imag ** 2
        th = p["beta"] * (tb - ta) * rho + self.trap(ta, tb, gamma)
        if self.nl:
            th = th + p["lam"] * self.convolve(rho, self.kernel(ta, tb))
        return self.kinetic(u * torch.exp(-1j * th), (tb - ta) / 4)

    def run(self, u, steps, gammas=None):
        p, dt = self.p, self.p["dt"]
        w1 = 1.0 / (2.0 - 2.0 ** (1.0 / 3.0))
        w = (w1, 1.0 - 2.0 * w1, w1) if p.get("order") == 4 else (1.0,)
        for n in range(steps):
            t = n * dt
            for v in w:
                u = self.step(u, t, t + v * dt, p["gamma"] if gammas is None else gammas[n])
                t += v * dt
        return u


def M_n3(p):
    return p["dip_n"][2] ** 2


def _exact_ground(E, psi, case):
    """Backward-Euler gradient-flow steps, each solved by BiCGStab to rounding."""
    p, cell, dt = E.p, _cell(E.p), case["dt"]
    P = 1.0 / (1.0 / dt + 0.5 * E.sym)
    pre = lambda f: torch.fft.ifftn(torch.fft.fftn(f, dim=E.dims) * P, dim=E.dims)  # noqa: E731
    dot = lambda a, b: complex((a.conj() * b).sum())  # noqa: E731
    kd = [torch.where(k.abs() * E.W[j] / (2 * math.pi) > p["n"][j] / 2 - 0.5, torch.zeros_like(k), k) for j, k in enumerate(E.k)]
    psi = psi / math.sqrt(cell * float((psi.abs() ** 2).sum()))
    V = sum(0.5 * p["gamma"][j] ** 2 * E.ax[j] ** 2 for j in range(E.d))
    change = 0.0
    for _ in range(case["outer"]):
        rho = psi.abs() ** 2
        Wn = V + p["beta"] * rho + p["lam"] * E.convolve(rho, E.kernel(0, 0, E.axis(0.0)))

        def M(u):
            f = Wn * u
            if p["omega"]:
                F = torch.fft.fftn(u, dim=E.dims)
                dx, dy = (torch.fft.ifftn(1j * kd[j] * F, dim=E.dims) for j in (0, 1))
                f = f + 1j * p["omega"] * (E.ax[0] * dy - E.ax[1] * dx)
            return u + pre(f)

        b = pre(psi / dt)
        x = psi.clone()
        r = b - M(x)
        rh, bn = r.clone(), math.sqrt(dot(b, b).real)
        rho_, pv = dot(rh, r), r.clone()
        for _ in range(500):
            if math.sqrt(dot(r, r).real) <= 1e-14 * bn or rho_ == 0:
                break
            v = M(pv)
            al = rho_ / dot(rh, v)
            s = r - al * v
            t = M(s)
            tt = dot(t, t).real
            om = dot(t, s) / tt if tt > 0 else 0.0
            x = x + al * pv + om * s
            r = s - om * t
            if om == 0:
                break
            new = dot(rh, r)
            pv = r + (new / rho_) * (al / om) * (pv - om * v)
            rho_ = new
        x = x / math.sqrt(cell * float((x.abs() ** 2).sum()))
        change = float((x - psi).abs().max()) / dt
        psi = x
    return dict(psi=psi, change=change)


def _exact_observables(E, u, t):
    p, cell, N = E.p, _cell(E.p), math.prod(E.p["n"])
    d, ax, om = E.d, E.ax, p["omega"]
    rho = u.real ** 2 + u.imag ** 2
    S = lambda f: cell * float((f * rho).sum())  # noqa: E731
    c, s = math.cos(om * t), math.sin(om * t)
    X, Y = c * ax[0] + s * ax[1], -s * ax[0] + c * ax[1]
    W = 0.5 * (p["gamma"][0] ** 2 * X ** 2 + p["gamma"][1] ** 2 * Y ** 2) + (0.5 * p["gamma"][2] ** 2 * ax[2] ** 2 if d == 3 else 0.0)
    F = torch.fft.fftn(u, dim=E.dims)
    kd = [torch.where(k.abs() * E.W[j] / (2 * math.pi) > p["n"][j] / 2 - 0.5, torch.zeros_like(k), k) for j, k in enumerate(E.k)]
    dx, dy = (torch.fft.ifftn(1j * kd[j] * F, dim=E.dims) for j in (0, 1))
    o = dict(mass=S(1.0), e_kin=0.5 * cell / N * float((E.sym * F.abs() ** 2).sum()), e_pot=S(W), e_int=0.5 * p["beta"] * cell * float((rho ** 2).sum()),
             e_non=0.5 * p["lam"] * S(E.convolve(rho, E.kernel(0, 0, E.axis(t)))) if E.nl else 0.0,
             lz=cell * float((u.conj() * -1j * (ax[0] * dy - ax[1] * dx)).real.sum()))
    o["e_rot"] = -om * o["lz"]
    o["energy"] = o["e_kin"] + o["e_pot"] + o["e_int"] + o["e_non"] + o["e_rot"]
    o["xc"] = np.array([S(X), S(Y)] + ([S(ax[2])] if d == 3 else []))
    o["width"] = np.array([S(X ** 2), S(Y ** 2)] + ([S(ax[2] ** 2)] if d == 3 else []))
    return o


def exact(case, seed):
    p, psi, extra = _inputs(case, seed)
    if case["kind"] == "batch":
        chat, out = {}, []
        for q, x in zip(p, psi):
            if q["n"] not in chat:
                chat[q["n"]] = _chat(q)
            out.append(_Exact(q, chat[q["n"]]).run(x.to(torch.complex128), case["steps"]).reshape(-1))
        return torch.cat(out)
    E = _Exact(p)
    u = psi.to(torch.complex128)
    if case["kind"] == "ground":
        return _exact_ground(E, u, case)
    if case["kind"] == "observables":
        return _exact_observables(E, u, 0.3)
    if case["kind"] == "gradient":
        u.requires_grad_(True)
        gam = extra[0].double().cuda().requires_grad_(True)
        out = E.run(u, case["steps"], gam)
        z = _cell(p) * (out * extra[1].to(torch.complex128).conj()).sum()
        J = z.real ** 2 + z.imag ** 2
        g = torch.autograd.grad(J, (u, gam))
        return dict(out=out.detach(), objective=J.detach(), psi=g[0], gamma=g[1].cpu())
    out = E.run(u, case["steps"], extra)
    if p.get("renormalize"):
        # the library's option holds the mass of the call's start, which the exact step conserves
        return out
    return out.cpu().numpy() if case["kind"] == "host" else out

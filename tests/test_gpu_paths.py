"""The transform engine's routes against the oracle, and the adjoint sweep against its single steps.

Tile widths follow the number of tiles (a warp's worth of columns or lines on
small grids, 128-byte rows on large ones) and the plans follow the length, so
the grids below put every length on every axis, partly filled tiles included,
on both sides of the widths' limits. Bounds: tolerances.py, per step.
"""
import math

import numpy as np
import pytest

import oracle as O
from tolerances import assert_parity, bounds

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SQ = 1.0 / math.sqrt(2.0)


def _params(n, prec, kernel, **kw):
    dim = len(n)
    d = dict(dim=dim, n=n, lo=(-6.0, -5.0, -4.0)[:dim], hi=(6.0, 5.0, 4.0)[:dim], s=0.7, m=0.0, omega=0.7, beta=60.0,
             lam=20.0, dt=2e-3, kernel=kernel, dip_n=(SQ, 0.0, SQ) if kernel == "ddi3d" else (0.48, -0.36, 0.8),
             gamma=(1.0, 1.2, 1.7)[:dim], prec=prec)
    d.update(kw)
    return d


def _state(d, seed):
    p = O.params(d)
    X = O.coords(p)
    rng = np.random.default_rng(seed)
    e = sum(-0.5 * (X[j] - rng.uniform(-0.5, 0.5)) ** 2 + 1j * rng.uniform(-0.6, 0.6) * X[j] for j in range(p.dim))
    psi = np.exp(e) * (1.0 + 0.05 * rng.standard_normal(X[0].shape))
    return psi / math.sqrt(O.mass(psi, p))


GRIDS = [(8, 12), (12, 8), (16, 24), (24, 512), (512, 16), (48, 96), (96, 32), (192, 12), (32, 384), (384, 48), (128, 64),
         (64, 192), (8, 16, 12), (12, 48, 8), (16, 8, 96), (96, 16, 24), (24, 192, 12), (8, 12, 384), (64, 64, 48),
         (192, 24, 64), (128, 96, 32)]


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("n", GRIDS, ids=["x".join(map(str, n)) for n in GRIDS])
def test_every_length_on_every_axis(lib, n, prec):
    d = _params(n, prec, "ddi3d" if len(n) == 3 else "ddi2d")
    psi = _state(d, sum(n))
    ref = O.evolve(psi, O.params(d), 0.1, 2)
    plan = lib.Plan(d)
    x = plan.to_device(psi)
    plan.step(x, 0.1, 2)
    torch.cuda.synchronize()
    assert_parity(x.cpu().numpy().astype(np.complex128), ref, *bounds(prec, 2), f"{n} {prec}")


SWEEPS = {
    "2d": ((48, 32), "ddi2d", {}),
    "2d_none": ((32, 24), "none", {}),
    "2d_lattice": ((64, 48), "coulomb", dict(lat_amp=5.0, lat_k=(2.0, 1.5))),
    "3d": ((16, 24, 12), "ddi3d", {}),
}


@pytest.mark.parametrize("nsteps", [1, 5])
@pytest.mark.parametrize("name", sorted(SWEEPS))
def test_adjoint_sweep_matches_single_steps(lib, name, nsteps):
    """fse_adjoint_sweep against fse_step and fse_step_adjoint step by step, in
    float64: the same map with the kinetic half steps merged, so within the
    float64 bound of that many forward and backward steps."""
    n, kernel, kw = SWEEPS[name]
    d = _params(n, "f64", kernel, **kw)
    plan = lib.Plan(d)
    gam = 1.0 + 0.1 * np.random.default_rng(3).standard_normal((nsteps, len(n)))
    psi0 = plan.to_device(_state(d, 1))
    g = plan.to_device(_state(d, 2) * (1.0 + 0.5j))
    g_sweep = g.clone()
    dg_sweep = plan.adjoint_sweep(psi0, g_sweep, 0.2, gam)
    states, x = [psi0], psi0.clone()
    for k in range(nsteps - 1):
        plan.step(x, 0.2 + k * d["dt"], 1, gam[k:k + 1])
        states.append(x.clone())
    dg = np.zeros_like(gam)
    for k in range(nsteps - 1, -1, -1):
        dg[k] = plan.adjoint(states[k], g, 0.2 + k * d["dt"], gam[k], want_dgamma=True)[:len(n)]
    torch.cuda.synchronize()
    assert torch.equal(psi0, plan.to_device(_state(d, 1)))
    rel, elem = bounds("f64", 2 * nsteps)
    assert_parity(g_sweep.cpu().numpy(), g.cpu().numpy(), rel, elem, f"sweep {name}")
    assert np.max(np.abs(dg_sweep - dg)) <= 10 * rel * np.max(np.abs(dg))

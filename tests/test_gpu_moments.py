"""Moments, trap energy and trap gradients in boxes to one side of the origin and in
turned anisotropic traps, against sums in extended precision over the same field.

Every sum below is one of terms of one sign. A value passes at most 64 rounded
operations on its way (products, per-thread and per-block sums), so 64 units
of 2^-53 bound its relative error.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

EPS = 64 * 2.0**-53
LD = np.longdouble


def _axes(d):
    dim = d["dim"]
    return [(LD(d["lo"][j]) + LD((d["hi"][j] - d["lo"][j]) / d["n"][j]) * np.arange(d["n"][j]).astype(LD)).reshape(
        [-1 if dim - 1 - j == q else 1 for q in range(dim)]) for j in range(dim)]


def _params(n, prec, lo, hi, gamma, omega=0.0):
    return dict(dim=len(n), n=n, lo=lo, hi=hi, s=0.7, omega=omega, beta=30.0, lam=0.0, dt=1e-3, kernel="none", gamma=gamma, prec=prec)


def _cloud(d, centre, width):
    rng = np.random.default_rng(5)
    e = sum(-0.5 * ((x - c) / width) ** 2 + 0.3j * x for x, c in zip(_axes(d), centre))
    return (np.exp(e.astype(np.complex128)) * (1.0 + 0.2 * rng.standard_normal(e.shape))).astype(np.complex128)


BOXES = {
    "positive": ((128, 96), (0.0, 0.0), (16.0, 12.0), (0.5, 0.4), 0.2),
    "mixed": ((64, 128), (-20.0, 3.0), (-4.0, 19.0), (-5.0, 4.0), 0.4),
    "3d": ((48, 64, 32), (0.0, 2.0, -9.0), (8.0, 18.0, -1.0), (0.5, 3.0, -1.5), 0.3),
}


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("name", sorted(BOXES))
def test_moments_off_the_origin(lib, name, prec):
    n, lo, hi, centre, width = BOXES[name]
    d = _params(n, prec, lo, hi, (1.0, 1.2, 2.0)[:len(n)])
    plan = lib.Plan(d)
    psi = plan.to_device(_cloud(d, centre, width))
    o = plan.observables(psi, 0.0)
    u = psi.cpu().numpy()
    rho = u.real.astype(LD) ** 2 + u.imag.astype(LD) ** 2
    cell = math.prod((h - l) / m for l, h, m in zip(lo, hi, n))
    ax = _axes(d)
    want = {"mass": rho, "e_int": 15 * rho * rho, "e_pot": sum(LD(0.5) * LD(g) ** 2 * x * x for g, x in zip(d["gamma"], ax)) * rho}
    got = {k: o[k] for k in want}
    for j, x in enumerate(ax):
        want[f"xc{j}"], got[f"xc{j}"] = x * rho, o["xc"][j]
        want[f"width{j}"], got[f"width{j}"] = x * x * rho, o["width"][j]
    for k, f in want.items():
        ref = float(cell * np.sum(f))
        assert abs(got[k] - ref) <= EPS * abs(ref), (k, got[k], ref, abs(got[k] / ref - 1))


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("gamma", [(1.0, 1.0), (1.0, 1.9), (2.1, 1.0), (100.0, 1.0), (1.0, 0.0)])
def test_trap_energy_in_a_turned_frame(lib, gamma, prec):
    t, omega = 1.0, 0.7
    d = _params((128, 128), prec, (-8.0, -8.0), (8.0, 8.0), gamma, omega)
    c, s = math.cos(omega * t), math.sin(omega * t)
    plan = lib.Plan(d)
    psi = plan.to_device(_cloud(d, (-5 * s, 5 * c), 0.3))  # along the Y axis
    u = psi.cpu().numpy()
    rho = u.real.astype(LD) ** 2 + u.imag.astype(LD) ** 2
    x, y = _axes(d)
    X, Y = LD(c) * x + LD(s) * y, LD(c) * y - LD(s) * x
    ref = float(LD(1 / 64) * np.sum(LD(0.5) * (LD(gamma[0]) ** 2 * X * X + LD(gamma[1]) ** 2 * Y * Y) * rho))
    # points: X is off by 2 (|c x| + |s y|) / |X| = 36 units, its square by twice that, and 64 for the
    # sum; moments (up to 2 : 1): 36 units for terms that add up to four times the energy
    assert abs(plan.observables(psi, t)["e_pot"] - ref) <= 144 * 2.0**-53 * ref


@pytest.mark.parametrize("sweep", [False, True])
@pytest.mark.parametrize("name", sorted(BOXES))
def test_trap_gradient_off_the_origin(lib, name, sweep):
    """With a step of 1e-18 the kinetic factors are 1 to 1e-15 and the phase vanishes:
    dJ/dgamma_v = gamma_v dt sum_x x_v^2 Im(conj(g) psi), one-signed for g = -i psi."""
    n, lo, hi, centre, width = BOXES[name]
    d = dict(_params(n, "f64", lo, hi, (1.0, 1.2, 2.0)[:len(n)]), beta=0.0, dt=1e-18)
    plan = lib.Plan(d)
    psi = plan.to_device(_cloud(d, centre, width))
    g = psi * -1j
    if sweep:
        dg = plan.adjoint_sweep(psi, g, 0.0, np.array([d["gamma"]]))[0]
    else:
        dg = plan.adjoint(psi, g, 0.0, None, want_dgamma=True)
    u = psi.cpu().numpy()
    rho = u.real.astype(LD) ** 2 + u.imag.astype(LD) ** 2
    for v, x in enumerate(_axes(d)):
        ref = float(LD(d["gamma"][v]) * LD(1e-18) * np.sum(x * x * rho))
        assert abs(dg[v] - ref) <= EPS * ref, (v, dg[v], ref, dg[v] / ref - 1)

"""Calls on long axes and wide tiles, and in float32, against the 64-bit restatement of the timed cases.

The grids put 128 to 512 points on y and z of 3D grids with tiles enough for
the wide column passes, their gathered tails included, and 384 and 512 with few
for the narrow ones; the ground states have more than one tile per SM, oblong
sides and lengths with factors of three.
"""
import numpy as np
import pytest

import perf.cases as cases
from tolerances import assert_parity, bounds

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GRIDS = [(8, 512, 16), (16, 8, 512), (64, 64, 512), (64, 512, 64), (48, 64, 384), (64, 384, 48), (32, 256, 64), (64, 32, 256),
         (32, 128, 128), (96, 192, 96)]


def _np(x):
    return x.detach().cpu().numpy().astype(np.complex128)


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("n", GRIDS, ids=["x".join(map(str, n)) for n in GRIDS])
def test_long_axes(lib, n, prec):
    case = dict(kind="step", nx=n[0], ny=n[1], nz=n[2], prec=prec, kernel="ddi3d", steps=1)
    got = cases.run(cases.prepare(case, 3))
    assert_parity(_np(got), _np(cases.exact(case, 3)), *bounds(prec, 1), f"{n} {prec}")


@pytest.mark.parametrize("n", [(64, 48), (192, 96), (256, 256)], ids=["64x48", "192x96", "256x256"])
def test_gradient_in_float32(lib, n):
    """Forward steps, their states again, and as many backward steps: three per step."""
    case = dict(kind="gradient", nx=n[0], ny=n[1], prec="f32", steps=7)
    got, ref = cases.run(cases.prepare(case, 4)), cases.exact(case, 4)
    rel, elem = bounds("f32", 3 * 7)
    assert_parity(_np(got["out"]), _np(ref["out"]), rel, elem, "out")
    assert_parity(_np(got["psi"]), _np(ref["psi"]), rel, elem, "dJ/dpsi")
    g, r = got["gamma"].double().cpu().numpy(), ref["gamma"].double().cpu().numpy()
    assert np.max(np.abs(g - r)) <= 10 * rel * np.max(np.abs(r))


@pytest.mark.parametrize("prec,tol", [("f64", 1e-12), ("f32", 1e-6)])
@pytest.mark.parametrize("n,omega", [((512, 512), 0.0), ((384, 192), 0.3), ((192, 384), 0.0), ((96, 256), 0.3), ((48, 96, 32), 0.3),
                                     ((64, 64, 64), 0.0)])
def test_ground_state_step(lib, n, omega, prec, tol):
    """One implicit step: with dt = 1e-3 the preconditioned operator is 1 plus less than one
    half, so that a residual of tol leaves an error of at most twice that; float32
    adds the rounding of a dozen passes."""
    case = dict(kind="ground", nx=n[0], ny=n[1], nz=n[2] if len(n) == 3 else 0, omega=omega, s=1.0, dt=1e-3, outer=1, prec=prec)
    st = cases.prepare(case, 5)
    st["gs"]["inner_tol"] = tol
    got, ref = cases.run(st), cases.exact(case, 5)
    bound = 4e-12 if prec == "f64" else 6e-6
    assert_parity(_np(got["psi"]), _np(ref["psi"]), bound, 2 * bound, f"{n} {prec} omega {omega}")


def test_sweep_longer_than_a_group_of_gradients(lib):
    """The trap gradients of a sweep are summed 512 steps at a time at most: 1100 steps in one
    call against eleven calls of 100, within the float64 bound of that many steps."""
    T, part = 1100, 100
    d = dict(dim=2, n=(8, 8), lo=(-4.0, -4.0), hi=(4.0, 4.0), s=0.7, omega=0.4, beta=20.0, lam=0.0, dt=1e-3, kernel="none", gamma=(1.0, 1.3), prec="f64")
    plan = lib.Plan(d)
    rng = np.random.default_rng(0)
    gam = 1.0 + 0.1 * rng.standard_normal((T, 2))
    psi, g0 = (plan.to_device(rng.standard_normal((8, 8)) + 1j * rng.standard_normal((8, 8))) for _ in range(2))
    g = g0.clone()
    dg = plan.adjoint_sweep(psi, g, 0.0, gam)
    states, x = [psi], psi.clone()
    for s in range(0, T - part, part):
        plan.step(x, s * d["dt"], part, gam[s:s + part])
        states.append(x.clone())
    h, dh = g0.clone(), np.zeros_like(gam)
    for k in range(len(states) - 1, -1, -1):
        dh[part * k:part * k + part] = plan.adjoint_sweep(states[k], h, part * k * d["dt"], gam[part * k:part * k + part])
    rel, elem = bounds("f64", 2 * T)
    assert_parity(_np(g), _np(h), rel, elem, "cotangent")
    assert np.max(np.abs(dg - dh)) <= 10 * rel * np.max(np.abs(dh))

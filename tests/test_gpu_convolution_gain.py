"""Gains of the float32 density transforms that act on many modes alike."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _plan(lib, n, prec="f32", **kw):
    d = dict(dim=3, n=n, lo=(-8.0,) * 3, hi=(8.0,) * 3, s=0.7, omega=0.6, beta=100.0, lam=10.0, dt=1e-3, kernel="ddi3d",
             gamma=(1.0, 1.2, 2.0), dip_n=(0.0, 0.0, 0.0), prec=prec)
    d.update(kw)
    return lib.Plan(d)


@pytest.mark.parametrize("n", [(64, 64, 64), (64, 128, 64), (128, 128, 128)])
def test_round_trip_of_a_white_density(lib, n):
    """With a zero dipole axis the kernel is -1, so the field energy is -lam / beta times
    the contact energy, up to the mean gain of six padded transforms over a white
    spectrum. Roundings of values average out (3e-7 over the root of 2^18 points);
    the heads of the twiddle tables add up to 3.3e-9 at most for these lengths
    (their pairs' mean errors, plan by plan); twice that and the values is 8e-9.
    The 16th roots rounded alone, 2.9e-8 short, would be -2.9e-8 to -5.7e-8."""
    plan = _plan(lib, n)
    rng = np.random.default_rng(1)
    psi = plan.to_device(rng.standard_normal(n[::-1]) + 1j * rng.standard_normal(n[::-1]))
    o = plan.observables(psi, 0.0)
    gain = o["e_non"] / (-0.1 * o["e_int"]) - 1
    print(f"{n}: {gain:.2e}")
    assert abs(gain) <= 8e-9


@pytest.mark.parametrize("n", [(64, 32, 48), (96, 64, 64), (32, 48, 128)])
def test_dipolar_terms_are_rounded_alike(lib, n):
    """N has one factor of three, so that -1 / (8 N) is 2.98e-8 off as a float. Over a
    white spectrum the dipolar kernel's two terms nearly cancel, and with them every
    gain that they share; an error of the first term alone stays whole. A quarter of it
    is the bound."""
    axis = dict(dip_n=(0.6, 0.0, 0.8))
    rng = np.random.default_rng(2)
    psi = (rng.standard_normal(n[::-1]) + 1j * rng.standard_normal(n[::-1])).astype(np.complex64)
    a, b = _plan(lib, n, **axis), _plan(lib, n, "f64", **axis)
    oa, ob = a.observables(a.to_device(psi), 0.0), b.observables(b.to_device(psi), 0.0)
    err = (oa["e_non"] - ob["e_non"]) / (0.1 * ob["e_int"])
    print(f"{n}: {err:.2e}, kernel mean {ob['e_non'] / (0.1 * ob['e_int']):.2f}")
    assert abs(err) <= 2.98e-8 / 4


@pytest.mark.parametrize("n", [(64, 64, 64), (48, 64, 96)])
def test_dipolar_factors_of_a_column_have_no_common_error(lib, n):
    """Field energies of smooth clouds, a few dozen columns of modes, in units of the
    kernel's two terms. One rounding of a value at most 2^-25 in every mode averages
    out to about 3e-9 over a hundred columns; C^, the factor in rows and the twiddles'
    heads give as much each: 6e-9 together, 1e-8 the bound on the root mean square of
    eight clouds. Columns whose factors are rounded product by product are at 2e-8."""
    axis = dict(dip_n=(0.5**0.5, 0.0, 0.5**0.5))
    a, b = _plan(lib, n, **axis), _plan(lib, n, "f64", **axis)
    rng = np.random.default_rng(4)
    err = []
    for _ in range(8):
        e = 0.0
        for j in range(3):
            x = (-8.0 + 16.0 / n[j] * np.arange(n[j])).reshape([-1 if 2 - j == q else 1 for q in range(3)])
            e = e - 0.5 * ((x - rng.uniform(-0.5, 0.5)) / rng.uniform(0.7, 1.4)) ** 2 + 1j * rng.uniform(-0.6, 0.6) * x
        psi = np.exp(e).astype(np.complex64)
        oa, ob = a.observables(a.to_device(psi), 0.3), b.observables(b.to_device(psi), 0.3)
        err.append((oa["e_non"] - ob["e_non"]) / (0.1 * ob["e_int"]))
    print(f"{n}: {np.sqrt(np.mean(np.square(err))):.2e}")
    assert np.sqrt(np.mean(np.square(err))) <= 1e-8

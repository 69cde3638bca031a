"""Sums over float32 fields (observables, trap gradients) follow powers of two exactly.

The products are split and added as sums of three floats after a scaling by a
power of two of each thread's largest value; the transforms of a field times
2^k are those of the field times 2^k, bit for bit, as long as nothing leaves
the normal range (2^-30 to 2^30 here, with 2^-60 to 2^60 for densities). So
quadratic sums follow 4^k and the field energy 16^k up to the rounding of
the float64 block sums, which scale exactly too: 1e-15 covers the divisions.
"""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# tiles, remainders and lines shorter than a warp; lengths of every kind of plan
SHAPES = [(8, 12), (96, 64), (384, 16), (512, 24), (48, 192), (32, 24, 16), (64, 96, 12), (16, 48, 128)]


def _plan(lib, n, **kw):
    dim = len(n)
    return lib.Plan(dict(dim=dim, n=n, lo=(-6.0, -5.0, -4.0)[:dim], hi=(6.0, 5.0, 4.0)[:dim], s=0.7, omega=0.6,
                         beta=0.0, lam=8.0, dt=1e-3, kernel="coulomb", gamma=(1.0, 1.4, 1.2)[:dim], prec="f32", **kw))


def _field(n, seed=3):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(np.complex64)


@pytest.mark.parametrize("n", SHAPES)
@pytest.mark.parametrize("k", [-30, -7, 14])
def test_observable_sums_follow_powers_of_two(lib, n, k):
    plan = _plan(lib, n)
    psi = plan.to_device(_field(n))
    a, b = plan.observables(psi, 0.3), plan.observables(psi * 2.0**k, 0.3)
    for key, p in (("mass", 2), ("e_kin", 2), ("lz", 2), ("e_non", 4)):
        assert abs(b[key] * 2.0 ** (-p * k) - a[key]) <= 1e-15 * abs(a[key]), (key, a[key], b[key])
        assert a[key] != 0.0


def test_observables_of_zero_are_zero_and_nan_is_refused(lib):
    plan = _plan(lib, (64, 48))
    psi = plan.to_device(np.zeros((64, 48)))
    z = plan.observables(psi, 0.0)
    assert all(z[k] == 0.0 for k in ("mass", "e_kin", "lz", "e_non", "energy"))
    psi.view(-1)[7] = complex(float("nan"), 0.0)
    with pytest.raises(lib.FseError):
        plan.observables(psi, 0.0)

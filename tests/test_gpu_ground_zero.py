"""A gradient-flow iterate that vanishes is reported, and returned as it is."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_vanishing_iterate_is_left_alone(lib):
    """A constant field in a flat potential of 2^32 per unit step: every value of the
    solve is a power of two, and one BiCGStab iteration takes 1/2 to 1/2 - 2^31 / 2^32 = 0."""
    plan = lib.Plan(dict(dim=2, n=(16, 16), lo=(-1.0, -1.0), hi=(1.0, 1.0), s=1.0, omega=0.0, beta=2.0**34, lam=0.0,
                         dt=1e-3, kernel="none", gamma=(0.0, 0.0), prec="f32"))
    x = plan.to_device(np.full((16, 16), 0.5))
    with pytest.raises(lib.FseError, match="zero field"):
        plan.ground_state(x, dt=1.0, max_outer=1)
    assert torch.equal(x, torch.zeros_like(x))

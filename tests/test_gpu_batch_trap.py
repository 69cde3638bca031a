"""Batched runs over more steps than one table of trap coefficients holds (64), against single runs."""
import numpy as np
import pytest

from test_gpu_batch import _psi, _runs
from tolerances import assert_parity, bounds

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("steps", [1, 64, 65, 130])
def test_batch_over_trap_tables(lib, steps):
    runs = _runs()[:5]
    for k, d in enumerate(runs):
        d.update(gamma=(1.0, 1.5 + 0.2 * k), dt=2e-3 * (1 + k))  # strongly time-dependent, another step each
    psis = [_psi(d, k) for k, d in enumerate(runs)]
    b = lib.Batch(runs)
    xs = b.to_device(psis)
    b.step(xs, 0.4, steps)
    for d, p0, x in zip(runs, psis, xs):
        plan = lib.Plan(d)
        y = plan.to_device(p0)
        plan.step(y, 0.4, steps)
        torch.cuda.synchronize()
        assert_parity(x.cpu().numpy().astype(np.complex128), y.cpu().numpy().astype(np.complex128),
                      *bounds("f32", steps), f"{d['n']} over {steps} steps")

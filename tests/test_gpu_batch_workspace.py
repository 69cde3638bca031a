"""Captured step sequences of a batch: another workspace, and more step counts than are kept."""
import pytest

from test_gpu_batch import _psi, _runs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _fresh(lib, runs, psis, calls):
    b = lib.Batch(runs)
    xs = b.to_device(psis)
    for t, n in calls:
        b.step(xs, t, n)
    torch.cuda.synchronize()
    return xs


def test_step_after_another_workspace(lib):
    """The same step count before and after: the later calls work in the second
    workspace alone, and the first one stays as it was left."""
    runs = _runs()
    psis = [_psi(d, 30 + k) for k, d in enumerate(runs)]
    ref = _fresh(lib, runs, psis, [(0.2, 3)])
    b = lib.Batch(runs)
    xs = b.to_device(psis)
    b.step(xs, 0.2, 3)
    torch.cuda.synchronize()
    first = b.ws
    first.fill_(0xA5)
    b.ws = torch.empty(b.ws_bytes, dtype=torch.uint8, device=b.device)
    lib.fse_batch_set_workspace(b.handle, b.ws, b.ws_bytes)
    lib.fse_batch_precompute(b.handle)
    for rep in range(2):
        ys = b.to_device(psis)
        b.step(ys, 0.2, 3)
        torch.cuda.synchronize()
        for x, y in zip(ref, ys):
            assert torch.equal(x, y)
    assert bool((first == 0xA5).all())


def test_more_step_counts_than_kept(lib):
    """Forty step counts, each captured, dropped and (the first ones) captured again."""
    runs = _runs()[:3]
    psis = [_psi(d, 40 + k) for k, d in enumerate(runs)]
    b = lib.Batch(runs)
    for rep in range(2):
        for n in list(range(1, 41)) + [1, 2]:
            ys = b.to_device(psis)
            b.step(ys, 0.1, n)
            if n in (1, 2, 17, 40):
                for x, y in zip(_fresh(lib, runs, psis, [(0.1, n)]), ys):
                    assert torch.equal(x, y)

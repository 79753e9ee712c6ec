"""Failure path of a launch of several steps: LBM_FLAG_TEST_STALL starts one
tile's count of finished items one short (a flag that nothing sets) and sets the
limit of the waits to 0.1 s.  The waits for it run out, every block ends, LBM_DEVFLAG_TIMEOUT is set,
lbm_diag reports LBM_ERR_TIMEOUT and the device stays usable.  No fault, no trap,
no hang is provoked."""
import ctypes

import pytest

from paper_2112_08479_gb300 import lbm

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _params(shape, model, flags):
    return lbm.lock_exchange(*shape, H=shape[2], x0=shape[0] // 2, u_b=0.03, Re=2000.0, model=model,
                             flags=flags)


@pytest.mark.parametrize("model", ["bgk", "cumulant"])
@pytest.mark.parametrize("shape,steps", [
    ((128, 48, 64), 24),        # one step slot
    ((300, 12, 600), 8),        # a wave of four
    ((2048, 128, 24), 6),       # slabs along x, two sweeps
])
def test_a_step_that_never_counts_gives_up(shape, steps, model):
    p = _params(shape, model, lbm.LBM_FLAG_TEST_STALL)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert lbm.lbm_step_plan(p.c(), sms, steps)["steps"] == steps
    lat = lbm.Lattice(p)
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    e[0].record()
    lat.step(steps)
    e[1].record()
    lat.sync()                                   # ends by itself, without an error
    assert 100.0 <= e[0].elapsed_time(e[1]) < 1000.0
    d = lbm.lbm_diagnostics()
    assert lbm.load().lbm_diag(lat.ctx, ctypes.byref(d)) == lbm.LBM_ERR_TIMEOUT
    assert d.flags & lbm.LBM_DEVFLAG_TIMEOUT
    del lat
    # the device goes on, in the same shape of launch
    a, b = (lbm.Lattice(_params(shape, model, 0)) for _ in range(2))
    a.step(steps)
    for _ in range(steps):
        b.step(1)
    assert torch.equal(a.get_state(), b.get_state())
    assert a.diag()["flags"] == 0

"""Calls whose steps share a launch, with the route asserted (lbm_step_plan on this
device), against the same steps launched one by one, bit for bit: one step slot
with wraps and one tile per plane, waves, few planes, several sweeps over several
slabs with and without periodic ends, and a call captured in a graph."""
import pytest

from paper_2112_08479_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PX, PZ = lbm.LBM_FLAG_PERIODIC_X, lbm.LBM_FLAG_PERIODIC_Z
KINDS = [(lbm.LBM_BGK_SMAG_Q19, lbm.LBM_SCALAR_Q7), (lbm.LBM_BGK_SMAG_Q19, lbm.LBM_SCALAR_Q6),
         (lbm.LBM_CUMULANT_Q27, lbm.LBM_SCALAR_Q7)]
W27 = [8 / 27] + [2 / 27] * 6 + [1 / 54] * 12 + [1 / 216] * 8
WEIGHTS = {19: [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, 27: W27}
SCALARS = {7: [1 / 4] + [1 / 8] * 6, 6: [1 / 6] * 6}


def _params(shape, kind, flags):
    nx, ny, nz = shape
    return lbm.Params(nx, ny, nz, model=kind[0], scalar=kind[1], flags=flags, nu=2e-3, D=3e-3,
                      gprime=1e-4, eg=(0.3, -0.4, -0.866), x0=0, H=nz)


def _plan(p, steps):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return lbm.lbm_step_plan(p.c(), sms, steps)


def _state(p):
    s = inputs.torch_uniform((p.Q + p.NS, p.N), 7, 0.02)
    s *= torch.tensor(WEIGHTS[p.Q] + SCALARS[p.NS], device="cuda").view(-1, 1)
    return s


def _check(p, steps, lead=0):
    s = _state(p)
    a, b = lbm.Lattice(p, device="cuda"), lbm.Lattice(p, device="cuda")
    a.set_state(s)
    b.set_state(s)
    for _ in range(lead):          # an odd lead starts the call on an odd step
        a.step(1)
        b.step(1)
    a.step(steps)
    for _ in range(steps):
        b.step(1)
    assert a.step_count == b.step_count == steps + lead
    a.get_state(s)
    assert torch.equal(s, b.get_state())
    assert a.diag()["flags"] == 0


@pytest.mark.parametrize("flags", [0, PX, PZ, PX | PZ])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape", [(64, 66, 66), (333, 17, 60), (35, 3, 1500), (40, 1, 4300)])
def test_one_slot(shape, kind, flags):
    p = _params(shape, kind, flags)
    pl = _plan(p, 25)
    assert (pl["steps"], pl["slots"]) == (25, 1)
    assert shape[1] > 3 or pl["tiles"] == 1
    _check(p, 25)
    _check(p, 24, lead=1)


@pytest.mark.parametrize("flags", [0, PX])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape,steps,slots", [
    ((300, 12, 600), 9, 4), ((64, 3, 5500), 8, 4),
    ((1000, 500, 4), 4, 2),                                  # few planes
])
def test_waves(shape, steps, slots, kind, flags):
    p = _params(shape, kind, flags)
    pl = _plan(p, steps)
    assert pl["slots"] == slots and pl["sweeps"] >= 2
    _check(p, steps, lead=steps % 2)


@pytest.mark.parametrize("flags", [0, PX])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape,steps", [((2048, 128, 24), 7), ((2500, 150, 40), 9)])
def test_sweeps_over_slabs(shape, steps, kind, flags):
    """The first slab of a sweep follows the last slab of the sweep before."""
    p = _params(shape, kind, flags)
    pl = _plan(p, steps)
    assert pl["sweeps"] >= 2 and pl["slabs"] >= 2 and pl["slots"] == 3
    _check(p, steps, lead=1)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape,steps", [((65, 33, 70), 25), ((300, 12, 600), 9)])
def test_captured(shape, steps, kind):
    p = _params(shape, kind, PX)
    assert _plan(p, steps)["steps"] >= 8
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        s = _state(p)
        ref = lbm.Lattice(p, stream=st)
        ref.set_state(s)
        for _ in range(2 * steps):
            ref.step(1)
        want = ref.get_state()
        lat = lbm.Lattice(p, stream=st)
        out = torch.empty_like(want)
        lat.step(steps)                     # first call outside the capture
        lat.set_state(s)
        st.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            lat.step(steps)
            lat.step(steps)
            lat.get_state(out)
        for _ in range(2):
            lat.set_state(s)
            g.replay()
            st.synchronize()
            assert torch.equal(out, want)
            out.zero_()
        assert lat.diag()["flags"] == 0

"""Many steps in one launch (lbm_step with nsteps > 1) against the same steps
launched one by one: the same arithmetic per node, so the states agree bit for
bit, whatever order the rows are taken in.  Boxes whose state fits the L2 (one
step slot), tall boxes (a wave of up to four slots) and boxes with wide planes
(slabs along x), with odd extents, partial tiles and wraps."""
import pytest

from paper_2112_08479_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PX, PZ = lbm.LBM_FLAG_PERIODIC_X, lbm.LBM_FLAG_PERIODIC_Z
KINDS = [(lbm.LBM_BGK_SMAG_Q19, lbm.LBM_SCALAR_Q7), (lbm.LBM_BGK_SMAG_Q19, lbm.LBM_SCALAR_Q6),
         (lbm.LBM_CUMULANT_Q27, lbm.LBM_SCALAR_Q7)]
W27 = [8 / 27] + [2 / 27] * 6 + [1 / 54] * 12 + [1 / 216] * 8
WEIGHTS = {19: [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, 27: W27}
SCALARS = {7: [1 / 4] + [1 / 8] * 6, 6: [1 / 6] * 6, 27: W27}


def _check(shape, kind, flags, steps, lead):
    nx, ny, nz = shape
    p = lbm.Params(nx, ny, nz, model=kind[0], scalar=kind[1], flags=flags, nu=2e-3, D=3e-3,
                   gprime=1e-4, eg=(0.3, -0.4, -0.866), x0=0, H=nz)
    a, b = lbm.Lattice(p, device="cuda"), lbm.Lattice(p, device="cuda")
    s = inputs.torch_uniform((p.Q + p.NS, p.N), 7, 0.02)
    s *= torch.tensor(WEIGHTS[p.Q] + SCALARS[p.NS], device="cuda").view(-1, 1)
    a.set_state(s)
    b.set_state(s)
    if lead:                       # start on an odd step
        a.step(1)
        b.step(1)
    a.step(steps)
    for _ in range(steps):
        b.step(1)
    assert a.step_count == b.step_count == steps + lead
    s = a.get_state(s)
    assert torch.equal(s, b.get_state())
    assert a.diag()["flags"] == 0


@pytest.mark.parametrize("flags", [0, PX, PZ])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape", [(1, 40, 40), (33, 5, 7), (64, 1, 64), (128, 8, 16),
                                   (200, 7, 19), (333, 17, 9), (256, 32, 40)])
def test_small_boxes(shape, kind, flags):
    _check(shape, kind, flags, 7, 0)
    _check(shape, kind, flags, 4, 1)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape,steps", [((300, 12, 600), 9), ((130, 5, 1500), 4),
                                         ((1000, 61, 90), 6), ((1024, 64, 64), 3),
                                         ((2048, 128, 24), 5), ((2500, 90, 20), 2),
                                         ((700, 200, 3), 5)])
def test_waves_and_slabs(shape, steps, kind):
    _check(shape, kind, 0, steps, steps % 2)
    _check(shape, kind, PX, steps, 0)


@pytest.mark.parametrize("flags", [0, PX, PZ])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape", [(3, 66, 66), (65, 33, 70), (129, 41, 37), (256, 32, 48)])
def test_boxes_in_l2(shape, kind, flags):
    """Enough rows and steps for one slot, with an odd count from either parity."""
    _check(shape, kind, flags, 25, 0)
    _check(shape, kind, flags, 24, 1)


@pytest.mark.parametrize("steps", [2, 3, 4, 5, 6, 7, 11])
@pytest.mark.parametrize("kind", KINDS)
def test_whole_sweeps_and_the_rest(kind, steps):
    _check((513, 61, 70), kind, 0, steps, steps % 2)

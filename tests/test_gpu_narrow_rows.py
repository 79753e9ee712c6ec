"""FP32 cumulant rows that leave half of a segment's pairs idle step one node per
thread: the same bits as pairs.  A box with periodic x ends equals itself repeated
along x, and the repeated rows are long enough for the pair kernel."""
import pytest

from paper_2112_08479_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PX, PZ = lbm.LBM_FLAG_PERIODIC_X, lbm.LBM_FLAG_PERIODIC_Z


def _one_node(nx):
    return (nx + 31) // 32 in (1, 3)


@pytest.mark.parametrize("flags", [PX, PX | PZ])
@pytest.mark.parametrize("steps", [1, 3, 30])
@pytest.mark.parametrize("nx,times", [(1, 64), (2, 20), (31, 2), (32, 2), (65, 2), (66, 3), (96, 2)])
def test_box_equals_itself_repeated(nx, times, steps, flags):
    assert _one_node(nx) and not _one_node(nx * times)
    ny, nz = 5, 7
    par = dict(model=lbm.LBM_CUMULANT_Q27, flags=flags, nu=2e-3, D=3e-3, gprime=1e-4,
               eg=(0.3, -0.4, -0.866), x0=0, H=nz)
    p, q = lbm.Params(nx, ny, nz, **par), lbm.Params(nx * times, ny, nz, **par)
    rows = p.Q + p.NS
    s = inputs.torch_uniform((rows, p.N), 5, 2e-3).view(rows, nz, ny, nx)
    a, b = lbm.Lattice(p, device="cuda"), lbm.Lattice(q, device="cuda")
    a.set_state(s.reshape(rows, -1).contiguous())
    b.set_state(s.repeat(1, 1, 1, times).view(rows, -1))
    for _ in range(steps):
        a.step(1)
        b.step(1)
        if steps > 3:
            continue
        got = b.get_state().view(rows, nz, ny, nx * times)
        assert torch.equal(got, a.get_state().view(rows, nz, ny, nx).repeat(1, 1, 1, times))
    got = b.get_state().view(rows, nz, ny, nx * times)
    assert torch.equal(got, a.get_state().view(rows, nz, ny, nx).repeat(1, 1, 1, times))
    assert a.diag()["flags"] == 0

"""FP32 boxes past 32-bit element offsets ((Q + NS) N >= 2^32) against the same box
cut into two x-slabs, whose offsets fit 32 bits: after even and odd steps every
population of the box equals the slabs' bit for bit (include/lbm.h, x-slab
decomposition), as it does between the two- and the one-node kernel."""
import pytest

from paper_2112_08479_gb300 import lbm, slab

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _swap(a, b):
    """The faces of two touching slabs, x = nx - 1 of a and x = 0 of b."""
    n = lbm.lbm_halo_bytes(a.params.c())
    fa, fb = (torch.empty(n, dtype=torch.uint8, device="cuda") for _ in range(2))
    a.halo_pack(1, fa)
    b.halo_pack(0, fb)
    a.halo_unpack(1, fb)
    b.halo_unpack(0, fa)


@pytest.mark.parametrize("flags", [0, lbm.LBM_FLAG_ONE_NODE])
@pytest.mark.parametrize("model", ["bgk", "cumulant"])
def test_wide_box_equals_its_slabs(model, flags):
    nx, ny, nz = 2048, 256, 320
    p = lbm.lock_exchange(nx, ny, nz, H=nz, x0=nz, u_b=0.03, Re=30000.0, model=model, flags=flags)
    p.gprime = 1e-3
    parts = [slab.slab_params(p, r, 2) for r in range(2)]
    rows = p.Q + p.NS
    assert rows * p.N >= 2**32 and all(rows * q.N < 2**32 for q in parts)
    g = torch.Generator(device="cuda")
    g.manual_seed(31)
    s = torch.empty(rows, nz, ny, nx, device="cuda")
    for r in range(rows):
        s[r].uniform_(-1e-3, 1e-3, generator=g)
    box = lbm.Lattice(p, device="cuda")
    box.set_state(s.view(rows, -1))
    lats = []
    for q in parts:
        lat = lbm.Lattice(q, device="cuda")
        lat.set_state(s[..., q.x_offset:q.x_offset + q.nx].contiguous().view(rows, -1))
        lats.append(lat)
    for step in range(3):
        box.step(1)
        for lat in lats:
            lat.step(1)
        _swap(*lats)
        box.get_state(s.view(rows, -1))
        for q, lat in zip(parts, lats):
            got = lat.get_state().view(rows, nz, ny, q.nx)
            for r in range(rows):
                assert torch.equal(got[r], s[r, :, :, q.x_offset:q.x_offset + q.nx]), (step, q.x_offset, r)
            del got
    assert box.diag()["flags"] == 0

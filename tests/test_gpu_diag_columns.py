"""Diagnostics with several threads per column against FP64 sums over the state:
spans shorter than the group, remainders, blocks of columns cut short, and a box
with enough columns for the other group size of the 27-velocity odd gather."""
import numpy as np
import pytest

from paper_2112_08479_gb300 import inputs, lbm

from helpers import weights, wscalar

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

KINDS = [(lbm.LBM_BGK_SMAG_Q19, lbm.LBM_SCALAR_Q7), (lbm.LBM_BGK_SMAG_Q19, lbm.LBM_SCALAR_Q6),
         (lbm.LBM_CUMULANT_Q27, lbm.LBM_SCALAR_Q7), (lbm.LBM_CUMULANT_Q27, lbm.LBM_SCALAR_Q27)]


@pytest.mark.parametrize("odd", [False, True])
@pytest.mark.parametrize("storage", [lbm.LBM_FP32, lbm.LBM_FP16S])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape", [(1, 1, 2), (127, 3, 2), (129, 4, 3), (200, 5, 2), (64, 11, 4),
                                   (2048, 2, 128)])
def test_diagnostics_against_fp64(shape, kind, storage, odd):
    nx, ny, nz = shape
    p = lbm.Params(nx, ny, nz, model=kind[0], scalar=kind[1], storage=storage, nu=2e-3, D=3e-3,
                   gprime=1e-4, sc_t=0.7, x0=nx // 2, H=nz)
    w = weights(p.model)
    f = w[:, None] * inputs.uniform((p.Q, p.N), 3, 0.05)
    chi = 0.5 * (1.0 + inputs.uniform(p.N, 4, 1.0))
    phi = wscalar(p)[:, None] * (chi * (1.0 + inputs.uniform((p.NS, p.N), 5, 0.05)) - 1.0)
    lat = lbm.Lattice(p)
    lat.set_state(torch.from_numpy(np.concatenate([f, phi]).astype(np.float32)).cuda())
    if odd:
        lat.step(1)
    s = lat.get_state().double().cpu().numpy()
    d = lat.diag(raise_unstable=False)
    m = lat.column_max().cpu().numpy()
    rho, c = s[:p.Q].sum(0), s[p.Q:].sum(0)
    # FP32 sums over one node's NS (Q) values of magnitude sum below 1.1 (0.06); the
    # sums over nodes are compensated; a mean and 1 + mean add a rounding each
    eps = 2.0 ** -24
    want = 1.0 + c.reshape(nz, ny, nx).mean(1).max(0)
    assert np.abs(m - want).max() <= (1.1 * p.NS + 3) * eps
    assert abs(d["scalar_mass"] - p.N - c.sum()) <= 1.1 * p.NS * eps * p.N
    assert abs(d["mass_delta"] - rho.sum()) <= 0.06 * p.Q * eps * p.N

"""FP32 kernels with two nodes per thread (x and x + 32, packed arithmetic)
against the one-node kernel (LBM_FLAG_ONE_NODE): the collision is written out
operation by operation and is odd or even under c -> -c, so the states agree
bit for bit, at segment edges (64 nodes), walls, wraps and extents of one."""
import dataclasses

import numpy as np
import pytest

from paper_2112_08479_gb300 import inputs, lbm

from helpers import weights, wscalar

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHAPES = [(1, 3, 4), (2, 1, 3), (33, 1, 5), (63, 4, 2), (64, 3, 1), (65, 5, 3), (66, 2, 4),
          (128, 3, 4), (129, 4, 6), (200, 5, 3), (333, 3, 5)]
PX, PZ = lbm.LBM_FLAG_PERIODIC_X, lbm.LBM_FLAG_PERIODIC_Z


def _state(p, seed):
    w = weights(p.model)
    f = w[:, None] * inputs.uniform((p.Q, p.N), seed, 0.05)
    chi = 0.5 * (1.0 + inputs.uniform(p.N, seed + 1, 1.0))
    phi = wscalar(p)[:, None] * (chi * (1.0 + inputs.uniform((p.NS, p.N), seed + 2, 0.05)) - 1.0)
    return torch.from_numpy(np.concatenate([f, phi]).astype(np.float32)).cuda()


def _params(shape, kind, flags):
    nx, ny, nz = shape
    return lbm.Params(nx, ny, nz, model=kind[0], scalar=kind[1], flags=flags, nu=2e-3, D=3e-3, gprime=1e-4,
                      eg=(0.3, -0.4, -0.866), sc_t=0.7, x0=0, H=nz)


@pytest.mark.parametrize("flags", [0, PX, PZ, PX | PZ])
@pytest.mark.parametrize("kind", [(lbm.LBM_BGK_SMAG_Q19, lbm.LBM_SCALAR_Q7),
                                  (lbm.LBM_BGK_SMAG_Q19, lbm.LBM_SCALAR_Q6),
                                  (lbm.LBM_CUMULANT_Q27, lbm.LBM_SCALAR_Q7)])
@pytest.mark.parametrize("shape", SHAPES)
def test_pair_step_equals_one_node_step(shape, kind, flags):
    p = _params(shape, kind, flags)
    a = lbm.Lattice(p, device="cuda")
    b = lbm.Lattice(dataclasses.replace(p, flags=flags | lbm.LBM_FLAG_ONE_NODE), device="cuda")
    s = _state(p, 11)
    a.set_state(s)
    b.set_state(s)
    for _ in range(5):
        a.step(1)
        b.step(1)
        assert torch.equal(a.get_state(), b.get_state())

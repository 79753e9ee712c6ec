"""The plan of a launch of several steps (lbm_step_plan), on the host: which calls
take it, and that its order of items is sound -- every unit of every step is done
once, the item groups of a tile follow each other with the counts that the waits
expect, everything an item waits for has a smaller ticket, and a unit runs in a
later group than the units of the step before on all its neighbours (what keeps
steps apart on the device).  The ticket order is restated here from the
description in csrc/lbm_chain.cuh."""
import itertools

import numpy as np
import pytest

from paper_2112_08479_gb300 import _build, lbm

PX, PZ = lbm.LBM_FLAG_PERIODIC_X, lbm.LBM_FLAG_PERIODIC_Z
BGK, CUM = lbm.LBM_BGK_SMAG_Q19, lbm.LBM_CUMULANT_Q27
SMS = 152


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()
    return lbm.load()


def _plan(shape, steps, flags=0, model=BGK, sms=SMS, **kw):
    nx, ny, nz = shape
    p = lbm.Params(nx, ny, nz, model=model, flags=flags, H=nz, **kw)
    return lbm.lbm_step_plan(p.c(), sms, steps)


def _check_order(shape, steps, flags, model, sms=SMS):
    """Enumerates the tickets of the plan; returns it."""
    nx, ny, nz = shape
    pl = _plan(shape, steps, flags, model, sms)
    T, nslab, M, R, bpt, U, ns, sw, lag = (pl[k] for k in (
        "slots", "slabs", "tiles", "rows", "items", "units", "segments", "slab_segments", "lag"))
    assert pl["steps"] and pl["steps"] == pl["sweeps"] * T
    assert ns == (nx + 63) // 64 and M == -(-ny // R) and bpt * U >= sw * R
    skew = 0 if nslab == 1 else (2 if flags & PX else 1)
    assert nslab * sw >= ns + skew * (T - 1)
    P, groups = M * nz, pl["sweeps"] * nslab
    t = np.arange(pl["tickets"])
    W, r = t // (T * bpt), t % (T * bpt)
    s, b = r // bpt, r % bpt
    v = W - s * lag
    live = (v >= 0) & (v // P < groups)
    t, s, b, v = t[live], s[live], b[live], v[live]
    J, q = v // P, v % P
    z, tile = q // M, (q % M + s) % M
    sweep, slab = J // nslab, J % nslab
    n, nu, p0 = sweep * T + s, J * T + s, slab * sw - skew * s
    # the groups of a tile: bpt items each, later groups after all 3 x 3 tiles of
    # the group before
    ng = groups * T
    first = np.full((ng, nz, M), np.iinfo(np.int64).max)
    last = np.full((ng, nz, M), -1)
    count = np.zeros((ng, nz, M), int)
    np.minimum.at(first, (nu, z, tile), t)
    np.maximum.at(last, (nu, z, tile), t)
    np.add.at(count, (nu, z, tile), 1)
    assert (count == bpt).all()
    for dz, dy in itertools.product((-1, 0, 1), repeat=2):
        need = np.roll(last[:-1], (-dz, -dy), (1, 2))
        if not flags & PZ and dz:
            need[:, 0 if dz < 0 else -1] = -1
        assert (first[1:] > need).all()
    # units
    g = b[:, None] * U + np.arange(U)
    row, seg = g // sw, p0[:, None] + g % sw
    y = tile[:, None] * R + row
    ok = (row < R) & (y < ny) & (seg >= 0) & (seg < ns)
    turn = s[:, None] if skew == 2 else 0
    seg = (seg + turn) % ns
    N = np.broadcast_to(n[:, None], g.shape)[ok], np.broadcast_to(z[:, None], g.shape)[ok]
    nuu = np.broadcast_to(nu[:, None], g.shape)[ok]
    done = np.zeros((pl["steps"], nz, ny, ns), int)
    group = np.zeros((pl["steps"], nz, ny, ns), int)
    np.add.at(done, (N[0], N[1], y[ok], seg[ok]), 1)
    group[N[0], N[1], y[ok], seg[ok]] = nuu
    assert (done == 1).all()
    for dz, dy, dx in itertools.product((-1, 0, 1), repeat=3):
        before = np.roll(group[:-1], (-dz, -dy, -dx), (1, 2, 3))
        if not flags & PZ and dz:
            before[:, 0 if dz < 0 else -1] = -1
        if not flags & PX and dx:
            before[..., 0 if dx < 0 else -1] = -1
        assert (group[1:] > before).all()
    return pl


@pytest.mark.parametrize("model", [BGK, CUM])
@pytest.mark.parametrize("shape,steps,flags,want", [
    # one slot, the state in L2: wraps, odd row counts, one tile per plane
    ((64, 66, 66), 24, 0, dict(slots=1, slabs=1, sweeps=24)),
    ((64, 66, 66), 25, PX | PZ, dict(slots=1, slabs=1, sweeps=25)),
    ((333, 17, 60), 24, PZ, dict(slots=1, slabs=1)),
    ((35, 3, 1500), 24, PX, dict(slots=1, tiles=1)),
    ((40, 1, 4300), 24, PZ, dict(slots=1, tiles=1)),
    # a wave over whole rows; one tile per plane; few planes
    ((300, 12, 600), 9, PX, dict(slots=4, slabs=1, sweeps=2)),
    ((64, 3, 5500), 9, 0, dict(slots=4, slabs=1, sweeps=2, tiles=1)),
    ((1000, 500, 4), 4, 0, dict(slots=2, slabs=3, sweeps=2)),
    # slabs along x, at least two sweeps
    ((2048, 128, 24), 7, 0, dict(slots=3, sweeps=2)),
    ((2048, 128, 24), 7, PX, dict(slots=3, sweeps=2)),
    ((2500, 150, 40), 6, PX, dict(slots=3, sweeps=2)),
])
def test_order_of_items(shape, steps, flags, want, model):
    pl = _check_order(shape, steps, flags, model)
    assert {k: pl[k] for k in want} == want
    assert pl["slabs"] >= 2 or "slabs" in want or want["slots"] == 1


@pytest.mark.parametrize("sms", [1, 7, 160])
def test_order_on_other_devices(sms):
    _check_order((1000, 61, 90), 6, PX, CUM, sms)


def test_which_calls_share_a_launch():
    """By state size (105 and 80 MB), steps, rows and kind of box."""
    assert _plan((512, 64, 32), 2)["steps"] == 2                    # 109 MB
    assert _plan((512, 64, 32), 1)["steps"] == 0
    assert _plan((333, 47, 59), 11)["steps"] == 0                   # 96 MB
    assert _plan((333, 47, 59), 12)["steps"] == 12
    assert _plan((256, 32, 64), 23)["steps"] == 0                   # 55 MB
    assert _plan((256, 32, 64), 24)["steps"] == 24
    assert _plan((128, 8, 16), 1000)["steps"] == 0                  # too few rows
    assert _plan((1024, 64, 128), 100, PZ)["steps"] == 0            # no end for a wave
    assert _plan((32, 60, 625), 100, 0, CUM)["steps"] == 0          # half-empty pairs
    assert _plan((33, 60, 625), 100, 0, CUM)["steps"] == 100
    assert _plan((32, 60, 625), 100)["steps"] == 100
    assert _plan((2, 60, 5000), 100)["steps"] == 0                  # nearly empty units
    assert _plan((3, 60, 5000), 100)["steps"] == 100
    big = (1024, 64, 64)
    for kw in (dict(storage=lbm.LBM_FP16S), dict(storage=lbm.LBM_BF16S),
               dict(flags=lbm.LBM_FLAG_ONE_NODE), dict(model=CUM, scalar=lbm.LBM_SCALAR_Q27)):
        assert _plan(big, 100, **kw)["steps"] == 0, kw
    assert _plan(big, 100, scalar=lbm.LBM_SCALAR_Q6)["steps"] == 100
    assert _plan((2048, 256, 320), 100)["steps"] == 0               # 64-bit offsets


def test_bench_box():
    pl = _plan((2048, 128, 256), 100)
    assert (pl["steps"], pl["slots"], pl["slabs"], pl["sweeps"]) == (99, 3, 3, 33)


@pytest.mark.parametrize("shape,flags,model", [
    ((2048, 128, 256), 0, BGK), ((2500, 150, 100), PX, BGK), ((1024, 64, 128), 0, CUM),
    ((256, 32, 64), PZ, BGK), ((65535, 2, 300), 0, CUM)])
@pytest.mark.parametrize("steps", [8000, 1000003, 2**31 - 1])
def test_long_calls_share_launches(shape, flags, model, steps):
    """A call of any length goes by launches of whole sweeps whose units stay
    below 2^31; only the steps short of a sweep are left."""
    short = _plan(shape, 100, flags, model)
    pl = _plan(shape, steps, flags, model)
    assert pl["tickets"] * pl["units"] < 2**31 and pl["steps"] <= steps
    for k in ("slots", "slabs", "tiles", "rows", "items", "lag"):
        assert pl[k] == short[k]
    assert pl["steps"] == pl["sweeps"] * pl["slots"]
    per_sweep = pl["slabs"] * pl["tiles"] * shape[2] * pl["slots"] * pl["items"]
    if pl["steps"] < steps - steps % pl["slots"]:      # cut: one sweep more does not fit
        assert (pl["tickets"] + per_sweep) * pl["units"] >= 2**31
    left, launches = steps, 0
    while (n := _plan(shape, left, flags, model)["steps"]):
        k = max(1, left // n - 1)                       # launches of this size in a row
        left, launches = left - k * n, launches + k
    assert left < 24 and launches <= steps / 1000 + 8


def test_arguments():
    import ctypes as C
    p, out = lbm.Params(64, 4, 8, H=8).c(), (C.c_int64 * 12)()
    lib = lbm.load()
    assert lib.lbm_step_plan(C.byref(p), 0, 1, out) == lbm.LBM_ERR_ARG
    assert lib.lbm_step_plan(C.byref(p), 1, -1, out) == lbm.LBM_ERR_ARG
    assert lib.lbm_step_plan(C.byref(p), 1, 1, None) == lbm.LBM_ERR_ARG
    assert lib.lbm_step_plan(None, 1, 1, out) == lbm.LBM_ERR_ARG
    assert lib.lbm_step_plan(C.byref(p), 1, 0, out) == lbm.LBM_OK and list(out) == [0] * 12

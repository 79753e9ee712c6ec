"""bench.py's count of step launches follows the library's plan, and its traffic
lookup covers every source that decides the traffic of the headline kernel."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402
from paper_2112_08479_gb300 import _build, lbm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()
    return lbm.load()


@pytest.mark.parametrize("model,storage,scalar,n,want", [
    ("bgk", "fp32", "q7", 100, 2),          # 33 sweeps of three, then one step
    ("bgk", "fp32", "q7", 99, 1),
    ("bgk", "fp32", "q7", 1, 1),
    ("bgk", "fp32", "q7", 0, 0),
    ("cumulant", "fp32", "q7", 100, 2),
    ("bgk", "fp16s", "q7", 100, 100),
    ("cumulant", "fp32", "q27", 100, 100),
])
def test_step_launches_of_the_bench_box(model, storage, scalar, n, want):
    w = bench.WORKLOADS["config3"]
    p = lbm.lock_exchange(w["nx"], w["ny"], w["nz"], H=w["H"], x0=w["x0"], u_b=w["u_b"],
                          Re=w["Re"], model=model, storage=storage, scalar=scalar)
    assert bench.step_launches(p.c(), 152, n) == want


def test_traffic_is_stale_after_a_change_of_the_plan():
    names = {os.path.basename(s) for s in bench.KERNEL_SOURCES}
    assert {"lbm_aux.cu", "lbm_bgk.cu", "lbm_bgk_collide.cuh", "lbm_chain.cuh", "lbm_common.cuh",
            "lbm_internal.h", "lbm_lanes.cuh", "lbm_pair.cuh"} <= names

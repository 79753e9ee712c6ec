"""Kernels whose launches overlap give what they give one at a time: back to back
on one stream, behind other work of the stream, across a fork and a join, and
captured in a graph with each of these."""
import pytest

from paper_2112_08479_gb300 import lbm

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = [("bgk", "fp16s", "q7"), ("cumulant", "bf16s", "q7"), ("cumulant", "fp32", "q27"),
         ("bgk", "fp32", "q6"), ("cumulant", "fp32", "q7")]


def _lattice(model, storage, scalar, stream=None):
    p = lbm.lock_exchange(96, 5, 24, H=24, x0=24, u_b=0.03, Re=2000, model=model,
                          storage=storage, scalar=scalar)
    return lbm.Lattice(p, stream=stream) if stream is not None else lbm.Lattice(p)


@pytest.mark.parametrize("case", CASES)
def test_steps_behind_other_work(case):
    s, side = torch.cuda.Stream(), torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        ref = _lattice(*case, stream=s)
        for _ in range(18):
            ref.step(1)
            s.synchronize()
        want = ref.get_state()
        lat = _lattice(*case, stream=s)
        out, other = torch.empty_like(want), torch.zeros(1 << 20, device="cuda")

        def work():
            other.zero_()
            lat.step(1)
            side.wait_stream(s)
            with torch.cuda.stream(side):
                other.add_(1.0)
            lat.step(1)
            s.wait_stream(side)
            lat.step(4)

        work()
        lat.get_state(out)
        work()
        s.synchronize()
        state = lat.get_state()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            work()
            lat.get_state(out)
        lat.set_state(state, 12)
        g.replay()
        s.synchronize()
    assert torch.equal(out, want)
    assert float(other[0]) == 1.0

"""The adjoint's zero pass starts during the gather's tail: captured in a
graph, replayed, and called back to back on two streams, it gives the eager
result bit for bit."""
import numpy as np
import pytest

from gpu_util import bits, flat, to_device, to_device_innermost
from paper_2605_14780_gb300 import bc, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", ["outermost", "innermost"])
@pytest.mark.parametrize("make", [
    lambda: synth.batching(nblocks=40, side_lo=8, side_hi=60, lev_lo=1, lev_hi=20, h=2, seed=71,
                           dtype="f32"),
    lambda: synth.cubed_sphere(24, 3, 6, 9, ("h", "u", "v"), "f64", seed=72)])
def test_captured_and_two_streams(make, layout):
    import torch
    dev = to_device if layout == "outermost" else to_device_innermost
    w = make()
    cots = [synth.cotangent_like(w, 73 + k) for k in range(2)]
    src = [dev(c) for c in cots]
    want = []
    plan = bc.plan_for_workload(w, src[0])
    for s in src:
        ts = [t.clone() for t in s]
        plan.adjoint(bc.slot_table(ts))
        torch.cuda.synchronize()
        want.append(flat([t.cpu().numpy() for t in ts]))
    ts = [t.clone() for t in src[0]]
    table = bc.slot_table(ts)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        plan.adjoint(table, stream=stream)
    for _ in range(3):
        for t, u in zip(ts, src[0]):
            t.copy_(u)
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(bits(flat([t.cpu().numpy() for t in ts])), bits(want[0]))
    streams = [torch.cuda.Stream() for _ in range(2)]
    for _ in range(5):
        work = [[t.clone() for t in s] for s in src]
        tables = [bc.slot_table(x) for x in work]
        torch.cuda.synchronize()
        for st, t in zip(streams, tables):
            plan.adjoint(t, stream=st)
        torch.cuda.synchronize()
        for x, r in zip(work, want):
            assert np.array_equal(bits(flat([t.cpu().numpy() for t in x])), bits(r))

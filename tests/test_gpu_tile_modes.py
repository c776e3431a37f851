"""Staged tiles against the per-lane rows in the launches that the default
options leave to larger plans (one kernel per family) and to small ones (one
kernel of all kinds), with CTAs of few and of many threads: FP64 CSR tiles ask
for 128 KB of shared memory at 512."""
import numpy as np
import pytest

from gpu_util import bits, flat, to_device
from paper_2605_14780_gb300 import bc, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads", [64, 512])
@pytest.mark.parametrize("mode", [bc.BC_BATCH_FAMILIES, bc.BC_BATCH_SINGLE])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("N,p,quad,levels", [(33, 6, None, 9), (64, 4, None, 5), (34, 4, 2, 9),
                                             (65, 4, 2, 4)])
def test_tiles_match_per_lane_rows(N, p, quad, levels, dtype, mode, threads):
    import torch
    w = synth.cubed_sphere(N, 3, p, levels, ("h", "u", "v"), dtype, seed=91, quad=quad)
    cot = synth.cotangent_like(w, 92)
    res, items = [], []
    for u in (0, 1):
        ts, cs = to_device(w["fields"]), to_device(cot)
        plan = bc.plan_for_workload(w, ts, {"unstaged_rows": u, "batch_mode": mode,
                                            "threads": threads})
        plan.apply(bc.slot_table(ts))
        plan.adjoint(bc.slot_table(cs))
        torch.cuda.synchronize()
        res.append(flat([t.cpu().numpy() for t in ts + cs]))
        items.append(plan.stats()["nitems"])
    assert items[0] != items[1]  # the first plan has tiles
    assert np.array_equal(bits(res[0]), bits(res[1]))

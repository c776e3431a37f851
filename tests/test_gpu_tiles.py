"""Staged tiles against the per-lane rows at the sizes where tiles end early
(odd panels, strips shorter than a tile, level counts around one stage), and
the adjoint's row records (levels innermost) against the oracle: rows of one,
two and many entries, rows that read several slots."""
import numpy as np
import pytest

from gpu_util import bits, flat, to_device, to_device_innermost
from oracle.operator import apply_adjoint, build_operator
from paper_2605_14780_gb300 import bc, synth

pytestmark = pytest.mark.gpu


def _both(w, opts, dev, cot):
    import torch
    ts, cs = dev(w["fields"]), dev(cot)
    plan = bc.plan_for_workload(w, ts, opts)
    plan.apply(bc.slot_table(ts))
    plan.adjoint(bc.slot_table(cs))
    torch.cuda.synchronize()
    return flat([t.cpu().numpy() for t in ts]), flat([c.cpu().numpy() for c in cs])


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("N,h,p,quad,levels", [
    (8, 2, 4, None, 2), (13, 3, 6, None, 5), (33, 3, 6, None, 8), (45, 2, 8, None, 9),
    (31, 1, 2, None, 17), (11, 3, 4, 2, 3), (34, 3, 4, 2, 9), (29, 2, 6, 2, 8)])
def test_tiles_match_per_lane_rows(N, h, p, quad, levels, dtype):
    w = synth.cubed_sphere(N, h, p, levels, ("h", "u", "v"), dtype, seed=51, quad=quad)
    cot = synth.cotangent_like(w, 52)
    res = [_both(w, {"unstaged_rows": u}, to_device, cot) for u in (0, 1)]
    for a, b in zip(*res):
        assert np.array_equal(bits(a), bits(b))


@pytest.mark.parametrize("dtype,tol", [("f32", 64 * 2.0 ** -24), ("f64", 1e-12)])
@pytest.mark.parametrize("make", [
    lambda dt: synth.batching(nblocks=30, side_lo=4, side_hi=12, lev_lo=1, lev_hi=7, h=2,
                              seed=53, dtype=dt),
    lambda dt: synth.cubed_sphere(9, 3, 6, 5, ("h", "u", "v"), dt, seed=54),
    lambda dt: synth.cubed_sphere(12, 2, 4, 1, ("scalar",), dt, seed=55, quad=2)])
def test_adjoint_levels_innermost(make, dtype, tol):
    w = make(dtype)
    cot = synth.cotangent_like(w, 56)
    _, got = _both(w, {}, to_device_innermost, cot)
    op = build_operator(w)
    ref = flat(apply_adjoint(op, cot))
    # the error's scale: the value's own cotangent and the terms it gathers;
    # FP32 rounds the weights and at most 62 terms
    mag = type(op)(op.layout, op.rows, abs(op.A), op.b)
    lim = flat(apply_adjoint(mag, [np.abs(c) for c in cot]))
    assert np.all(np.abs(got - ref) <= tol * lim)
    assert np.all(got[op.rows] == 0)

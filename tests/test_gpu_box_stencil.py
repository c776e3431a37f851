"""The box form of the fused stencil (27 points, one weight off the centre)
against the general kernel, which the same stencil takes when its centre is
listed as two points: tile edges, odd planes, levels, both dtypes, and
values whose sums overflow or are not finite."""
import numpy as np
import pytest

from gpu_util import to_device, to_device_innermost
from paper_2605_14780_gb300 import bc, synth

pytestmark = pytest.mark.gpu

EPS = {"f32": 2.0 ** -23, "f64": 2.0 ** -52}
BOX = bc.box_stencil(3, 1)


def _work(n, variant, dtype, nlevels):
    w = synth.hpcg_block(n, variant, dtype=dtype, nblocks=2, seed=31)
    w["blocks"] = [dict(b, nlevels=nlevels) for b in w["blocks"]]
    w["fields"] = synth.uniform_fields(w["blocks"], dtype, -1.0, 1.0, 31)
    return w


def _run(w, a, c0, split, layout="outermost"):
    import torch
    dev = to_device_innermost if layout == "innermost" else to_device
    ts, outs = dev(w["fields"]), dev([np.zeros_like(f) for f in w["fields"]])
    plan = bc.plan_for_workload(w, ts, {"stencil_fusion": 1})
    off, coef = BOX, np.where(BOX.any(axis=1), a, c0)
    if split:  # 28 points: the general kernel
        off = np.concatenate([BOX, [(0, 0, 0)]])
        coef = np.append(np.where(BOX.any(axis=1), a, c0 / 2), c0 / 2)
    plan.apply_stencil(bc.slot_table(ts), bc.slot_table(outs), off, coef)
    torch.cuda.synchronize()
    return [t.cpu().numpy() for t in ts], [o.cpu().numpy() for o in outs]


@pytest.mark.parametrize("n,nlevels,layout", [
    ((1, 1, 1), 1, "outermost"), ((2, 3, 4), 1, "outermost"), ((31, 32, 33), 1, "outermost"),
    ((33, 31, 5), 1, "outermost"), ((64, 65, 7), 1, "outermost"), ((5, 97, 34), 1, "outermost"),
    ((34, 9, 6), 3, "outermost"), ((34, 9, 6), 3, "innermost")])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("variant,a,c0", [("P", -1.0, 26.0), ("S", 0.375, -2.5), ("Z", 1.0, 1.0)])
def test_box_against_general(n, nlevels, layout, dtype, variant, a, c0):
    w = _work(n, variant, dtype, nlevels)
    f1, o1 = _run(w, a, c0, False, layout)
    f2, o2 = _run(w, a, c0, True, layout)
    # each side rounds fewer than 40 times against sum |c x| (|x| <= 1), the
    # box form also the centre's a x0 and (c0 - a) x0
    lim = 40 * EPS[dtype] * (26 * abs(a) + 2 * (abs(c0) + abs(a)))
    for x, y in zip(f1, f2):
        assert np.array_equal(x, y, equal_nan=True)
    for x, y in zip(o1, o2):
        assert np.max(np.abs(x.astype(np.float64) - y)) <= lim


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_box_values_not_finite(dtype):
    big = np.finfo(np.float64 if dtype == "f64" else np.float32).max
    w = _work((37, 12, 9), "P", dtype, 1)
    d = synth.data_view(w["fields"][0], w["blocks"][0])
    d[0, 0, 4, 5, 6] = np.inf
    d[0, 0, 7, 2, 35] = -np.inf
    d[0, 0, 1, 9, 20] = np.nan
    d[0, 0, 8, 11, 0] = np.inf
    synth.data_view(w["fields"][1], w["blocks"][1])[...] = big / 2  # box sums overflow
    for a, c0 in ((-1.0, 26.0), (1.0 / 27, 1.0 / 27)):
        (_, o1), (_, o2) = _run(w, a, c0, False), _run(w, a, c0, True)
        assert np.array_equal(np.isnan(o1[0]), np.isnan(o2[0]))
        assert np.array_equal(np.isinf(o1[0]), np.isinf(o2[0]))
        inf = np.isinf(o1[0])
        assert np.array_equal(o1[0][inf], o2[0][inf])
        if a > 0:
            assert np.all(np.isfinite(o1[1]))
            assert np.max(np.abs(o1[1] / 2 - o2[1] / 2)) <= 40 * EPS[dtype] * (big / 2)

"""The box form of the fused stencil: that FP64 calls take it and FP32 calls do
not, that it is not the slower one where the grid fills few SMs, and its sums
against sums in higher precision on grids the other tests leave out (a halo
wider than the stencil, blocks stored with other axis orders, pruned plans,
ghosts that are table rows, one plan on two streams)."""
import numpy as np
import pytest

from gpu_util import bits, flat, to_device
from paper_2605_14780_gb300 import bc, synth

pytestmark = pytest.mark.gpu

BOX = bc.box_stencil(3, 1)
COEF = np.where(BOX.any(axis=1), -1.0, 26.0)
GENERAL = np.concatenate([BOX, [(0, 0, 0)]])  # 28 points: the general kernel
GENERAL_COEF = np.append(np.where(BOX.any(axis=1), -1.0, 13.0), 13.0)
EPS = 2.0 ** -52


def _work(n, variant="P", h=1, nlevels=1, dtype="f64"):
    w = synth.hpcg_block(n, variant, dtype=dtype, nblocks=2, seed=41)
    w["blocks"] = [dict(b, h=(h, h, h), nlevels=nlevels) for b in w["blocks"]]
    w["fields"] = synth.uniform_fields(w["blocks"], dtype, -1.0, 1.0, 42)
    return w


def _table_rows(n):
    """The low-x faces as rows over two cells of the block itself."""
    w = _work(n)
    bcs = [dict(d, faces=[f for f in d["faces"] if (f["axis"], f["side"]) != (0, 0)])
           for d in w["bcs"]]
    jk = [(j, k) for k in range(n[2]) for j in range(n[1])]
    ijk = np.array([(i, j, k) for j, k in jk for i in (0, n[0] - 1)], np.int32)
    m = len(jk)
    for b in range(2):
        bcs.append({"kind": "csr", "block": b, "lo": (-1, 0, 0), "hi": (0, n[1], n[2]),
                    "comps": [0], "row_ptr": np.arange(0, 2 * m + 1, 2, dtype=np.int64),
                    "col_block": np.full(2 * m, b, np.int32),
                    "col_comp": np.zeros(2 * m, np.int32), "col_ijk": ijk,
                    "val": np.tile([0.75, 0.25], m)})
    return dict(w, bcs=bcs)


def _stored(order):
    """Device copies whose axes (C, L, F2, F1, F0) are stored in `order`."""
    def dev(fields):
        import torch
        back = np.argsort(order)
        return [torch.from_numpy(np.ascontiguousarray(a.transpose(order))).cuda().permute(*back)
                for a in fields]
    return dev


def _run(w, off=BOX, coef=COEF, dev=to_device, stencil=None):
    import torch
    ts, outs = dev(w["fields"]), dev([np.zeros_like(f) for f in w["fields"]])
    plan = bc.plan_for_workload(w, ts, {"stencil_fusion": 1}, stencil=stencil)
    plan.apply_stencil(bc.slot_table(ts), bc.slot_table(outs), off, coef)
    torch.cuda.synchronize()
    return [t.cpu().numpy() for t in ts], [o.cpu().numpy() for o in outs]


@pytest.mark.parametrize("dtype,differs", [("f64", True), ("f32", False)])
def test_route(dtype, differs):
    # random values: the two orders of the sums round differently somewhere
    # (a 28th weight of zero adds nothing to a finite sum)
    w = _work((40, 24, 12), dtype=dtype)
    (_, a), (_, b) = _run(w), _run(w, GENERAL, np.append(COEF, 0.0))
    assert np.array_equal(bits(flat(a)), bits(flat(b))) != differs


@pytest.mark.parametrize("make,dev,pruned", [
    (lambda: _work((33, 18, 7), h=2), to_device, False),
    (lambda: _work((33, 18, 7), h=2), to_device, True),
    (lambda: _work((21, 35, 6), "S", nlevels=3), to_device, True),
    (lambda: _work((21, 35, 6), "S", nlevels=3), _stored((0, 1, 4, 3, 2)), False),
    (lambda: _work((34, 17, 9)), _stored((0, 3, 1, 4, 2)), False),
    (lambda: _table_rows((35, 19, 8)), to_device, False)])
def test_box_against_exact_sums(make, dev, pruned):
    w = make()
    fields, outs = _run(w, dev=dev, stencil=BOX if pruned else None)
    # 28 weights of 1 and 26 on |x| <= 1; fewer than 40 roundings of it, the
    # centre's x0 and 27 x0 among the terms
    lim = 40 * EPS * (26 + 2 * 27)
    for f, o, blk in zip(fields, outs, w["blocks"]):
        n, h = blk["n"], blk["h"]
        x = f.astype(np.longdouble)
        want = 0
        for (i, j, k), c in zip(BOX, COEF):
            want = want + np.longdouble(c) * x[..., h[2] + k:h[2] + k + n[2],
                                               h[1] + j:h[1] + j + n[1], h[0] + i:h[0] + i + n[0]]
        got = o[..., h[2]:h[2] + n[2], h[1]:h[1] + n[1], h[0]:h[0] + n[0]]
        assert np.max(np.abs(got - want)) <= lim


def test_one_plan_on_two_streams():
    import torch
    w = _table_rows((35, 19, 8))
    _, want = _run(w)
    sides = []
    for _ in range(2):
        ts, outs = to_device(w["fields"]), to_device([np.zeros_like(f) for f in w["fields"]])
        sides.append((ts, outs, bc.slot_table(ts), bc.slot_table(outs), torch.cuda.Stream()))
    plan = bc.plan_for_workload(w, sides[0][0], {"stencil_fusion": 1})
    torch.cuda.synchronize()
    for _ in range(20):
        for _, _, table, out_table, stream in sides:
            plan.apply_stencil(table, out_table, BOX, COEF, stream=stream)
    torch.cuda.synchronize()
    for _, outs, _, _, _ in sides:
        assert np.array_equal(bits(flat([o.cpu().numpy() for o in outs])), bits(flat(want)))


@pytest.mark.parametrize("n,nblocks", [((128, 128, 128), 1), ((64, 64, 64), 4),
                                       ((100, 37, 61), 3)])
def test_box_is_not_the_slower_form(n, nblocks):
    # the general kernel took 0.7 of the box form's time where tiles of too many
    # planes left the SMs with one or none; it takes 1.5 to 2.4 times as long
    import torch
    w = synth.hpcg_block(n, "Z", nblocks=nblocks, seed=43)
    ts, outs = to_device(w["fields"]), to_device(w["fields"])
    plan = bc.plan_for_workload(w, ts, {"stencil_fusion": 1})
    table, out_table = bc.slot_table(ts), bc.slot_table(outs)

    def best(off, coef):
        times = []
        for _ in range(8):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(20):
                plan.apply_stencil(table, out_table, off, coef)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    assert best(BOX, COEF) < best(GENERAL, GENERAL_COEF)

"""bc_pack_run against slicing: tiles' edges (cells and levels past one
tile), both level layouts, odd boxes, 3-D boxes, both element sizes."""
import numpy as np
import pytest

from gpu_util import bits, to_device, to_device_innermost
from paper_2605_14780_gb300 import bc, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", ["outermost", "innermost"])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("n,levels,ncomp,boxes", [
    ((37, 5, 1), 1, 1, [((-2, -2, 0), (39, 7, 1))]),
    ((40, 70, 1), 3, 2, [((0, 0, 0), (2, 70, 1)), ((0, 0, 0), (40, 2, 1)), ((5, 6, 0), (6, 7, 1))]),
    ((33, 9, 1), 64, 1, [((0, 0, 0), (33, 9, 1)), ((1, 1, 0), (32, 3, 1))]),
    ((21, 8, 1), 65, 1, [((0, 0, 0), (21, 8, 1))]),
    ((16, 4, 1), 130, 2, [((-1, -1, 0), (17, 5, 1))]),
    ((7, 6, 5), 4, 1, [((-2, 0, 1), (3, 6, 4)), ((6, 5, -2), (9, 8, 7))])])
def test_pack_tiles(n, levels, ncomp, boxes, dtype, layout):
    import torch
    h = (2, 2, 2 if n[2] > 1 else 0)
    blocks = [{"n": n, "h": h, "nlevels": levels, "ncomp": ncomp} for _ in range(2)]
    rng = np.random.default_rng(3)
    fields = [rng.uniform(-1, 1, synth.full_shape(b)).astype(synth.DTYPES[dtype]) for b in blocks]
    ts = (to_device_innermost if layout == "innermost" else to_device)(fields)
    every = [(b, lo, hi) for b in (1, 0) for lo, hi in boxes]
    pk = bc.Pack(bc.block_descriptors(ts, blocks), every, dtype)
    buf = torch.full((pk.size,), float("nan"), dtype=ts[0].dtype, device="cuda")
    pk.run(bc.slot_table(ts), buf)
    want = np.concatenate([fields[b][:, :, lo[2] + h[2]:hi[2] + h[2], lo[1] + h[1]:hi[1] + h[1],
                                     lo[0] + h[0]:hi[0] + h[0]].ravel() for b, lo, hi in every])
    assert np.array_equal(bits(buf.cpu().numpy()), bits(want))

"""Which rows are staged in tiles: rows whose columns lie apart cut short tiles,
which take a warp each and leave most of its lanes idle, so they keep the
per-lane path; rows of long tiles stay staged."""
import numpy as np
import pytest

from paper_2605_14780_gb300 import bc, specs, synth


def _plan(w, **opts):
    blocks = [specs.contiguous_block(b) for b in w["blocks"]]
    plan = bc.Plan(blocks, specs.submatrices(w), w["dtype"], dict(opts, host_only=1))
    n, bad, msg = plan.check_work()
    assert n > 0 and bad == 0, msg
    return plan.stats()


def _staged(w, what="nitems"):
    return _plan(w)[what] != _plan(w, unstaged_rows=1)[what]


def grouped_interp(group, dtype, p=4, n=96, nlevels=8):
    """Two blocks; the ghosts left of each read rows of p nodes along y in the
    other, `group` neighbours in a column before the next column, 37 cells on."""
    blocks = [synth.block2d(n, n, 1, nlevels, 3) for _ in range(2)]
    q = np.arange(n)
    start = np.stack([(q // group * 37) % n, (q // group * 41) % (n - p - group) + q % group,
                      np.zeros(n, int)], 1)
    rng = np.random.default_rng(7)
    bcs = [{"kind": "interp", "block": b, "lo": (-1, 0, 0), "hi": (0, n, 1), "comps": [0, 1, 2],
            "src_block": 1 - b, "p": p, "start": start.astype(np.int32),
            "axis": np.ones(n, np.int32), "w": rng.uniform(-1, 1, (n, p)), "rot_comp": (1, 2),
            "rot": rng.uniform(-1, 1, (n, 4))} for b in range(2)]
    return {"dtype": dtype, "blocks": blocks, "bcs": bcs,
            "fields": synth.uniform_fields(blocks, dtype, -1.0, 1.0, 8)}


@pytest.mark.parametrize("dtype,group,staged", [
    ("f32", 1, False), ("f32", 3, False), ("f32", 12, True), ("f32", 32, True),
    ("f64", 1, False), ("f64", 12, False), ("f64", 32, True)])
def test_interpolation_rows(dtype, group, staged):
    assert _staged(grouped_interp(group, dtype)) == staged

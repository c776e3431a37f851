"""Which rows are staged in tiles: rows whose columns lie apart cut short tiles,
which take a warp each and leave most of its lanes idle, so they keep the
per-lane path; rows of long tiles stay staged."""
import numpy as np
import pytest

from paper_2605_14780_gb300 import bc, specs, synth


def _plan(w, check=True, **opts):
    blocks = [specs.contiguous_block(b) for b in w["blocks"]]
    plan = bc.Plan(blocks, specs.submatrices(w), w["dtype"], dict(opts, host_only=1))
    if check:
        n, bad, msg = plan.check_work()
        assert n > 0 and bad == 0, msg
    return plan.stats()


def _staged(w, what="nitems"):
    # chunks of levels of which a tile and a per-lane item hold different counts
    opts = {"level_chunk": 8} if w["dtype"] == "f64" else {}
    return _plan(w, **opts)[what] != _plan(w, check=False, unstaged_rows=1, **opts)[what]


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
    return {"dtype": dtype, "blocks": blocks, "bcs": bcs}


@pytest.mark.parametrize("dtype,group,staged", [
    ("f32", 1, False), ("f32", 3, False), ("f32", 12, True), ("f32", 32, True),
    ("f64", 1, False), ("f64", 12, False), ("f64", 32, True)])
def test_interpolation_rows(dtype, group, staged):
    assert _staged(grouped_interp(group, dtype)) == staged


def grouped_csr(group, dtype, n=96, nlevels=520):
    """As grouped_interp, with rows over patches of 4 x 4 cells."""
    blocks = [synth.block2d(n, n, 1, nlevels, 1) for _ in range(2)]
    q = np.arange(n)
    i0, j0 = (q // group * 37) % (n - 4), (q // group * 41) % (n - 4 - group) + q % group
    di, dj = np.meshgrid(np.arange(4), np.arange(4))
    ijk = np.stack([(i0[:, None] + di.ravel()).ravel(), (j0[:, None] + dj.ravel()).ravel(),
                    np.zeros(16 * n, int)], 1)
    val = np.random.default_rng(9).uniform(-1, 1, 16 * n)
    bcs = [{"kind": "csr", "block": b, "lo": (-1, 0, 0), "hi": (0, n, 1), "comps": [0],
            "row_ptr": np.arange(0, 16 * n + 1, 16, dtype=np.int64),
            "col_block": np.full(16 * n, 1 - b, np.int32), "col_comp": np.zeros(16 * n, np.int32),
            "col_ijk": ijk.astype(np.int32), "val": val} for b in range(2)]
    return {"dtype": dtype, "blocks": blocks, "bcs": bcs}


@pytest.mark.parametrize("dtype,group,staged", [
    ("f32", 1, False), ("f32", 8, False), ("f32", 16, True), ("f32", 32, True),
    ("f64", 8, False), ("f64", 24, False), ("f64", 32, True)])
def test_csr_rows(dtype, group, staged):
    assert _staged(grouped_csr(group, dtype)) == staged


def quad_like(n, dtype="f32", nlevels=8):
    """A strip of n x 3 ghosts over 4 x 4 patches, as at a panel edge."""
    blocks = [synth.block2d(n, n, 3, nlevels, 1)]
    i, j = [v.ravel() for v in np.meshgrid(np.arange(n), np.arange(3))]
    di, dj = np.meshgrid(np.arange(4), np.arange(4))
    m = 16 * len(i)
    ijk = np.stack([(np.clip(i - 1, 0, n - 4)[:, None] + di.ravel()).ravel(),
                    (j[:, None] + dj.ravel()).ravel(), np.zeros(m, int)], 1)
    return {"dtype": dtype, "blocks": blocks, "bcs": [
        {"kind": "csr", "block": 0, "lo": (0, -3, 0), "hi": (n, 0, 1), "comps": [0],
         "row_ptr": np.arange(0, m + 1, 16, dtype=np.int64),
         "col_block": np.zeros(m, np.int32), "col_comp": np.zeros(m, np.int32),
         "col_ijk": ijk.astype(np.int32),
         "val": np.random.default_rng(11).uniform(-1, 1, m)}]}


@pytest.mark.parametrize("n", [33, 65, 97, 257])
def test_a_short_last_tile_keeps_the_others_staged(n):
    # 32 rows and then one, in every row of the strip: both are tiles
    w = quad_like(n)
    tiles = 3 * -(-n // 32)
    assert _plan(w)["nitems"] <= tiles * 2  # 8 levels, four a stage
    assert _staged(w)


@pytest.mark.parametrize("dtype,group,staged", [
    ("f32", 4, False), ("f32", 8, False), ("f32", 16, True), ("f32", 32, True),
    ("f64", 4, False), ("f64", 8, False), ("f64", 32, True)])
def test_transpose_rows(dtype, group, staged):
    # a group of g ghosts reads a column of g + 3 cells: as many rows
    assert _staged(grouped_interp(group, dtype), "nitems_adjoint") == staged

"""Closed groups of Sync rows (the copies of one node, summed in place from the
group's record): rows whose entries come in any order, with weights of their
own, that read one, some or all of the group's cells, or nothing; values that
are not finite stay out of rows that do not read them; rows of more entries
than a record holds keep the staged route."""
import numpy as np
import pytest

from gpu_util import bits, compare, flat, run, to_device, to_device_innermost
from paper_2605_14780_gb300 import bc, specs, synth


def _grid(kind, dtype, nlevels, ncomp=2, open_row=False):
    w = synth.sync_grid(3, 2, 7, 2, nlevels, ncomp, dtype=dtype, seed=91)
    rng = np.random.default_rng(92)
    for b in w["bcs"]:
        if b["kind"] != "sync":
            continue
        ptr, out = [0], {"col_block": [], "col_comp": [], "col_ijk": [], "val": []}
        for r in range(len(b["row_ptr"]) - 1):
            e = list(range(b["row_ptr"][r], b["row_ptr"][r + 1]))
            if kind == "shuffled":
                rng.shuffle(e)
            elif kind == "some":  # one cell or more, or none
                rng.shuffle(e)
                e = e[:rng.integers(0, len(e) + 1)]
            elif kind == "repeated":  # a cell twice: up to five entries
                e = e + e[:1]
            for k in e:
                out["col_block"].append(b["col_block"][k])
                out["col_comp"].append(b["col_comp"][k])
                out["col_ijk"].append(b["col_ijk"][k])
                out["val"].append(rng.uniform(-1, 1))
            ptr.append(len(out["val"]))
        b["row_ptr"] = np.array(ptr, np.int64)
        b["col_block"] = np.array(out["col_block"], np.int32)
        b["col_comp"] = np.array(out["col_comp"], np.int32)
        b["col_ijk"] = np.array(out["col_ijk"], np.int32).reshape(-1, 3)
        b["val"] = np.array(out["val"], np.float64)
    if open_row:
        # an interior node nobody shares is replaced by another one: every row
        # of the plan takes the staged route
        w["bcs"].append({"kind": "sync", "block": 0, "lo": (3, 3, 0), "hi": (4, 4, 1),
                         "comps": [0], "row_ptr": np.array([0, 1], np.int64),
                         "col_block": np.zeros(1, np.int32), "col_comp": np.zeros(1, np.int32),
                         "col_ijk": np.array([[2, 3, 0]], np.int32), "val": np.ones(1),
                         "rhs": None})
    return w


KINDS = ["plain", "shuffled", "some", "repeated"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("nlevels", [1, 5])
def test_records_replay_on_the_host(kind, dtype, nlevels):
    w = _grid(kind, dtype, nlevels)
    blocks = [specs.contiguous_block(b) for b in w["blocks"]]
    n, bad, msg = bc.Plan(blocks, specs.submatrices(w), dtype, {"host_only": 1}).check_work()
    assert n > 0 and bad == 0, msg


@pytest.mark.gpu
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("nlevels", [1, 5, 33])
@pytest.mark.parametrize("inner", [False, True])
def test_in_place_against_staged(kind, dtype, nlevels, inner):
    dev = to_device_innermost if inner else to_device
    res = []
    for open_row in (False, True):
        w = _grid(kind, dtype, nlevels, open_row=open_row)
        plan, out = run(w, tensors=dev(w["fields"]))
        res.append((plan, out))
        if kind in ("plain", "shuffled"):
            compare(w, out)
    (closed, a), (staged, b) = res
    same = kind == "repeated"
    assert closed.stats()["launches_fwd"] == staged.stats()["launches_fwd"] - (not same)
    synth.data_view(b[0], w["blocks"][0])[0, :, 0, 3, 3] = \
        synth.data_view(a[0], w["blocks"][0])[0, :, 0, 3, 3]
    assert np.array_equal(bits(flat(a)), bits(flat(b)))


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_values_not_finite(dtype):
    res = []
    for open_row in (False, True):
        w = _grid("some", dtype, 3, open_row=open_row)
        for k, v in ((0, np.inf), (3, np.nan), (4, -np.inf)):
            synth.data_view(w["fields"][k], w["blocks"][k])[:, 1, 0, :, (0, -1)] = v
        _, out = run(w, tensors=to_device(w["fields"]))
        res.append(out)
    a, b = res
    synth.data_view(b[0], w["blocks"][0])[0, :, 0, 3, 3] = \
        synth.data_view(a[0], w["blocks"][0])[0, :, 0, 3, 3]
    assert np.array_equal(flat(a), flat(b), equal_nan=True)

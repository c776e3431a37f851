"""Sync rows that also read a cell no Sync row writes are not in closed
groups: they keep the staged rows and the commit after the ghost kernels."""
import numpy as np
import pytest

from gpu_util import compare, run, to_device_innermost
from paper_2605_14780_gb300 import synth

pytestmark = pytest.mark.gpu


def _open_grid(dtype, nlevels):
    w = synth.sync_grid(3, 2, 9, 2, nlevels, 2, dtype=dtype, seed=9)
    b = next(b for b in w["bcs"] if b["kind"] == "sync")
    b["col_ijk"] = b["col_ijk"].copy()
    b["col_ijk"][0] = (4, 4, 0)  # an interior node
    return w


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("nlevels", [1, 6])
@pytest.mark.parametrize("inner", [False, True])
def test_open_rows(dtype, nlevels, inner):
    w = _open_grid(dtype, nlevels)
    ts = to_device_innermost(w["fields"]) if inner else None
    plan, out = run(w, tensors=ts)
    compare(w, out)
    closed, _ = run(synth.sync_grid(3, 2, 9, 2, nlevels, 2, dtype=dtype, seed=9))
    # the closed rows save the staging launch
    assert plan.stats()["launches_fwd"] == closed.stats()["launches_fwd"] + 1

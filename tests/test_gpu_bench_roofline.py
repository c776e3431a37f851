"""The fused record's roofline counts what the kernel issues: it cannot pass
the part's FP64 rate."""
import pytest

import bench

pytestmark = pytest.mark.gpu


def test_fused_record():
    import torch
    r = bench.measure_fused(torch.device("cuda:0"), torch.cuda.Stream(), 5, 3, nblocks=4)
    assert 0 < r["roofline"]["frac"] <= 1

"""Host replay of the work lists at sizes where staged tiles are cut short:
panels that are not a multiple of a tile, few and many levels, both dtypes,
user interpolation tables along either axis."""
import pytest

from paper_2605_14780_gb300 import bc, specs, synth

CASES = [
    lambda dt: synth.cubed_sphere(11, 3, 4, 3, ("h", "u", "v"), dt, seed=61, quad=2),
    lambda dt: synth.cubed_sphere(34, 2, 4, 9, ("scalar",), dt, seed=62, quad=2),
    lambda dt: synth.cubed_sphere(29, 2, 6, 8, ("h", "u", "v"), dt, seed=63, quad=2),
    lambda dt: synth.staggered_interp(nx=9, ny=37, h=3, nlevels=5, p=6, dtype=dt),
    lambda dt: synth.swap_xy(synth.staggered_interp(nx=7, ny=45, h=2, nlevels=9, p=8, dtype=dt)),
    lambda dt: synth.batching(nblocks=16, side_lo=2, side_hi=40, lev_lo=1, lev_hi=19, h=2,
                              seed=64, dtype=dt)]


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("k", range(len(CASES)))
def test_replay(k, dtype):
    w = CASES[k](dtype)
    blocks = [specs.contiguous_block(b) for b in w["blocks"]]
    for opts in ({}, {"batch_mode": bc.BC_BATCH_SINGLE}, {"level_chunk": 2}):
        plan = bc.Plan(blocks, specs.submatrices(w), w["dtype"], dict(opts, host_only=1))
        n, bad, msg = plan.check_work()
        assert n > 0 and bad == 0, msg

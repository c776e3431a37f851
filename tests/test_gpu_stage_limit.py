"""Threads apply two plans whose launches take different amounts of
dynamic shared memory from one kernel (CTAs of 512 threads in FP64: 128 KB
with staged CSR tiles, 64 KB with tiles of vector pairs only): neither call may
lower the kernel's limit under the other's launch.  The calls are looped in
C, where no interpreter lock spaces them out."""
import ctypes
import shutil
import subprocess
import threading

import numpy as np
import pytest

from gpu_util import bits, flat, to_device
from paper_2605_14780_gb300 import bc, synth

pytestmark = pytest.mark.gpu

LOOP = """
typedef int (*apply_fn)(void*, void*, int, void*);
int loop_apply(apply_fn f, void* plan, void* slots, void* stream, int n) {
  for (int k = 0; k < n; ++k) {
    for (volatile int j = k * 7919 % 997; j > 0; --j) {} /* drift between the threads */
    const int st = f(plan, slots, 0, stream);
    if (st) return st;
  }
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("gcc") is None, reason="needs gcc")
@pytest.mark.parametrize("mode,ctas", [(bc.BC_BATCH_SINGLE, 0), (bc.BC_BATCH_SINGLE, 1),
                                       (bc.BC_BATCH_PERSISTENT, 0)])
def test_two_plans_two_threads(tmp_path, mode, ctas):
    import torch
    assert bc.BC_FORM_BATCHED == 0
    src = tmp_path / "loop.c"
    src.write_text(LOOP)
    so = tmp_path / "loop.so"
    subprocess.run(["gcc", "-O2", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    loop = ctypes.CDLL(str(so)).loop_apply
    loop.argtypes = [ctypes.c_void_p] * 4 + [ctypes.c_int]
    apply = ctypes.cast(bc.load_library().bc_apply_form, ctypes.c_void_p)
    work = [synth.cubed_sphere(16, 3, 4, 8, ("scalar",), "f64", seed=81, quad=2),
            synth.cubed_sphere(16, 3, 6, 8, ("h", "u", "v"), "f64", seed=82)]
    opts = {"threads": 512, "batch_mode": mode, "ctas_per_sm": ctas}
    sides = []
    for w in work * 2:
        ts = to_device(w["fields"])
        plan = bc.plan_for_workload(w, ts, opts)
        plain = bc.plan_for_workload(w, ts, dict(opts, unstaged_rows=1))
        assert plan.stats()["nitems"] != plain.stats()["nitems"]  # it has staged tiles
        stream = torch.cuda.Stream()
        plan.apply(bc.slot_table(ts), stream=stream)
        torch.cuda.synchronize()
        sides.append((plan, ts, bc.slot_table(ts), stream, flat([t.cpu().numpy() for t in ts])))
    torch.cuda.synchronize()
    status = [None] * len(sides)

    def go(k):
        plan, _, table, stream, _ = sides[k]
        torch.cuda.set_device(0)
        status[k] = loop(apply, plan._h, table.data_ptr(), stream.cuda_stream, 20000)

    threads = [threading.Thread(target=go, args=(k,)) for k in range(len(sides))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert status == [0] * len(sides)
    for _, ts, _, _, want in sides:
        assert np.array_equal(bits(flat([t.cpu().numpy() for t in ts])), bits(want))

"""A process that resets its device and builds new contexts gets the same iterates: nothing the
library puts on the device is taken to outlive a reset. The reset has to come from the CUDA
runtime that the library is linked with, so the library's objects are linked once more beside
a function that calls it, and run in a process of their own."""
import glob
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu

RESET = '#include <cuda_runtime.h>\nextern "C" int reset_device() { return (int)cudaDeviceReset(); }\n'

RUN = """
import sys
import numpy as np
sys.path.insert(0, sys.argv[1])
from paper_1709_00803_gb300 import build, igks
build.build = lambda *a, **k: sys.argv[2]
build.LIB = sys.argv[2]
from igks_inputs import fields as F, meshgen as G
m, fl = G.laminar_plate(), F.laminar_plate_flow()

def run(precision):
    ctx = igks.Context(precision=precision)
    s = ctx.mesh_upload(m); ctx.set_flow(s, fl); ctx.init_freestream(s)
    ctx.set_fields(s, F.perturbed_state(m, fl, seed=3, amp=0.02))
    ctx.iterate(2)
    W = ctx.get_fields(s)
    ctx.destroy()
    return W

before = [run(p) for p in (0, 1, 2)]
assert igks.lib().reset_device() == 0
for p in (0, 1, 2):
    assert np.array_equal(run(p), before[p]), p
"""


def test_same_iterates_after_a_device_reset(tmp_path):
    from paper_1709_00803_gb300 import build
    build.build()
    src, so = tmp_path / "reset.cu", tmp_path / "libigks_reset.so"
    src.write_text(RESET)
    objs = sorted(glob.glob(os.path.join(build.OUT_DIR, "*.o")))
    assert len(objs) == len(build.sources())
    subprocess.check_call([build.nvcc(), *build.ARCH, "-shared", "-Xcompiler", "-fPIC", "-o", str(so), str(src), *objs])
    subprocess.run([sys.executable, "-c", RUN, ROOT, str(so)], check=True, timeout=300)

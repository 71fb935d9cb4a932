"""mc_sweep_noalloc in whatever context is current: brick sweeps that take more
than 48 KB of shared memory a block, which a kernel must be let to on each device,
run in a second context of the process as in the first.  (A second device needs
the same and cannot be had here.)  Runs in a process of its own; memory comes
from the driver interface.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import ctypes as C
import numpy as np
import paper_2103_03517_gb300 as mc
cu = C.CDLL("libcuda.so.1")
def ok(r):
    assert r == 0, r
ok(cu.cuInit(0))
ctx = C.c_void_p()
dims = (8192, 8, 4)   # rows of 98 KB: every block needs more than 48 KB
N = 8192 * 32
start = np.zeros((6, N // 2), np.float32)
start[[2, 5]] = 1.0
def run(n):
    d = C.c_uint64()
    ok(cu.cuMemAlloc_v2(C.byref(d), C.c_size_t(start.nbytes)))
    ok(cu.cuMemcpyHtoD_v2(d, start.ctypes.data_as(C.c_void_p), C.c_size_t(start.nbytes)))
    th = mc.mc_sweep_noalloc(d.value, dims, 1.0, 0.02, (0, 0, 1.0), 0.0, (0, 0, 0.1), 0.8, 3, 0, n, 30)
    out = np.empty_like(start)
    ok(cu.cuMemcpyDtoH_v2(out.ctypes.data_as(C.c_void_p), d, C.c_size_t(start.nbytes)))
    ok(cu.cuMemFree_v2(d))
    return th, out
ok(cu.cuDevicePrimaryCtxRetain(C.byref(ctx), 0))
ok(cu.cuCtxSetCurrent(ctx))
a1, a4 = run(1), run(4)
two = C.c_void_p()
ok(cu.cuCtxCreate_v2(C.byref(two), 0, 0))  # and makes it current
for a, b in ((a1, run(1)), (a4, run(4))):
    assert a[0] == b[0] and np.array_equal(a[1], b[1])
print("ok")
"""


def test_brick_sweeps_in_a_second_context():
    from paper_2103_03517_gb300 import build as libbuild
    libbuild.build()
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=120,
                       env=dict(os.environ, PYTHONPATH=ROOT))
    assert r.stdout.strip() == "ok", r.stdout + r.stderr

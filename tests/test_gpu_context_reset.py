"""The library goes on after the caller's device reset: nothing of the former
context is kept by the process or the thread."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes, sys
import numpy as np
sys.path.insert(0, sys.argv[1])
import gen
from paper_2602_05686_gb300 import api
gen.build()
L = api.lib(False)
p = gen.layered_2d(32)
a = [np.ascontiguousarray(p[k]) for k in ("row_ptr", "col", "val", "coords")]
b = np.ascontiguousarray(p["b"])

def solve():
    o = api.default_options()
    o.max_coarse, o.measure = 64, 0
    pr = api.Problem()
    pr.dim, pr.host, pr.n, pr.nnz = 2, 1, p["n"], p["nnz"]
    pr.row_ptr, pr.col, pr.val, pr.coords = [q.ctypes.data for q in a]
    h = ctypes.c_void_p()
    st = L.sa_setup(ctypes.byref(pr), ctypes.byref(o), ctypes.byref(h))
    assert st == 0, (st, L.sa_last_error())
    x, info = np.zeros_like(b), api.SolveInfo()
    assert L.sa_solve(h, b.ctypes.data, x.ctypes.data, 1e-8, ctypes.byref(info)) == 0
    assert L.sa_free(h) == 0
    return x

cu = ctypes.CDLL("libcuda.so.1")
dev = ctypes.c_int()
first = solve()
for _ in range(10):  # more contexts than a thread keeps buffers for
    assert cu.cuDeviceGet(ctypes.byref(dev), 0) == 0 and cu.cuDevicePrimaryCtxReset_v2(dev) == 0
    assert np.array_equal(solve(), first) and np.array_equal(solve(), first)
print("same")
"""


def test_setup_and_solve_after_a_device_reset():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2602_05686_gb300 as sa
    sa.build()
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "same", (r.returncode, r.stdout, r.stderr)

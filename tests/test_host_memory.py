"""A process with little host memory gets an error status from lb_create_grid,
not an abort: the device allocation, which fails first on a machine that
cannot hold the grid (here: one without a GPU), comes before the host
tables, and running out of host memory is LB_ERR_OOM."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes, resource, sys
import paper_1505_03271_gb300 as lb
L = lb.load(build=False)
used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (used + (1 << 30), used + (1 << 30)))
nx, store = int(sys.argv[1]), int(sys.argv[2])
d = lb.lb_grid_desc(nx, 1, float(nx), 1.0, 0, 0, 0.0, 0.0, 0, 0, 0, store, None)
h = ctypes.c_void_p()
print("status", L.lb_create_grid(ctypes.byref(d), ctypes.byref(h)))
"""


@pytest.mark.parametrize("nx,status", [
    (1 << 22, "any"),      # axes 100 MB: the device allocation fails before tables of 2 GB
    (1 << 27, "LB_ERR_OOM")])  # axes 3 GB: no host memory
@pytest.mark.parametrize("store", ["f64", "f32"])
def test_create_grid_returns_a_status(nx, status, store):
    import torch
    if torch.cuda.is_available():
        pytest.skip("needs a machine whose device allocation fails")
    import paper_1505_03271_gb300 as lb
    lb.load()
    r = subprocess.run([sys.executable, "-c", CHILD, str(nx), str(lb.STORE_NAMES[store])], cwd=ROOT,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stderr[-500:])
    got = int(r.stdout.split("status")[1])
    assert got != lb.LB_OK
    if status != "any":
        assert got == getattr(lb, status)

"""Host-only plan queries on a machine with a GPU: none of them creates a context on it."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import ctypes
import paper_1508_01326_gb300 as R
for mode in ("fp64", "mixed", "pair", "exact"):
    for m, n in ((4, 12), (8, 20), (10, 24)):
        assert R.prefix_plan_host(m, n, mode)["tasks"] > 0
R.batch_tasks_host([(4, 12), (8, 20)], mode="fp64")
cu = ctypes.CDLL("libcuda.so.1")
assert cu.cuInit(0) == 0
flags, active = ctypes.c_uint(), ctypes.c_int(-1)
assert cu.cuDevicePrimaryCtxGetState(0, ctypes.byref(flags), ctypes.byref(active)) == 0
print("active", active.value)
"""


def test_host_queries_leave_the_device_alone():
    out = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    assert out.stdout.split()[-2:] == ["active", "0"]

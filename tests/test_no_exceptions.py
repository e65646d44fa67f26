"""No C++ exception crosses the C boundary: host tables that cannot be allocated are DD_ENOMEM."""
import subprocess
import sys

CODE = """
import numpy as np
from paper_2507_00294_gb300 import binding as b, workloads as w
lib = b.load()
scan = b.Scan(w.ScanSpec(8, 8))
t, out = np.zeros(1), np.zeros(1, np.int64)
st = lib.dd_field_grid_split(scan.handle, 0.0, 0.0, 1e-9, 1e-9, 64, 64, t.ctypes.data, 1 << 59, out.ctypes.data, None)
print(st, lib.dd_last_error().decode())
"""


def test_absurd_count_is_an_error():
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-500:]
    assert r.stdout.startswith("-2 dd_field_grid_split")

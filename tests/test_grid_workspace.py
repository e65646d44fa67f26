"""The scratch of an FP32-mixed grid call off the dwell lattice: snapshots are taken in passes whose
tables stay within 1 GiB, also where a visit takes tens of contraction nodes (a grid far wider than the
scan: 4 GiB for all snapshots at once)."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import numpy as np, torch
from paper_2507_00294_gb300 import binding as b, workloads as w
spec = w.ScanSpec(512, 512, D_m2s=6e-14)
p, n, n_t = spec.pitch_m, 512 * 512, 80
times = (n - 0.37 - 1000.0 * np.arange(n_t)) * spec.dwell_s
grid = (0.0, 0.0, 16000 * p, 16000 * p, 64, 64)
scan, out = b.Scan(spec), torch.empty((n_t, 64 * 64), dtype=torch.float64, device="cuda:0")
b.dd_field_on_grid(scan, *grid, times[:1], "mixed", out=out[:1])
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
b.dd_field_on_grid(scan, *grid, times, "mixed", out=out)
torch.cuda.synchronize()
used = free - torch.cuda.mem_get_info()[0]
exact = b.dd_field_on_grid(scan, *grid, times[-1:], "fp64", device="cuda:0")[0]
m = exact > 1e-6 * exact.max()
assert ((out[-1] / exact - 1.0).abs()[m] <= 1e-5).all()
print(used)
"""


def test_tables_within_budget(cuda):
    """Two passes' blocks may be alive at once, and the allocator rounds sizes up."""
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert int(r.stdout.split()[-1]) <= 2.5 * (1 << 30)

"""FP32-mixed grids below 64 columns with many snapshots of more than 256 visits (the final kernel of
dd_grid.cu for every visit, its longest lists split over CTAs), and both sides of the rule that takes them
there, against the FP64 path."""
import numpy as np
import pytest

from paper_2507_00294_gb300 import binding as b
from paper_2507_00294_gb300 import workloads as w
from parity_util import assert_mixed

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cols,rows", [(16, 16), (33, 31), (63, 64)])
@pytest.mark.parametrize("nx,ny,n_t", [(16, 16, 31), (16, 16, 32), (257, 1, 32), (257, 1, 127), (257, 1, 128),
                                       (32, 32, 128), (41, 25, 128)])
def test_many_snapshots(cuda, nx, ny, n_t, cols, rows):
    spec = w.ScanSpec(nx, ny, D_m2s=6e-14)
    p, n = spec.pitch_m, nx * ny
    g = (-0.3 * p, 0.7 * p, 0.9 * p * nx / cols, 0.6 * p, cols, rows)
    scan = b.Scan(spec)
    for off in (0.0, 0.37):
        times = (np.rint(np.linspace(1, n, n_t)) + off) * spec.dwell_s
        mixed = b.dd_field_on_grid(scan, *g, times, "mixed", device=cuda).cpu().numpy()
        exact = b.dd_field_on_grid(scan, *g, times, "fp64", device=cuda).cpu().numpy()
        # (terms with rho^2/w1 >= 87 are below the FP32 range and add 0 in this precision)
        live = exact.max(axis=1) > 1e-37 * spec.Q0 / (4 * np.pi * spec.D_m2s)
        assert live.sum() > n_t // 2
        assert_mixed(mixed[live], exact[live], exact[live].max(axis=1), "%d snapshots" % n_t)

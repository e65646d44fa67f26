"""FP32-mixed grids below 64 columns (dd_grid.cu without the contraction): widths and heights at the
edges of its 32-column, 16-row tiles and of the rule that selects it, against the FP64 path."""
import numpy as np
import pytest

from paper_2507_00294_gb300 import binding as b
from paper_2507_00294_gb300 import workloads as w
from parity_util import assert_mixed

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cols,rows", [(1, 1), (1, 512), (2, 16), (15, 17), (16, 16), (31, 33), (32, 32), (33, 15), (63, 1),
                                       (63, 64), (64, 40)])
@pytest.mark.parametrize("spec", [
    w.ScanSpec(16, 16, D_m2s=6e-14), w.ScanSpec(32, 32, D_m2s=1e-12),         # 1024 visits: only the tallest grid qualifies
    w.ScanSpec(13, 19, order=w.RANDOM, seed=5, keep_fraction=0.8, D_m2s=1e-15)])
def test_narrow_grid(cuda, spec, cols, rows):
    p, n = spec.pitch_m, w.n_visits(spec)
    g = (-0.3 * p, 1.7 * p, 0.45 * p, -0.4 * p if cols == 33 else 0.5 * p, cols, rows)
    # 34 snapshots (tiles enough for the rule), among them an empty one and a late one
    marks = np.concatenate([[0.0, 1.0, 2.0], np.linspace(3, n, 30), [20.0 * n]])
    scan = b.Scan(spec)
    for times in (np.rint(marks), marks + 0.37):
        mixed = b.dd_field_on_grid(scan, *g, times * spec.dwell_s, "mixed", device=cuda).cpu().numpy()
        exact = b.dd_field_on_grid(scan, *g, times * spec.dwell_s, "fp64", device=cuda).cpu().numpy()
        # (terms with rho^2/w1 >= 87 are below the FP32 range and add 0 in this precision)
        live = exact.max(axis=1) > 1e-37 * spec.Q0 / (4 * np.pi * spec.D_m2s)
        assert live.sum() > 20
        assert np.all(mixed[exact.max(axis=1) == 0.0] == 0.0)
        assert_mixed(mixed[live], exact[live], exact[live].max(axis=1), "grid %dx%d" % (cols, rows))

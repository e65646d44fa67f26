"""FP32-mixed grids with thousands of visits outside the contraction's bands ("recent" visits of
dd_grid_quad.cuh): a grid far wider than the scan, on which hardly any visit is smooth everywhere."""
import numpy as np
import pytest

from paper_2507_00294_gb300 import binding as b
from paper_2507_00294_gb300 import workloads as w
from parity_util import assert_mixed

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec_of_time", [0.0, 0.37])
def test_rounding_of_many_recent_visits(cuda, prec_of_time):
    """65,536 recent visits that contribute alike at the 64 points beside them: the sum over 2048
    stages is compensated.  Bound: 2.5e-7 of a term from its series and 2^-24 of a stage's sum, whose
    signs average out over the stages; a plain FP32 sum over them rounds to 6e-7."""
    spec = w.ScanSpec(256, 256, D_m2s=6e-14)
    p, n = spec.pitch_m, 256 * 256
    g = (128.0 * p, 96.0 * p, 66000.0 * p, 1.0 * p, 64, 64)
    times = np.array([4.0 * n + prec_of_time]) * spec.dwell_s
    scan = b.Scan(spec)
    mixed = b.dd_field_on_grid(scan, *g, times, "mixed", device=cuda).cpu().numpy()
    exact = b.dd_field_on_grid(scan, *g, times, "fp64", device=cuda).cpu().numpy()
    assert_mixed(mixed, exact, exact.max(axis=1))
    err = mixed[0, ::64] / exact[0, ::64] - 1.0
    assert np.sqrt(np.mean(err ** 2)) <= 3e-7, (err.mean(), err.std())

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
    exact = b.dd_field_on_grid(scan, *g, times, "fp64", device=cuda).cpu().numpy()
    plan = b.Batch([scan], None, times, "mixed", grids=[g])       # (a single call leaves it to the grid tile)
    for mixed in (b.dd_field_on_grid(scan, *g, times, "mixed", device=cuda), plan.run(device=cuda)[None]):
        mixed = mixed.cpu().numpy()
        assert_mixed(mixed, exact, exact.max(axis=1))
        err = mixed[0, ::64] / exact[0, ::64] - 1.0
        assert np.sqrt(np.mean(err ** 2)) <= 3e-7, (err.mean(), err.std())


def against_fp64(cuda, spec, g, marks):
    scan, p = b.Scan(spec), spec.pitch_m
    grid = (g[0] * p, g[1] * p, g[2] * p, g[3] * p, g[4], g[5])
    times = np.asarray(marks, float) * spec.dwell_s
    mixed = b.dd_field_on_grid(scan, *grid, times, "mixed", device=cuda).cpu().numpy()
    exact = b.dd_field_on_grid(scan, *grid, times, "fp64", device=cuda).cpu().numpy()
    assert_mixed(mixed, exact, exact.max(axis=1), "grid %s" % (g,))
    return scan, grid, times, exact


@pytest.mark.parametrize("n,D", [(256, 1e-16), (257, 1e-16), (320, 1e-16), (321, 1e-16), (4096, 6e-15), (20011, 6e-15),
                                 (4096, 6e-16)])
def test_split_over_ctas(cuda, n, D):
    """Recent visits at the edges of the rule (256) and of a part (64), in one snapshot, several, off the dwell lattice,
    and in a batch; three of them take the grid tile in a single call."""
    spec = w.ScanSpec(n, 1, D_m2s=D)
    g = (0.0, -31.0, max(n / 63.0, 4.0), 1.0, 64, 65)
    scan, grid, times, exact = against_fp64(cuda, spec, g, [float(n)])
    against_fp64(cuda, spec, g, [n - 0.63, 0.5 * n + 0.1, 2.0])
    plan = b.Batch([scan, scan], None, np.repeat(times, 2), "mixed", grids=[grid, grid[:5] + (33,)])
    out = plan.run(device=cuda).cpu().numpy()
    assert_mixed(out[:64 * 65], exact[0], exact.max(), "batch")
    assert_mixed(out[64 * 65:], exact[0, :64 * 33], exact[0, :64 * 33].max(), "batch")


def test_split_segments(cuda):
    """Snapshots of a raster that share their sums (a grid that covers the scan), hundreds of recent
    visits in a segment of lags, beside one that stands alone."""
    spec = w.ScanSpec(64, 96, D_m2s=6e-15)
    scan, grid, times, _ = against_fp64(cuda, spec, (-1000.0, -1.0, 32.0, 1.0, 64, 98),
                                        list(64.0 * np.arange(16, 97, 16)) + [3001.0])
    b.dd_profile_reset()
    b.dd_profile_enable(True)
    try:
        b.dd_field_on_grid(scan, *grid, times, "mixed", device=cuda)
    finally:
        b.dd_profile_enable(False)
    assert "field_reduce" in b.dd_profile_read()

"""Snapshots of a raster that share their sums by a shift of whole scan rows (dd_grid_quad.cuh):
phases, gaps, repeats, rows of several heights per pitch and snapshots past the scan's end, against
the FP64 path; and grids that do not cover the scan or whose rows do not fall on the scan's, which
sum every snapshot by itself."""
import numpy as np
import pytest

from paper_2507_00294_gb300 import binding as b
from paper_2507_00294_gb300 import workloads as w
from parity_util import assert_mixed

pytestmark = pytest.mark.gpu


def on_grid(spec, g, dwells, cuda):
    scan, p = b.Scan(spec), spec.pitch_m
    grid = (g[0] * p, g[1] * p, g[2] * p, g[3] * p, g[4], g[5])
    times = np.asarray(dwells, float) * spec.dwell_s
    b.dd_profile_reset()
    b.dd_profile_enable(True)
    try:
        mixed = b.dd_field_on_grid(scan, *grid, times, "mixed", device=cuda).cpu().numpy()
    finally:
        b.dd_profile_enable(False)
    names = b.dd_profile_read()
    exact = b.dd_field_on_grid(scan, *grid, times, "fp64", device=cuda).cpu().numpy()
    live = exact.max(axis=1) > 1e-37 * spec.Q0 / (4 * np.pi * spec.D_m2s)
    assert live.any()
    assert np.all(mixed[exact.max(axis=1) == 0.0] == 0.0)
    assert_mixed(mixed[live], exact[live], exact[live].max(axis=1), "grid %s" % (g,))
    return names


@pytest.mark.parametrize("grid", [
    (0.0, 0.0, 0.5, 0.5, 64, 64), (-3.0, 1.0, 0.3, 1.0, 129, 33), (10.0, 5.3, -0.25, 0.25, 80, 130),
    (0.1, 0.2, 0.37, 1.0 / 3.0, 127, 129), (0.0, -40.0, 1.0, 1.0, 64, 64),
    (-0.1, 0.0, 0.37, 1.0 / 3.0, 127, 129), (35.0, -2.5, -0.5, 0.5, 80, 131), (-9.0, -1.0, 1.0, 1.0, 64, 72)])
@pytest.mark.parametrize("nx,ny,D", [(32, 24, 6e-14), (17, 40, 1e-12), (33, 31, 1e-15)])
def test_groups(cuda, nx, ny, D, grid):
    spec = w.ScanSpec(nx, ny, D_m2s=D)
    n = nx * ny
    rows = nx * np.arange(1, ny + 1)
    dwells = np.concatenate([rows, rows[::3] - 1, rows[:-1:2] + 5, [0, 1, n, 2 * n]])   # three phases; one twice
    np.random.default_rng(1).shuffle(dwells)
    x = sorted((grid[0], grid[0] + (grid[4] - 1) * grid[2]))
    covers = x[0] <= 0 and x[1] >= nx - 1 and grid[1] <= 0 and grid[1] + (grid[5] - 1) * grid[3] >= ny - 1
    assert ("field_reduce" in on_grid(spec, grid, dwells, cuda)) == covers


@pytest.mark.parametrize("grid,order", [((0.0, 0.0, 0.5, -0.5, 64, 64), w.RASTER), ((0.0, 0.0, 0.5, 0.45, 64, 64), w.RASTER),
                                        ((0.0, 0.0, 0.5, 2.0, 64, 64), w.RASTER),
                                        ((0.0, 0.0, 0.5, 0.5, 64, 64), w.SERPENTINE)])
def test_not_shared(cuda, grid, order):
    spec = w.ScanSpec(32, 24, order=order, D_m2s=6e-14)
    assert "field_reduce" not in on_grid(spec, grid, 32 * np.arange(1, 25), cuda)


def test_few_snapshots_far_apart(cuda):
    """Two snapshots of one phase gain nothing from sharing."""
    spec = w.ScanSpec(32, 64, D_m2s=6e-14)
    assert "field_reduce" not in on_grid(spec, (0.0, 0.0, 0.5, 0.5, 64, 64), [32, 2048], cuda)

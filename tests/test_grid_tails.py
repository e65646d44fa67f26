"""FP32-mixed grids far below the field's peak: the contraction (dd_grid_quad.cuh) keeps FP32's relative
accuracy at every point, in single calls, snapshots that share their sums, and batches; and sums of few
visits carry no correction for what full stages of MMAs lose."""
import numpy as np
import pytest

from paper_2507_00294_gb300 import binding as b
from paper_2507_00294_gb300 import workloads as w

pytestmark = pytest.mark.gpu


def relative_errors(mixed, exact, floor):
    m = exact >= floor * exact.max(axis=-1, keepdims=True)
    return np.abs(mixed[m] / exact[m] - 1.0)


# A term's exponent reaches 83 (in powers of two) at 1e-25 of the peak; its FP32 rounding and that of
# the squared distance are 2^-23 of that together: 83 ln2 2^-23 = 7e-6, and twice that for a product of two factors.
TAIL, RTOL = 1e-25, 1.5e-5


@pytest.mark.parametrize("spec", [
    w.ScanSpec(64, 64, D_m2s=1e-15), w.ScanSpec(64, 64, D_m2s=6e-14), w.ScanSpec(40, 90, order=w.SERPENTINE, D_m2s=2e-14),
    w.ScanSpec(64, 64, order=w.RANDOM, seed=3, keep_fraction=0.5, D_m2s=1e-14)])
def test_tail(cuda, spec):
    p, n = spec.pitch_m, w.n_visits(spec)
    g = (0.0, 0.0, 0.5 * p, 0.5 * p, 2 * spec.nx, 2 * spec.ny)
    scan = b.Scan(spec)
    for marks in ([0.02 * n, 0.5 * n, n, 5.0 * n], spec.nx * np.arange(1.0, spec.ny + 1, 3)):
        for off in (0.0, 0.37):
            times = (np.rint(marks) + off) * spec.dwell_s
            mixed = b.dd_field_on_grid(scan, *g, times, "mixed", device=cuda).cpu().numpy()
            exact = b.dd_field_on_grid(scan, *g, times, "fp64", device=cuda).cpu().numpy()
            assert relative_errors(mixed, exact, TAIL).max() <= RTOL
    plan = b.Batch([scan, scan], None, times[:2], "mixed", grids=[g, g])
    out = plan.run(device=cuda).cpu().numpy().reshape(2, -1)
    assert relative_errors(out, exact[:2], TAIL).max() <= RTOL


@pytest.mark.parametrize("n", [4, 16, 48, 64, 80, 128, 512])
def test_mean_error_of_few_visits(cuda, n):
    """Visits that contribute alike: the mean error is at most half of 2^-22, the largest factor that puts
    back what four MMAs lose (a sum of one to three MMAs loses less than 2^-24)."""
    spec = w.ScanSpec(n, 1, D_m2s=6e-14)
    p = spec.pitch_m
    g = (0.0, -32.0 * p, n / 64.0 * p, p, 64, 64)
    times = np.array([3e5, 1e6, 3e6]) * spec.dwell_s
    scan = b.Scan(spec)
    mixed = b.dd_field_on_grid(scan, *g, times, "mixed", device=cuda).cpu().numpy()
    exact = b.dd_field_on_grid(scan, *g, times, "fp64", device=cuda).cpu().numpy()
    assert abs((mixed / exact - 1.0).mean()) <= 2.0 ** -23

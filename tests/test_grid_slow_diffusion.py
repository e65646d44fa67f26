"""FP32-mixed grids where most visits lie far outside the FP32 range of a term (q rho^2 past 2^25):
hardly any diffusion on a large scan, a very narrow probe, and a grid far from the scan.  Such a visit
adds nothing, whatever its exponent's rounding; single calls, snapshots that share their sums, and
batches, against the FP64 path."""
import numpy as np
import pytest

from paper_2507_00294_gb300 import binding as b
from paper_2507_00294_gb300 import workloads as w
from parity_util import assert_mixed

pytestmark = pytest.mark.gpu

NM = 1e-9
# (scan, grid in pitches, snapshots in dwells)
LARGE = (w.ScanSpec(512, 512, pitch_m=NM, sigma_m=0.05 * NM, D_m2s=1e-22), (0.0, 384.0, 1.0, 1.0, 512, 128), [262144.0])
NARROW = (w.ScanSpec(150, 130, pitch_m=NM, sigma_m=0.004 * NM, D_m2s=1e-22), (0.0, 0.0, 1.0, 1.0, 150, 130),
          [4500.37, 19500.0])
SHARED = (w.ScanSpec(150, 130, pitch_m=NM, sigma_m=0.004 * NM, D_m2s=1e-22), (0.0, 0.0, 1.0, 1.0, 150, 130),
          list(150.0 * np.arange(10, 131, 10)))


def si(spec, g):
    return (g[0] * spec.pitch_m, g[1] * spec.pitch_m, g[2] * spec.pitch_m, g[3] * spec.pitch_m, g[4], g[5])


def check(mixed, exact, what):
    assert np.all(np.isfinite(mixed)), what
    assert_mixed(mixed, exact, exact.max(axis=-1), what)


@pytest.mark.parametrize("case", [LARGE, NARROW, SHARED], ids=["large", "narrow", "shared"])
def test_single(cuda, case):
    spec, grid, marks = case
    scan, g, times = b.Scan(spec), si(spec, grid), np.array(marks) * spec.dwell_s
    mixed = b.dd_field_on_grid(scan, *g, times, "mixed", device=cuda).cpu().numpy()
    exact = b.dd_field_on_grid(scan, *g, times, "fp64", device=cuda).cpu().numpy()
    check(mixed, exact, "single")


def test_batch(cuda):
    cases = [LARGE, NARROW, (NARROW[0].with_(order=w.RANDOM, seed=2, keep_fraction=0.5), NARROW[1], [9000.0])]
    scans = [b.Scan(c[0]) for c in cases]
    times = np.array([c[2][-1] * c[0].dwell_s for c in cases])
    plan = b.Batch(scans, None, times, "mixed", grids=[si(c[0], c[1]) for c in cases])
    out = plan.run(device=cuda).cpu().numpy()
    for k, c in enumerate(cases):
        exact = b.dd_field_on_grid(scans[k], *si(c[0], c[1]), times[k:k + 1], "fp64", device=cuda).cpu().numpy()
        check(out[plan.offsets[k]:plan.offsets[k + 1]][None], exact, "scan %d" % k)


@pytest.mark.parametrize("x0,y0", [(1e6, 0.0), (0.0, -1e6), (3e6, 2e6)])
def test_far_grid(cuda, x0, y0):
    """A grid a million pitches from the scan, long after it: every term is below e^-745."""
    spec = w.ScanSpec(64, 64, D_m2s=1e-15)
    got = b.dd_field_on_grid(b.Scan(spec), *si(spec, (x0, y0, 1.0, 1.0, 64, 64)), np.array([1e6, 3e6]) * spec.dwell_s,
                             "mixed", device=cuda).cpu().numpy()
    assert np.all(got == 0.0)

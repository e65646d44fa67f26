"""Point lists of FP32-mixed calls that the caller already gave in compact runs keep their order
(dd_sort_points.cuh): row-major lists, runs of other shapes, a list that is compact in some blocks only,
and points on a line, against the FP64 path."""
import numpy as np
import pytest

from paper_2507_00294_gb300 import binding as b
from paper_2507_00294_gb300 import workloads as w
from parity_util import assert_mixed

pytestmark = pytest.mark.gpu


def lists():
    rng = np.random.default_rng(5)
    r, c = np.divmod(np.arange(128 * 65), 128)
    grid = np.stack([c * 0.5, r * 0.97], 1)
    return {"row-major": grid[:128 * 64], "ragged": grid[:8191], "half shuffled": np.concatenate([grid[:4096], rng.permutation(grid[4096:])]),
            "line": np.stack([np.linspace(0, 60, 5003), np.full(5003, 7.3)], 1), "one place": np.full((4097, 2), 11.25),
            "far run": np.concatenate([grid[:2048], grid[:2050] + 1e7])}


@pytest.mark.parametrize("name", lists())
def test_lists(cuda, name):
    import torch
    pts = lists()[name]
    spec = w.ScanSpec(64, 64, order=w.RANDOM, seed=4, keep_fraction=0.8)
    n = w.n_visits(spec)
    scan = b.Scan(spec)
    xy = torch.from_numpy(pts * spec.pitch_m).to(cuda)
    times = (np.linspace(0.1, 1.0, 36) * n + 0.4) * spec.dwell_s           # enough pairs to look at the order
    mixed = b.dd_field_at_times(scan, xy, times, "mixed").cpu().numpy()
    exact = b.dd_field_at_times(scan, xy, times[::7], "fp64").cpu().numpy()
    assert_mixed(mixed[::7], exact, exact.max(axis=1), name)


def test_kept_order_in_batches(cuda):
    """A plan over a row-major list and the same points shuffled."""
    import torch
    pts = lists()["row-major"]
    spec = w.ScanSpec(40, 36, order=w.RANDOM, seed=2, keep_fraction=0.6)
    p = np.random.default_rng(1).permutation(len(pts))
    scans, end = [b.Scan(spec), b.Scan(spec)], np.full(2, w.n_visits(spec) * spec.dwell_s)
    offs = [0, len(pts), 2 * len(pts)]
    xy = torch.from_numpy(np.concatenate([pts, pts[p]]) * spec.pitch_m).to(cuda)
    mixed = b.Batch(scans, offs, end, "mixed").run(xy).cpu().numpy().reshape(2, -1)
    exact = b.Batch(scans, offs, end, "fp64").run(xy).cpu().numpy().reshape(2, -1)
    assert_mixed(mixed, exact, exact.max(axis=1), "batch")

"""Small field calls, whose visit blocks shrink to one 32-visit stage until the launch fills the
GPU: scans around one and two stages, few points and snapshots, against the oracle."""
import numpy as np
import pytest

from paper_2507_00294_gb300 import binding as b
from paper_2507_00294_gb300 import workloads as w
from parity_util import assert_fp64, assert_mixed, oracle_pairs, peak_lower_bound

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(1, 1), (31, 1), (8, 4), (3, 11), (21, 3), (13, 5), (32, 31)])
@pytest.mark.parametrize("n_pts", [1, 130, 700])
def test_small(cuda, nx, ny, n_pts):
    import torch
    spec = w.ScanSpec(nx, ny, order=w.INTERLEAVED if nx * ny > 900 else w.RASTER, interleave_stride=3, D_m2s=3e-13)
    n = w.n_visits(spec)
    rng = np.random.default_rng(n + n_pts)
    pts = rng.uniform(-1, max(nx, ny), (n_pts, 2)) * spec.pitch_m
    for times in (np.array([1.0, n, 3.0 * n]), np.array([0.5 * n + 0.3])):
        times = times * spec.dwell_s
        ip, it = w.sample_pairs(n_pts, len(times), 200, seed=2)
        ref = oracle_pairs(spec, pts, times, ip, it)
        for prec, check in (("mixed", None), ("fp64", assert_fp64)):
            got = b.dd_field_at_times(b.Scan(spec), torch.from_numpy(pts).to(cuda), times, prec).cpu().numpy()[it, ip]
            if check:
                check(got, ref, "small fp64")
            else:
                assert_mixed(got, ref, peak_lower_bound(spec, times)[it], "small mixed")

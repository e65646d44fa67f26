"""FP32-mixed point lists are evaluated in spatial order and written back in the caller's
(dd_sort_points.cuh): list lengths around the warp, the tile and the sorting block, scattered,
repeated and far-off points, against the oracle and against the same points in another order."""
import numpy as np
import pytest

from paper_2507_00294_gb300 import binding as b
from paper_2507_00294_gb300 import workloads as w
from parity_util import assert_mixed, oracle_pairs, peak_lower_bound

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_pts", [256, 257, 511, 512, 513, 4095, 4096, 4097, 5000, 9001])
def test_scattered_list(cuda, n_pts):
    import torch
    spec = w.ScanSpec(64, 64, order=w.RANDOM, seed=4, keep_fraction=0.8)
    n = w.n_visits(spec)
    rng = np.random.default_rng(n_pts)
    pts = rng.uniform(-2, 65, (n_pts, 2)) * spec.pitch_m
    pts[: n_pts // 8] = np.rint(pts[: n_pts // 8] / spec.pitch_m) * spec.pitch_m      # on probes, some repeated
    pts[-1] = (400 * spec.pitch_m, -300 * spec.pitch_m)
    n_t = max(3, int(np.ceil(3.6e8 / (n_pts * n))))                      # enough pairs to be sorted
    for times in (np.rint(np.linspace(0.2, 1.0, n_t) * n), np.linspace(0.2, 1.3, n_t) * n + 0.4):
        times = times * spec.dwell_s
        scan = b.Scan(spec)
        out = b.dd_field_at_times(scan, torch.from_numpy(pts).to(cuda), times, "mixed").cpu().numpy()
        ip, it = w.sample_pairs(n_pts, len(times), 400, seed=1)
        assert_mixed(out[it, ip], oracle_pairs(spec, pts, times, ip, it), peak_lower_bound(spec, times)[it], "sorted list")
        # another order of the same points: other warps, so other series degrees, within the sum
        # of the two results' tolerances
        p = rng.permutation(n_pts)
        again = b.dd_field_at_times(scan, torch.from_numpy(pts[p]).to(cuda), times, "mixed").cpu().numpy()
        m = out[:, p] >= 1e-6 * out.max(axis=1, keepdims=True)
        np.testing.assert_allclose(again[m], out[:, p][m], rtol=2e-5)


def test_batch_lists_of_uneven_length(cuda):
    import torch
    rng = np.random.default_rng(2)
    counts = [0, 1, 31, 997, 513, 4096, 5001, 128, 0]
    specs = [w.ScanSpec(40, 36, order=w.RANDOM, seed=k, keep_fraction=0.6, D_m2s=10 ** rng.uniform(-14, -12))
             for k in range(len(counts))]
    lists = [rng.uniform(0, 39, (c, 2)) * specs[0].pitch_m for c in counts]
    offs = np.concatenate([[0], np.cumsum(counts)])
    times = np.array([w.n_visits(s) * s.dwell_s for s in specs])
    scans = [b.Scan(s) for s in specs]
    pts = torch.from_numpy(np.concatenate(lists)).to(cuda)
    got = b.Batch(scans, offs, times, "mixed").run(pts).cpu().numpy()
    ref = b.Batch(scans, offs, times, "fp64").run(pts).cpu().numpy()
    for k, c in enumerate(counts):
        if c:
            s = slice(offs[k], offs[k + 1])
            assert_mixed(got[s], ref[s], ref[s].max(), "scan %d" % k)

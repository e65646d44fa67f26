"""A grid batch with a side past the contraction's 32-bit tile numbers (dd_grid.h): the most points a
plan takes in one row, beside an ordinary grid, at seeded points against the oracle."""
import numpy as np
import pytest

from paper_2507_00294_gb300 import binding as b
from paper_2507_00294_gb300 import workloads as w
from parity_util import assert_mixed, oracle_field

pytestmark = pytest.mark.gpu


def test_widest_row(cuda):
    import torch
    if torch.cuda.mem_get_info()[0] < 190 << 30:
        pytest.skip("needs 190 GiB of free device memory")
    spec = w.ScanSpec(3, 2, D_m2s=6e-14)
    p, few = spec.pitch_m, 10 * 6
    wide = (1 << 31) - few
    grids = [(-0.2 * p, 0.1 * p, 0.3 * p, 0.3 * p, 10, 6), (-p, 0.3 * p, 6.0 * p / wide, p, wide, 1)]
    times = np.array([6.0, 5.5]) * spec.dwell_s
    scans = [b.Scan(spec) for _ in grids]
    plan = b.Batch(scans, None, times, "mixed", grids=grids)
    out = plan.run(device=cuda)
    at = np.concatenate([[0, 1, wide // 2, 1 << 30, wide - 1], np.random.default_rng(3).integers(0, wide, 40)])
    got = out[torch.from_numpy(at + few).to(cuda)].cpu().numpy()
    first = out[:few].cpu().numpy()
    del out
    plan.close()
    x0, y0, dx = grids[1][:3]
    ref = oracle_field(spec, np.stack([at * dx + x0, np.full(len(at), y0)], 1), times[1:])[0]
    assert_mixed(got, ref, ref.max(), "wide row")
    r, c = np.divmod(np.arange(few), 10)
    x0, y0, dx, dy = grids[0][:4]
    ref = oracle_field(spec, np.stack([c * dx + x0, r * dy + y0], 1), times[:1])[0]
    assert_mixed(first, ref, ref.max(), "beside it")
    torch.cuda.empty_cache()

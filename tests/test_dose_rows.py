"""The row-invariant dose of whole raster and serpentine scans (dd_dose_rows.cuh) against the
oracle and, through the same visits as a custom order (which takes the direct sum), against the
direct path: rows below, at and past the 128-target tile and the 32-visit staging, few and many
rows, and ranges of targets."""
import numpy as np
import pytest

from paper_2507_00294_gb300 import binding as b
from paper_2507_00294_gb300 import workloads as w
from parity_util import assert_fp64, assert_mixed, oracle_dose

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [w.RASTER, w.SERPENTINE])
@pytest.mark.parametrize("nx,ny,D", [(2, 2, 6e-14), (3, 40, 1e-12), (31, 33, 1e-15), (32, 2, 6e-14), (33, 5, 6e-14),
                                     (128, 3, 6e-14), (129, 4, 1e-15), (300, 2, 1e-12), (5, 300, 6e-14)])
def test_dose_rows(cuda, order, nx, ny, D):
    spec = w.ScanSpec(nx, ny, order=order, D_m2s=D)
    scan = b.Scan(spec)
    direct = b.Scan(spec.with_(order=w.CUSTOM, custom_visit=scan.visits()[0]))
    n = nx * ny
    ref = oracle_dose(spec)
    g64 = b.dd_per_probe_dose(scan, "fp64", device=cuda).cpu().numpy()
    assert g64[0] == 0.0
    assert_fp64(g64, ref, "rows fp64")
    # both sides within 1e-12 of the exact sum, so within twice that of each other
    d64 = b.dd_per_probe_dose(direct, "fp64", device=cuda).cpu().numpy()
    m = ref > 1e-290
    np.testing.assert_allclose(g64[m], d64[m], rtol=2e-12, atol=0)
    gm = b.dd_per_probe_dose(scan, "mixed", device=cuda).cpu().numpy()
    assert gm[0] == 0.0
    assert_mixed(gm[1:], ref[1:], ref.max(), "rows mixed")
    for j0, j1 in ((0, n - 1), (1, n), (n // 3, n // 3 + nx + 1), (n - 1, n)):
        for prec, whole in (("fp64", g64), ("mixed", gm)):
            part = b.dd_per_probe_dose_range(scan, j0, j1, prec, device=cuda).cpu().numpy()
            rtol = 2e-12 if prec == "fp64" else 2e-5
            k = whole[j0:j1] > (1e-290 if prec == "fp64" else 1e-6 * whole.max())
            np.testing.assert_allclose(part[k], whole[j0:j1][k], rtol=rtol, atol=0)


def test_dose_rows_host_output(cuda):
    spec = w.ScanSpec(20, 20)
    scan = b.Scan(spec)
    host = b.dd_per_probe_dose(scan, "fp64")
    np.testing.assert_array_equal(host, b.dd_per_probe_dose(scan, "fp64", device=cuda).cpu().numpy())

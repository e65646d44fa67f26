"""The dose of rasters whose rows are longer than one chunk of 256 terms (dd_dose_rows.cuh), and of
single rows, against the oracle and the direct sum of the same visits in a custom order: rows at the
edges of a chunk, and ranges of targets."""
import numpy as np
import pytest

from paper_2507_00294_gb300 import binding as b
from paper_2507_00294_gb300 import workloads as w
from parity_util import assert_fp64, assert_mixed, oracle_dose

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [w.RASTER, w.SERPENTINE])
@pytest.mark.parametrize("nx,ny", [(256, 3), (257, 3), (258, 2), (511, 2), (512, 2), (513, 3), (1025, 2), (4096, 1), (1, 300)])
def test_wide_rows(cuda, order, nx, ny):
    # a pitch of 2^-31 m: the oracle's SI coordinates are then exact (at 0.5 nm their rounding, 2^-53 of
    # a position against a distance of one pitch, moves its dose by 1.4e-12 at the end of 4096 visits)
    spec = w.ScanSpec(nx, ny, pitch_m=2.0 ** -31, order=order, D_m2s=6e-14)
    scan, n = b.Scan(spec), nx * ny
    direct = b.Scan(spec.with_(order=w.CUSTOM, custom_visit=scan.visits()[0]))
    ref = oracle_dose(spec)
    g64 = b.dd_per_probe_dose(scan, "fp64", device=cuda).cpu().numpy()
    gm = b.dd_per_probe_dose(scan, "mixed", device=cuda).cpu().numpy()
    assert g64[0] == 0.0 and gm[0] == 0.0
    assert_fp64(g64, ref, "fp64")
    assert_mixed(gm[1:], ref[1:], ref.max(), "mixed")
    d64 = b.dd_per_probe_dose(direct, "fp64", device=cuda).cpu().numpy()
    np.testing.assert_allclose(g64[1:], d64[1:], rtol=2e-12, atol=0)
    for j0, j1 in ((0, nx), (0, max(nx - 7, 2)), (n // 3, min(n, n // 3 + nx + 1)), (n - 2, n)):
        for prec, whole, rtol in (("fp64", g64, 2e-12), ("mixed", gm, 2e-5)):
            part = b.dd_per_probe_dose_range(scan, j0, j1, prec, device=cuda).cpu().numpy()
            np.testing.assert_allclose(part, whole[j0:j1], rtol=rtol, atol=0)

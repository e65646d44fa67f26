"""The Gauss-Legendre contraction of the FP32-mixed grid field (dd_grid_quad.cuh): the node bands'
stated limits on the CPU, and the kernel at the edges of its tiles, pieces and bands against the
FP64 path."""
import re
from pathlib import Path

import numpy as np
import pytest

from paper_2507_00294_gb300 import binding as b
from paper_2507_00294_gb300 import workloads as w
from parity_util import assert_mixed

SRC = Path(b.__file__).parent / "csrc" / "dd_grid_quad.cuh"


def bands():
    text = SRC.read_text()
    row = {n: [float(v) for v in re.search(r"%s\[kGqBands\] = \{([^}]*)\}" % n, text).group(1).split(",")]
           for n in ("kGqNodes", "kGqH", "kGqR")}
    return [(int(n), h, r) for n, h, r in zip(row["kGqNodes"], row["kGqH"], row["kGqR"])]


def gauss(n):
    u, c = np.polynomial.legendre.leggauss(n)
    return (u + 1) / 2, c / 2


@pytest.mark.parametrize("n,h_max,r_max", bands())
def test_band_limits(n, h_max, r_max):
    """n nodes give int_0^L exp(-a e^y) dy, L = ln(1 + r), to 1e-7 for every h = a r up to the
    band's limit and every r up to its limit (against 300 nodes)."""
    (u, c), (U, C) = gauss(n), gauss(300)
    for r in np.geomspace(1e-6, r_max, 12):
        L = np.log1p(r)
        a = np.geomspace(1e-3, 1.0, 40)[:, None] * h_max / r
        got = (np.exp(-a * np.expm1(L * u)) * c).sum(1)
        ref = (np.exp(-a * np.expm1(L * U)) * C).sum(1)
        assert np.abs(got / ref - 1).max() <= 1.0e-7 * 1.001


def test_rule_constants():
    """The device's nodes and weights are Gauss-Legendre's, in FP32."""
    text = SRC.read_text()
    body = text[text.index("kGqRule = {"):]
    lists = [[float(v.rstrip("f")) for v in re.findall(r"[-+0-9.e]+f", part)]
             for part in re.findall(r"\{([^{}]*)\}", body)[:2]]
    u = np.concatenate([gauss(n)[0] for n, _, _ in bands()])
    c = np.concatenate([gauss(n)[1] for n, _, _ in bands()])
    np.testing.assert_allclose(lists[0], u, rtol=1e-7, atol=0)
    np.testing.assert_allclose(lists[1], c, rtol=1e-7, atol=0)


# grids in units of the pitch: (x0, y0, dx, dy, columns, rows)
GRIDS = [
    (0.0, 0.0, 0.5, 0.5, 64, 64), (0.0, 0.0, 0.5, 0.5, 128, 32), (-3.0, 1.0, 0.3, 0.7, 129, 33),
    (0.0, 0.0, 0.25, 0.25, 257, 130), (10.0, 5.0, -0.25, 0.5, 80, 52), (0.1, 0.2, 0.37, 0.41, 127, 129),
    (60.0, 0.0, 0.5, 0.5, 64, 64),            # beside the scan: every column far from every visit
    (0.0, 24.0, 1.0, 1.0, 64, 64),
]


@pytest.mark.gpu
@pytest.mark.parametrize("grid", GRIDS)
@pytest.mark.parametrize("spec", [
    w.ScanSpec(32, 24, D_m2s=6e-14), w.ScanSpec(31, 27, order=w.RANDOM, seed=3, keep_fraction=0.7, D_m2s=1e-12),
    w.ScanSpec(40, 20, order=w.INTERLEAVED, interleave_stride=4, D_m2s=1e-15)])
def test_tiles_and_bands(cuda, spec, grid):
    p = spec.pitch_m
    g = (grid[0] * p, grid[1] * p, grid[2] * p, grid[3] * p, grid[4], grid[5])
    n = w.n_visits(spec)
    # 1 visit, one node row and piece borders, part of the scan, its end and long after; off the
    # dwell lattice in the second call
    marks = np.array([1.0, 17.0, 65.0, 0.5 * n, float(n), 20.0 * n])
    scan = b.Scan(spec)
    for times in (np.rint(marks), marks + 0.41):
        mixed = b.dd_field_on_grid(scan, *g, times * spec.dwell_s, "mixed", device=cuda).cpu().numpy()
        exact = b.dd_field_on_grid(scan, *g, times * spec.dwell_s, "fp64", device=cuda).cpu().numpy()
        # terms with rho^2/w1 >= 87 are below the FP32 range and add 0 in this precision: a snapshot
        # that holds no others has no relative accuracy to check
        live = exact.max(axis=1) > 1e-37 * spec.Q0 / (4 * np.pi * spec.D_m2s)
        assert live.any()
        assert_mixed(mixed[live], exact[live], exact[live].max(axis=1), "grid %s" % (grid,))


@pytest.mark.gpu
def test_host_output_and_empty_snapshots(cuda):
    spec = w.ScanSpec(24, 24)
    g = (0.0, 0.0, spec.pitch_m / 3, spec.pitch_m / 3, 72, 66)
    times = np.array([-1.0, 0.0, 100.0, 576.0]) * spec.dwell_s
    scan = b.Scan(spec)
    host = b.dd_field_on_grid(scan, *g, times, "mixed")
    np.testing.assert_array_equal(host, b.dd_field_on_grid(scan, *g, times, "mixed", device=cuda).cpu().numpy())
    assert np.all(host[:2] == 0.0)


@pytest.mark.gpu
def test_batch_of_uneven_grids(cuda):
    """One plan over grids from a single point to several tiles."""
    spec = w.ScanSpec(20, 20, D_m2s=1e-13)
    p = spec.pitch_m
    grids = [(0.0, 0.0, p, p, c, r) for c, r in ((1, 1), (1, 40), (40, 1), (5, 3), (16, 17), (130, 20), (20, 140), (0, 5))]
    scans = [b.Scan(spec) for _ in grids]
    times = np.full(len(grids), 380.0) * spec.dwell_s
    mixed = b.Batch(scans, None, times, "mixed", grids=grids)
    got = mixed.run(device=cuda).cpu().numpy()
    ref = b.Batch(scans, None, times, "fp64", grids=grids).run(device=cuda).cpu().numpy()
    for k in range(len(grids) - 1):
        part = slice(mixed.offsets[k], mixed.offsets[k + 1])
        assert_mixed(got[part], ref[part], ref[part].max(), "grid %d" % k)

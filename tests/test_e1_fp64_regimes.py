"""FP64 pair terms around the borders of their regimes (the moment series up to h = 1/2, the Ein
series up to 2, the rational of x e^x E1(x) above, h = 40 where E1(b) is dropped; the moments'
forward and downward recurrences around r = 0.4): single-visit fields at radii that sweep a and b
over every border, against the oracle."""
import numpy as np
import pytest

from paper_2507_00294_gb300 import binding as b
from paper_2507_00294_gb300 import workloads as w
from parity_util import assert_fp64, oracle_field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [1e-15, 6e-14, 1e-12, 1e-11])
@pytest.mark.parametrize("age", [0.3, 1.0, 1.5, 2.0, 3.0, 3.4, 3.6, 7.0, 60.0])
def test_single_visit_radii(cuda, D, age):
    import torch
    spec = w.ScanSpec(1, 1, D_m2s=D)
    s, kappa = (spec.sigma_m / spec.pitch_m) ** 2, D * spec.dwell_s / spec.pitch_m ** 2
    w1 = 2 * s + 4 * kappa * age
    w0 = w1 - 4 * kappa * min(age, 1.0)
    a = np.concatenate([np.geomspace(1e-6, 600.0, 600), 2.0 * w0 / w1 * (1 + np.array([-1e-9, 1e-9])),
                        2.0 * (1 + np.array([-1e-9, 1e-9])), 0.5 * w0 / (w1 - w0) * (1 + np.array([-1e-9, 1e-9])),
                        40.0 * w0 / (w1 - w0) * (1 + np.array([-1e-9, 1e-9]))])
    rho = np.sqrt(a[a <= 600.0] * w1) * spec.pitch_m
    pts = np.stack([rho * 0.6, rho * 0.8], axis=1)
    times = np.array([age]) * spec.dwell_s
    out = b.dd_field_at_times(b.Scan(spec), torch.from_numpy(pts).to(cuda), times, "fp64").cpu().numpy()
    assert_fp64(out, oracle_field(spec, pts, times), "single visit")

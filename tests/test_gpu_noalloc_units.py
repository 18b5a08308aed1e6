"""sdpd_density_noalloc in any unit of length: the same particle set in units
2^80 times larger and smaller has the same density per volume and the same
pressure (r_c^2 then leaves the range of FP32, in which candidates are tested)."""
import numpy as np
import pytest

from paper_2002_03120_gb300 import binding as B
from paper_2002_03120_gb300 import cases

from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def _run(scale, periodic):
    import torch
    p = cases.base_params(dx=1e-3)
    p.update(box=[0.013, 0.033, 0.012], periodic=periodic, origin=[0.5e-3, -2e-3, 0.0])
    x = np.asarray(p["origin"]) + np.asarray(p["box"]) * np.random.default_rng(2).uniform(size=(4001, 3))
    for key in ("dx", "r_c"):
        p[key] *= scale
    for key in ("box", "origin"):
        p[key] = [c * scale for c in p[key]]
    xd = torch.tensor(x * scale, device="cuda")
    td = torch.zeros(len(x), dtype=torch.int32, device="cuda")
    d = torch.empty(len(x), dtype=torch.float64, device="cuda")
    pr = torch.empty_like(d)
    B.density_noalloc(p, xd, td, d, pr)
    return d.cpu().numpy() * scale ** 3, pr.cpu().numpy(), p


@pytest.mark.parametrize("periodic", [[1, 1, 1], [0, 1, 0]])
@pytest.mark.parametrize("scale", [2.0 ** 80, 2.0 ** -80])
def test_density_in_any_unit_of_length(scale, periodic):
    need_gpu()
    d0, p0, prm = _run(1.0, periodic)
    d, p, _ = _run(scale, periodic)
    # a power of two changes no rounding; the order of the sums may differ
    assert np.max(np.abs(d / d0 - 1.0)) < 1e-13
    assert np.max(np.abs(p - p0)) < 1e-11 * (prm["p0"] + np.max(np.abs(p0)))

"""Particles at the same place: a pair of fluid particles, and a fluid particle
at a sphere's centre.  The kernel weight of such a pair is W(0) in every sum
(density, both Shepard averages, the drag's fluid sums), as in the oracle."""
import numpy as np
import pytest

import oracle
from paper_2002_03120_gb300 import binding as B
from paper_2002_03120_gb300 import cases

from _gpu_common import TOL_FORCE, need_gpu, rel_l2

pytestmark = pytest.mark.gpu

# FP64: sums of a few hundred terms; FP32: weights to a few 2^-24 and the
# coordinates' unit to 2^-25 (three times in the density), the pressure 7 times
TOL_D = {B.SDPD_PREC_FP64: 1e-12, B.SDPD_PREC_SPLIT: 1e-6}
TOL_P = {B.SDPD_PREC_FP64: 1e-11, B.SDPD_PREC_SPLIT: 1e-5}


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("precision", list(TOL_D))
@pytest.mark.parametrize("extra", [{}, {"pressure_filter": 1}, {"density_reinit": 1}, {"pressure_filter": 1, "density_reinit": 1}])
def test_coincident_particles_weigh_w0(extra, precision, mode):
    need_gpu()
    case = cases.sedimentation(nx=12, ny=12, nz=24)
    case["params"] = dict(case["params"], clamp_negative_p=0, **extra)
    t = case["type"]
    x = case["x"].copy()
    fluid, sphere = np.nonzero(t == 0)[0], np.nonzero(t == 1)[0][0]
    x[fluid[700]] = x[fluid[701]]
    x[fluid[5]] = x[sphere]
    case["x"] = x
    case["v"] = np.where((t <= 1)[:, None], np.random.default_rng(3).normal(0.0, 1e-3, x.shape), 0.0)
    sim = B.Sim(case, precision=precision)
    sim.set_force_mode(mode)
    sim.build_cells()
    sim.compute_density()
    sim.couple_drag()
    s = sim.state()
    eps, fdg = sim.drag()
    sim.close()
    orc = oracle.OracleSim(case)
    orc.evaluate(1)
    so = orc.state()
    eps_o, fdg_o = orc.fpi()[0][t == 1], orc.component("dg")[t == 1]
    assert np.isfinite(s["d"]).all() and np.isfinite(s["p"]).all() and np.isfinite(fdg).all()
    assert np.max(np.abs(s["d"] / so["d"] - 1.0)) < TOL_D[precision]
    scale = np.max(np.abs(so["p"])) + case["params"]["p0"]
    assert np.max(np.abs(s["p"] - so["p"])) < TOL_P[precision] * scale
    np.testing.assert_allclose(eps, eps_o, rtol=1e-12)
    assert rel_l2(fdg, fdg_o) < TOL_FORCE[precision]

"""Calls on a context whose particles no build has put in slots yet: the update
is refused (no forces to integrate), the diagnostics report the state with no
density."""
import numpy as np
import pytest

from paper_2002_03120_gb300 import binding as B
from paper_2002_03120_gb300 import cases

from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu
SDPD_E_STATE = 8


@pytest.mark.parametrize("precision", [B.SDPD_PREC_FP64, B.SDPD_PREC_SPLIT])
def test_update_and_diagnostics_before_the_first_build(precision):
    need_gpu()
    case = cases.poiseuille_si(nx=12, ny=12, nz=12)
    case["v"] = np.random.default_rng(1).normal(0.0, 1e-3, case["v"].shape)
    sim = B.Sim(case, precision=precision)
    d = sim.diagnostics()                        # derives the grid, builds nothing
    np.testing.assert_allclose(d[:3], (case["mass"][:, None] * case["v"]).sum(0), rtol=1e-9)
    assert d[6] == 0.0 and d[7] == 0.0
    for velver in (1, 2):
        with pytest.raises(B.SdpdError) as err:
            sim.integrate(velver)
        assert err.value.code == SDPD_E_STATE
    s = sim.state(density=False)
    assert np.array_equal(s["x"], case["x"]) and np.array_equal(s["v"], case["v"])
    sim.evaluate(1)
    sim.integrate(1)
    assert sim.diagnostics()[6] > 0.0
    sim.close()

"""The captured step.  Steps run in graphs of five and of one, with the list
build in a conditional node that a drift opens: any split of a run into calls
gives the same bits, with and without builds on the way.  The second
evaluation's ring of cached normals takes groups of four particles that
straddle instances with and without noise, rebuilt and not: the same bits as
drawing them again, and as each instance by itself."""
import numpy as np
import pytest

from paper_2002_03120_gb300 import binding as B
from paper_2002_03120_gb300 import cases

from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu
KEYS = ("x", "v", "w", "F", "N")


def _cut(case, drop, **params):
    n = len(case["x"]) - drop
    out = {k: (v[:n] if isinstance(v, np.ndarray) and len(v) > n else v) for k, v in case.items()}
    out["params"] = dict(case["params"], **params)
    return out


def _run(case, precision, calls, skin, cache=1):
    sim = B.Sim(case, precision=precision)
    sim.set_force_mode(0)
    sim.set_cell_factor(2)
    sim.set_skin(skin)
    sim.set_noise_cache(cache)
    for n in calls:
        sim.step(n)
    n_inst = len(case) if isinstance(case, list) else 1
    out = [sim.state(k, density=False) for k in range(n_inst)], sim.build_count()
    sim.close()
    return out


@pytest.mark.parametrize("precision", [B.SDPD_PREC_FP64, B.SDPD_PREC_SPLIT])
@pytest.mark.parametrize("name,skin", [("meso", 0.001), ("meso", 0.06), ("spheres", 0.06)])
def test_any_split_of_a_run(precision, name, skin):
    need_gpu()
    case = cases.poiseuille_meso() if name == "meso" else cases.sedimentation(nx=12, ny=12, nz=24)
    runs = [_run(case, precision, calls, skin) for calls in ([13], [1] * 13, [4, 6, 0, 3])]
    if skin < 0.01:
        assert runs[0][1] > 2   # the build ran inside the steps
    for r in runs[1:]:
        assert r[1] == runs[0][1]
        for k in KEYS:
            assert np.array_equal(runs[0][0][0][k], r[0][0][k]), k


@pytest.mark.parametrize("skin", [0.001, 0.01, 0.06])
def test_cached_normals_of_mixed_instances(skin):
    need_gpu()
    noisy = _cut(cases.poiseuille_meso(seed=1), 1)
    still = _cut(cases.poiseuille_meso(seed=2), 2, kBT=0.0)
    other = _cut(cases.poiseuille_meso(seed=3), 3)
    batch = [noisy, still, other]
    a = _run(batch, B.SDPD_PREC_SPLIT, [7], skin)
    b = _run(batch, B.SDPD_PREC_SPLIT, [7], skin, cache=0)
    for i in range(3):
        for k in KEYS:
            assert np.array_equal(a[0][i][k], b[0][i][k]), (i, k)
    alone = _run(noisy, B.SDPD_PREC_SPLIT, [7], skin)   # (instance 0: the same key of the generator)
    for k in KEYS:
        assert np.array_equal(a[0][0][k], alone[0][0][k]), k

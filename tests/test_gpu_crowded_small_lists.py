"""A cell too crowded for the list kernel's 16-bit entries (128 particles in a
half cell, 512 in a full one) in a context with tiny neighbour lists: the
lane-per-particle routine that scans it stages 32 records of its own, whatever
the list capacity, and the overflow is reported."""
import numpy as np
import pytest

from paper_2002_03120_gb300 import binding as B
from paper_2002_03120_gb300 import cases

from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu
SDPD_E_CAPACITY = 4


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("max_neighbors", [1, 8, 9])
@pytest.mark.parametrize("cells,k", [(2, 140), (1, 530)])
def test_capacity_error_next_to_a_crowded_cell(cells, k, max_neighbors, mode):
    need_gpu()
    base = cases.tiny_box(n=8, r_c_dx=1.6, jitter=0.1, seed=5)
    lo, wide = (2.8, 0.5) if cells == 2 else (2.3, 0.8)   # inside one cell
    blob = lo + np.random.default_rng(6).uniform(0.0, wide, (k, 3))
    case = dict(base)
    case["x"] = np.concatenate([base["x"], blob])
    for key in ("v", "w"):
        case[key] = np.zeros((len(case["x"]), 3))
    for key in ("type", "radius", "mass"):
        case[key] = np.concatenate([base[key], np.full(k, base[key][0])])
    sim = B.Sim(case, precision=B.SDPD_PREC_SPLIT, max_neighbors=max_neighbors)
    sim.set_cell_factor(cells)
    sim.set_force_mode(mode)
    with pytest.raises(B.SdpdError) as err:
        sim.build_cells()
        sim.check()
    assert err.value.code == SDPD_E_CAPACITY
    sim.close()

"""The list kernel's runs of neighbour cells and its 16-bit entries at their
limits: crowded cells on both sides of the largest cell the entries hold (128
particles in a half cell, 512 in a full one; beyond it the cells around are
scanned one lane per particle), runs cut at a bucket of the flattened index,
tiny grids whose neighbour cells are one run, and empty cells between filled
ones.  Pair sets and forces against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2002_03120_gb300 import binding as B
from paper_2002_03120_gb300 import cases

from _gpu_common import TOL_FORCE, need_gpu, pair_set, rel_l2

pytestmark = pytest.mark.gpu


def _check(case, cells, mode, max_neighbors):
    precision = B.SDPD_PREC_SPLIT
    sim = B.Sim(case, precision=precision, max_neighbors=max_neighbors)
    sim.set_cell_factor(cells)
    sim.set_force_mode(mode)
    sim.evaluate(1)
    orc = oracle.OracleSim(case)
    orc.neighbors()
    assert pair_set(sim.pairs()) == pair_set(orc.pairs())
    orc.evaluate(1)
    assert rel_l2(sim.state()["F"], orc.state()["F"]) < TOL_FORCE[precision]
    sim.close()


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("cells,k", [(2, 120), (2, 140), (2, 270), (1, 500), (1, 530)])
def test_crowded_cells(cells, k, mode):
    need_gpu()
    base = cases.tiny_box(n=8, r_c_dx=1.6, jitter=0.1, seed=5)
    # inside cell 3 of 9 half cells (width 8/9), or cell 1 of 4 full ones (width 2)
    lo, wide = (2.8, 0.5) if cells == 2 else (2.3, 0.8)
    blob = lo + np.random.default_rng(6).uniform(0.0, wide, (k, 3))
    case = dict(base)
    case["x"] = np.concatenate([base["x"], blob])
    for key in ("v", "w"):
        case[key] = np.zeros((len(case["x"]), 3))
    for key in ("type", "radius", "mass"):
        case[key] = np.concatenate([base[key], np.full(k, base[key][0])])
    _check(case, cells, mode, 1024)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("cells", [1, 2])
def test_sparse_and_tiny_grids(cells, mode):
    need_gpu()
    tiny = cases.poiseuille_si(nx=12, ny=12, nz=12, seed=3)     # 3 x 3 x 3 full cells: one run
    _check(tiny, cells, mode, 0)
    rng = np.random.default_rng(9)
    thin = cases.tiny_box(n=10, r_c_dx=1.6, jitter=0.3, seed=4)  # most cells emptied
    keep = rng.uniform(size=len(thin["x"])) < 0.15
    thin = {k: (v[keep] if isinstance(v, np.ndarray) else v) for k, v in thin.items()}
    _check(thin, cells, mode, 0)

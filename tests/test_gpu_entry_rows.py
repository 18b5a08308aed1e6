"""The per-entry layout of the pair passes (rows of eight entries of four
slots, eight lanes a particle, one to eight groups of four particles a warp)
at its edges, and the per-instance list builds."""
import numpy as np
import pytest

import oracle
from paper_2002_03120_gb300 import binding as B
from paper_2002_03120_gb300 import cases

from _gpu_common import TOL_FORCE, need_gpu, pair_set, rel_l2

pytestmark = pytest.mark.gpu
PRECISIONS = [B.SDPD_PREC_FP64, B.SDPD_PREC_SPLIT]


def _cluster(n, seed):
    """n fluid particles in a small blob of a periodic box (kernel radius 1.6):
    lists of up to n - 1 entries."""
    c = cases.tiny_box(n=6, r_c_dx=1.6, jitter=0.1, seed=seed)
    rng = np.random.default_rng(seed)
    x = 2.0 + rng.uniform(0.0, 1.2, (n, 3))
    m = c["mass"][0]
    c.update(x=x, v=rng.normal(0, 0.1, (n, 3)), w=rng.normal(0, 0.1, (n, 3)), type=np.zeros(n, np.int32),
             radius=np.full(n, 0.5), mass=np.full(n, m))
    return c


# list lengths below, at and above one, two and three rows; particle counts
# around a group of four and a warp of 32
@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("mode", [0, 1, 4])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 8, 9, 10, 17, 18, 25, 33, 35])
def test_short_lists(n, mode, precision):
    need_gpu()
    case = _cluster(n, 20 + n)
    for cells in (1, 2):
        sim = B.Sim(case, precision=precision, max_neighbors=37)   # not a multiple of a row
        sim.set_cell_factor(cells)
        sim.set_force_mode(mode)
        sim.step_count = 3
        sim.evaluate(1)
        orc = oracle.OracleSim(case)
        orc.step = 3
        orc.evaluate(1)
        if n > 1:
            assert pair_set(sim.pairs()) == pair_set(orc.pairs())
        g, o = sim.state(), orc.state()
        assert rel_l2(g["d"], o["d"]) < (1e-12 if precision == B.SDPD_PREC_FP64 else 1e-6)
        assert rel_l2(g["F"], o["F"]) < TOL_FORCE[precision]
        sim.close()


@pytest.mark.parametrize("precision", PRECISIONS)
def test_groups_do_not_change_results(precision):
    # 21,296 particles alone run one group of four a warp, in a batch of
    # several boxes four or more: the same sums bit for bit
    need_gpu()
    one = cases.poiseuille_si(nx=22, ny=44, nz=22, seed=5, coeff_t=0.0)
    single = B.Sim(one, precision=precision)
    batch = B.Sim([one] * 5, precision=precision)
    for s in (single, batch):
        s.set_force_mode(0 if precision == B.SDPD_PREC_SPLIT else 1)
        s.step(2)
    a = single.state()
    for k in (0, 4):
        b = batch.state(k)
        for q in ("x", "v", "w", "F", "N", "d"):
            assert np.array_equal(a[q], b[q]), (k, q)
    single.close()
    batch.close()


@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("mode", [0, 1])
def test_lists_rebuilt_per_instance(precision, mode):
    # a fast instance beside a slow one: the fast one's rebuilds leave the slow
    # one's lists alone, so each repeats its own run bit for bit
    need_gpu()
    slow = cases.poiseuille_si(nx=12, ny=12, nz=12, seed=2, coeff_t=0.0)
    fast = cases.sedimentation(nx=12, ny=12, nz=24, coeff_t=0.0)
    rng = np.random.default_rng(3)
    fast["v"] = np.where((fast["type"] <= 1)[:, None], rng.normal(0, 2.0, fast["v"].shape), 0.0)

    def sim(c):
        s = B.Sim(c, precision=precision)
        s.set_force_mode(mode)
        s.step(8)
        return s

    both, alone = sim([slow, fast]), [sim(slow), sim(fast)]
    assert alone[0].build_count() == 1 and alone[1].build_count() > 1
    for k in (0, 1):
        a, b = alone[k].state(density=False), both.state(k, density=False)
        for q in ("x", "v", "w", "F", "N"):
            assert np.array_equal(a[q], b[q]), (k, q)

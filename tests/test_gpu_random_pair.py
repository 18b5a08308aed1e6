"""The random force of a fluid pair in split precision is the same seen from
either particle (Eq. FijT; sigma holds 1/sqrt(d_i d_j)): in the direct pass,
which evaluates the pair from both sides, the two forces are opposite bit for
bit also where the densities differ, drawn and with the normals from the cache.
A sphere near one of the two changes its density and, at rest, adds no force."""
import numpy as np
import pytest

from paper_2002_03120_gb300 import binding as B
from paper_2002_03120_gb300 import cases

from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("dx", [1e-3, 1.0, 1e-7])
def test_random_forces_of_a_pair_are_opposite(dx, mode):
    need_gpu()
    p = cases.base_params(dx=dx)
    h, n = p["r_c"], 6
    p.update(coeff_c=0.0, coeff_d=0.0, coeff_r=0.0, body_amp=0.0, g=[0.0, 0.0, 0.0], origin=[0.0, 0.0, 0.0],
             box=[3.0 * n * h] * 3, periodic=[1, 1, 1])
    rng = np.random.default_rng(4)
    c = (np.stack(np.meshgrid(*[np.arange(n)] * 3), -1).reshape(-1, 3) + 0.5) * 3.0 * h
    u, w = rng.normal(size=c.shape), rng.normal(size=c.shape)
    u /= np.linalg.norm(u, axis=1)[:, None]
    w -= (w * u).sum(1)[:, None] * u
    w /= np.linalg.norm(w, axis=1)[:, None]
    a = rng.uniform(0.3, 0.9, len(c))[:, None] * h
    b = rng.uniform(0.3, 0.9, len(c))[:, None] * h
    xi, xj = c + a * u, c                          # the pair
    xk = xj - b * (0.9 * u + 0.43 * w)             # the sphere: beyond h of i for most
    x = np.concatenate([xi, xj, xk])
    t = np.repeat([0, 0, 1], len(c)).astype(np.int32)
    R = np.where(t == 1, 0.3 * dx, 0.5 * dx)
    m = np.full(len(x), p["rho0"] * dx ** 3)
    z = np.zeros_like(x)
    sim = B.Sim(dict(params=p, x=x, v=z, w=z, type=t, radius=R, mass=m), precision=B.SDPD_PREC_SPLIT)
    sim.set_force_mode(mode)
    sim.evaluate(1)
    drawn = sim.state()
    sim.compute_forces(2)
    cached = sim.state()
    sim.close()
    d = drawn["d"]
    k = len(c)
    assert np.mean(np.abs(d[:k] / d[k:2 * k] - 1.0) > 0.05) > 0.5
    for s in (drawn, cached):
        assert np.isfinite(s["F"]).all() and np.all(np.linalg.norm(s["F"][:k], axis=1) > 0.0)
        assert np.array_equal(s["F"][:k], -s["F"][k:2 * k])

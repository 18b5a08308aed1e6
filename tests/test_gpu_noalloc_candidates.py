"""sdpd_density_noalloc's fixed-point candidate test and neighbour compaction
against a brute-force sum in numpy: boxes of one and of several windows, odd
cell counts, positions folded from far away, particles outside the grid on
wall axes, coincident particles, fewer particles than a warp."""
import numpy as np
import pytest

from paper_2002_03120_gb300 import binding as B
from paper_2002_03120_gb300 import cases

from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def _brute(p, x, t):
    h, dx, L = p["r_c"], p["dx"], np.asarray(p["box"])
    lucy = lambda r: 105.0 / (16.0 * np.pi * h ** 3) * (1 + 3 * r / h) * (1 - r / h) ** 3  # noqa: E731
    m = int(np.ceil(h / dx)) + 1
    a = np.arange(-m, m + 1) * dx
    r = np.sqrt(a[:, None, None] ** 2 + a[None, :, None] ** 2 + a[None, None, :] ** 2)
    cn = 1.0 / (dx ** 3 * lucy(r[r < h]).sum())
    d = np.empty(len(x))
    for i in range(len(x)):
        v = x[i] - x
        for k in range(3):
            if p["periodic"][k]:
                v[:, k] -= L[k] * np.rint(v[:, k] / L[k])
        r = np.sqrt((v * v).sum(1))
        d[i] = cn * lucy(r[r < h]).sum()
    d[t == 3] = 1.0 / dx ** 3
    return d


SHAPES = {
    "one_window": ((12, 12, 15), (1, 1, 1)),       # 3.08 r_c: below 4 r_c
    "windows": ((33, 17, 12), (1, 1, 1)),          # 8.46 and 4.36 r_c
    "walls": ((9, 14, 12), (0, 1, 0)),
    "warp_remainder": ((12, 12, 12), (1, 1, 1)),
}


@pytest.mark.parametrize("shape", list(SHAPES))
def test_noalloc_density_equals_brute_force(shape):
    need_gpu()
    import torch
    (nx, ny, nz), per = SHAPES[shape]
    p = cases.base_params(dx=1e-3)
    p.update(box=[nx * 1e-3, ny * 1e-3, nz * 1e-3], periodic=list(per), origin=[0.5e-3, -2e-3, 0.0])
    rng = np.random.default_rng(11)
    lo, L = np.asarray(p["origin"]), np.asarray(p["box"])
    x = lo + L * rng.uniform(size=(nx * ny * nz, 3))
    if shape == "warp_remainder":
        x = x[:29]
    x[5] = x[4]                                     # coincident
    t = np.zeros(len(x), np.int32)
    t[::7] = 3
    raw = x.copy()
    for k in range(3):
        if per[k]:
            raw[::5, k] += 3.0 * L[k]               # folded by the call
            raw[1::5, k] -= 2.0 * L[k]
        else:
            x[:6, k] += 40.0 * L[k]                 # a clump far outside the grid
            raw[:6, k] = x[:6, k]
    xd = torch.tensor(raw, device="cuda")
    td = torch.tensor(t, device="cuda")
    d = torch.empty(len(x), dtype=torch.float64, device="cuda")
    pr = torch.empty_like(d)
    B.density_noalloc(p, xd, td, d, pr)
    # FP64 sums of up to a few hundred positive terms of coordinates folded
    # from three boxes away: 4e2 x 2^-53 x (coordinate / r_c < 60) x slack
    ref = _brute(p, x, t)
    assert np.max(np.abs(d.cpu().numpy() - ref) / ref) < 1e-11

"""The FP64 normals' radius sqrt(-2 ln U) where U is next to 1 and the
logarithm next to 0: relative to its own size, not to 1.

The table's logarithm is off by at most 0.4 r^5 (r < 2^-12) plus 2.5 x 2^-64 of
roundings there, 5e-19: 4.2e-12 of -2 ln U at U = 1 - 2^-24, half of that of
the radius."""
import numpy as np
import pytest

from paper_2002_03120_gb300 import binding as B

from _gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def _philox(c, k0, k1):
    """Philox4x32-10 of arrays of counters (uint64 words below 2^32)."""
    M = np.uint64(0xFFFFFFFF)
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & M, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & M]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def test_radius_of_uniforms_next_to_one():
    need_gpu()
    seed, step = 0x1234_5678_9ABC_DEF0, 7
    rng = np.random.default_rng(1)
    n = 3_000_000
    gi, gj = (rng.integers(0, 1 << 22, n).astype(np.uint32) for _ in range(2))
    gj[gj == gi] += 1
    lo, hi = np.minimum(gi, gj).astype(np.uint64), np.maximum(gi, gj).astype(np.uint64)
    s = np.full_like(lo, step)
    a = _philox([lo, hi, s, np.zeros_like(lo)], seed & 0xFFFFFFFF, seed >> 32)
    b = _philox([lo, hi, s, np.ones_like(lo)], seed & 0xFFFFFFFF, seed >> 32)
    m = np.stack([a[0], a[2], b[0]], 1) >> np.uint64(9)          # U = (m + 1/2) 2^-23
    near = m >= (1 << 23) - 128
    rows = np.nonzero(near.any(1))[0]
    assert near.sum() > 60
    z = B.noise_normals(B.SDPD_PREC_FP64, seed, 0, step, gi[rows], gj[rows])
    got = np.hypot(z[:, 0::2], z[:, 1::2])[near[rows]]
    d = (((1 << 23) - m[rows][near[rows]]).astype(np.float64) - 0.5) / 8388608.0   # 1 - U, exact
    exact = np.sqrt(-2.0 * np.log1p(-d))                          # to a few 1e-16 of its value
    assert np.max(np.abs(got / exact - 1.0)) < 3e-12

"""Gradients at the edges of the gradient kernel's row tiles (16 rows up to a
batch of 512, 32 beyond): one row, a full and an overfull tile, both sides of
the change of the tile, the largest batch.  Oracle and tolerance (BF16 operands
against the same rounding points, FP32 sums) as in test_gpu_mlp.py."""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from paper_2002_03120_gb300 import binding as B

from _gpu_common import need_gpu, rel_l2
from test_gpu_mlp import ORDER, _dev, _params, flat, unflat

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 15, 16, 17, 33, 511, 512, 513, 545, 4096])
def test_gradients_at_tile_edges(batch):
    need_gpu()
    p = _params(6)
    net = B.Mlp(seed=0, batch_max=batch)
    net.set_params(flat(p))
    rng = np.random.default_rng(batch)
    X = rng.uniform(size=(batch, 3)).astype(np.float32)
    T = (1.0 + rng.normal(size=batch)).astype(np.float32)
    loss = net.gradients(_dev(X), _dev(T))
    g = unflat(net.grads().astype(np.float64), p)
    y, cache = M.forward(p, X.astype(np.float64), "bf16")
    ref = M.backward(p, cache, y, T.astype(np.float64))
    # the loss and the gradients carry the forward pass's 1e-3 (twice for a square)
    assert loss == pytest.approx(M.loss(y, T), rel=4e-3)
    for k in ORDER:
        assert rel_l2(g[k], ref[k]) < 5e-3, (k, rel_l2(g[k], ref[k]))
    net.close()

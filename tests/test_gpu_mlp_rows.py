"""Inference on both sides of the changes of the row tile (16, 32 and 64 rows
with one CTA per SM, then 128-row tiles round the CTAs).  Every form performs
the same operations on a row in the same order, so a row's output is the same
bits in a call of any size; nothing is written past the last row."""
import numpy as np
import pytest
import torch

from paper_2002_03120_gb300 import binding as B

from _gpu_common import need_gpu
from test_gpu_mlp import _dev, _params, flat

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_sm,more", [(0, 1), (0, 17), (16, 0), (16, 1), (32, 0), (32, 1), (64, 0), (64, 1), (128, 1),
                                         (512, 129)])
def test_inference_at_tile_changes(per_sm, more):
    need_gpu()
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + more
    p = _params(8)
    net = B.Mlp(seed=0)
    net.set_params(flat(p))
    X = _dev(np.random.default_rng(n).uniform(size=(n, 3)).astype(np.float32))
    Y = torch.full((n + 64,), 7.0, device="cuda")
    net.infer(X, Y[:n])
    net.check()
    assert bool(torch.all(Y[n:] == 7.0))
    # the same rows behind others, in a call that takes the largest tiles
    lead = 100003
    Z = torch.empty(lead + n, device="cuda")
    net.infer(torch.cat([torch.rand((lead, 3), device="cuda"), X]), Z)
    net.check()
    assert bool(torch.all(Y[:n] == Z[lead:]))
    net.close()

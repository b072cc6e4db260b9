"""The MLP's hidden layer on the smallest batches (GPU), against the oracle: every number of prompts
on both sides of the rule that picks its kernel (8), widths that are no multiple of the block's 4
units, hidden sizes around a warp's 128 columns and off the 16-byte loads.

Tolerance: as in test_gpu_mlp_head.py, 1e-4 relative to the largest reference magnitude of each output."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_mlp_head import _case, _close, _dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,F", [(1, 1), (3, 5), (127, 6), (128, 64), (130, 67), (1000, 33), (4096, 9)])
@pytest.mark.parametrize("B", [1, 2, 3, 4, 5, 7, 8, 9])
def test_hidden_layer_of_a_small_batch(cuda_lib, B, D, F):
    h, W1, b1, W2, b2, c, y = _case(B, D, F, 7, seed=B + D, bias=D != 130)
    ctx = cuda_lib.Context(0)
    head = _dev(cuda_lib, W1, b1, W2, b2, c)
    hd, yd = torch.from_numpy(h).cuda(), torch.from_numpy(y).cuda()
    pred, probs = ctx.mlp_head_predict(hd, head, probs=True)
    out = ctx.mlp_head_loss(hd, head, yd, 0.5)
    again = ctx.mlp_head_loss(hd, head, yd, 0.5)
    ctx.sync_status()
    assert all(torch.equal(a, b) for a, b in zip(out, again))
    ref_y, ref_p = oracle.mlp_length_head(h.astype(np.float64), W1, b1, W2, b2, c, return_probs=True)
    _close(probs.cpu().numpy(), ref_p, "p_hat")
    _close(pred.cpu().numpy(), ref_y, "y_hat")
    ref = oracle.mlp_head_loss(h.astype(np.float64), W1, b1, W2, b2, c, y, 0.5)
    names = ("loss", "dL/dW1", "dL/db1", "dL/dW2", "dL/db2", "dL/dpooled")
    for name, g, r in zip(names, out, ([ref[0]], *ref[1:])):
        if r is not None and g is not None:
            _close(g.cpu().numpy(), r, name)

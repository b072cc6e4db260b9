"""The MLP predictor at sizes whose tiles along one side pass 65535, the limit of a grid's y and z
(GPU): a hidden layer of 8.4 million units, a batch of 8.4 million prompts.  Inputs are small
multiples of 1/8, so that the hidden units are exact and none changes sides by rounding.

Tolerance: as in test_gpu_mlp_head.py, 1e-4 relative to the largest reference magnitude (sums in
chains of 64 and over partial sums: a relative error of 1e-5 at these lengths)."""
import numpy as np
import torch
import pytest

import oracle
from test_gpu_mlp_head import _close, _dev

pytestmark = pytest.mark.gpu


def _eighths(rng, *shape):
    return (rng.integers(-16, 17, shape) / 8).astype(np.float32)


def test_wide_hidden_layer(cuda_lib):
    rng = np.random.default_rng(1)
    B, D, F, K = 9, 2, 65536 * 128 + 1, 3
    h, W1, b1 = _eighths(rng, B, D), _eighths(rng, F, D), _eighths(rng, F)
    W2 = (_eighths(rng, K, F) / np.sqrt(F)).astype(np.float32)
    c, y = np.asarray([10, 20, 40], np.float32), rng.uniform(0, 50, B).astype(np.float32)
    ctx = cuda_lib.Context(0)
    head = _dev(cuda_lib, W1, b1, W2, None, c)
    out = ctx.mlp_head_loss(torch.from_numpy(h).cuda(), head, torch.from_numpy(y).cuda(), 0.5)
    ctx.sync_status()
    ref = oracle.mlp_head_loss(h.astype(np.float64), W1, b1, W2, None, c, y, 0.5)
    names = ("loss", "dL/dW1", "dL/db1", "dL/dW2", "dL/db2", "dL/dpooled")
    for name, g, r in zip(names, out, ([ref[0]], *ref[1:])):
        if g is not None:
            _close(g.cpu().numpy(), r, name)


def test_many_prompts(cuda_lib):
    rng = np.random.default_rng(2)
    B, D, F, K = 65536 * 128 + 1, 2, 3, 2
    W1, b1, W2 = _eighths(rng, F, D), _eighths(rng, F), _eighths(rng, K, F)
    c = np.asarray([100, 300], np.float32)
    h = torch.randint(-16, 17, (B, D), device="cuda").float() / 8
    ctx = cuda_lib.Context(0)
    pred, probs = ctx.mlp_head_predict(h, _dev(cuda_lib, W1, b1, W2, None, c), probs=True)
    ctx.sync_status()
    t = lambda a: torch.from_numpy(a).cuda().double()
    p = torch.softmax((h.double() @ t(W1).T + t(b1)).clamp(min=0) @ t(W2).T, dim=1)
    assert float((probs.double() - p).abs().max()) <= 1e-4
    assert float((pred.double() - p @ t(c)).abs().max()) <= 1e-4 * 300

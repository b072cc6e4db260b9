"""The head's fp32 tiles at their edges, against the oracle (GPU): batches around every tile
height of the wide products (16, 32, 64, 128 prompts), hidden sizes around the 64-value
slices, the cluster splits and the 16-byte loads, bins around the 32-wide tiles.

Tolerance: as in test_gpu_head_loss.py, 1e-4 relative to the largest reference magnitude of
each output (fp32 sums of length up to D, F or B, relative error below 1e-5)."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_head_loss import _case as linear_case, _close, _run as linear_run
from test_gpu_mlp_head import _case as mlp_case, _dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,D,K", [(31, 63, 31), (32, 64, 32), (33, 65, 33), (130, 1030, 70),
                                   (257, 129, 1024), (1, 1, 1)])
def test_linear_head_tiles(cuda_lib, B, D, K):
    pooled, W, b, c, y = linear_case(B, D, K, seed=B, spread=5.0)
    got = linear_run(cuda_lib, pooled, W, b, c, y, 0.5)
    ref = oracle.head_loss(pooled.astype(np.float64), W, b, c, y, 0.5)
    for name, g, r in zip(("loss", "dL/dW", "dL/dbias", "dL/dpooled"), got, ([ref[0]], *ref[1:])):
        _close(g, r, name)


@pytest.mark.parametrize("B,D,F,K", [(16, 1023, 63, 32), (17, 1024, 64, 33), (32, 1026, 65, 5),
                                     (33, 260, 129, 31), (64, 500, 127, 7), (65, 2047, 130, 40),
                                     (128, 64, 257, 3), (129, 129, 128, 32), (1, 4097, 1, 2)])
def test_mlp_head_tiles(cuda_lib, B, D, F, K):
    h, W1, b1, W2, b2, c, y = mlp_case(B, D, F, K, seed=B)
    head = _dev(cuda_lib, W1, b1, W2, b2, c)
    ctx = cuda_lib.Context(0)
    out = ctx.mlp_head_loss(torch.from_numpy(h).cuda(), head, torch.from_numpy(y).cuda(), 0.5)
    ctx.sync_status()
    ref = oracle.mlp_head_loss(h.astype(np.float64), W1, b1, W2, b2, c, y, 0.5)
    names = ("loss", "dL/dW1", "dL/db1", "dL/dW2", "dL/db2", "dL/dpooled")
    for name, g, r in zip(names, out, ([ref[0]], *ref[1:])):
        _close(g.cpu().numpy(), r, name)

"""Entropy from hidden states where the vocabulary splits and the row tile are ragged (GPU), against
the fp64 oracle within 1e-3 nats: batches below one row tile (1, 7, 8, 9, 127, 128 rows: the
copied box follows them) and above (129, 300), vocabularies around one unit of 32, one tile of
256, and sizes whose splits end inside a tile."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_entropy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,V", [(1, 1), (7, 31), (8, 32), (9, 33), (127, 255), (128, 257), (129, 4864),
                                    (1, 4865), (300, 5000), (37, 39000)])
def test_lm_head_splits(cuda_lib, rows, V):
    g = torch.Generator().manual_seed(rows + V)
    D = 192
    h = torch.randn(rows, D, generator=g).bfloat16()
    W = (torch.randn(V, D, generator=g) * (3.0 / D ** 0.5)).bfloat16()
    bits = lambda t: t.contiguous().view(torch.int16).numpy().view(np.uint16)
    ctx = cuda_lib.Context(0)
    hd, Wd = h.cuda(), W.cuda()
    out = ctx.lm_head_entropy(hd, Wd)
    again = ctx.lm_head_entropy(hd, Wd)
    ctx.sync_status()
    assert torch.equal(out, again)
    assert_entropy(out.cpu().numpy(), oracle.lm_head_entropy(bits(h), bits(W)))

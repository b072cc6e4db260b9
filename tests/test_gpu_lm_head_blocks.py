"""Entropy from hidden states over many row blocks (GPU), against the fp64 oracle: several items an
SM, splits of whole vocabulary tiles whose last one is not full (a vocabulary that is no multiple of
256, of 32), splits cut in units over several row blocks, one split for all (more row blocks than
SMs), a last row block of one row.

Tolerance: a logit is an fp32 sum of D <= 256 products of size 1 (error below D 2^-24 = 2e-5) and
moves H by at most its own error times a factor of order 1; the fp32 entropy sums add below 1e-5."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,D,V", [(4500, 128, 5003), (1000, 256, 6000), (385, 256, 1999), (129, 64, 39001),
                                      (20001, 64, 2600), (2048, 192, 8192)])
def test_lm_head_blocks(cuda_lib, rows, D, V):
    g = torch.Generator().manual_seed(rows + V)
    h = torch.randn(rows, D, generator=g).bfloat16()
    W = (torch.randn(V, D, generator=g) * (3.0 / D ** 0.5)).bfloat16()
    bits = lambda t: t.contiguous().view(torch.int16).numpy().view(np.uint16)
    ctx = cuda_lib.Context(0)
    hd, Wd = h.cuda(), W.cuda()
    out = ctx.lm_head_entropy(hd, Wd)
    again = ctx.lm_head_entropy(hd, Wd)
    ctx.sync_status()
    assert torch.equal(out, again)
    ref = oracle.lm_head_entropy(bits(h), bits(W))
    assert np.max(np.abs(out.cpu().numpy() - ref)) <= 1e-4

"""Misalignment counts at the edge of what a block keeps in registers (2048 tokens) and with the
two selections of a value inside one bin, exactly equal to the oracle (GPU)."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_misalignment_ties import _values

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kinds", [("range", "ulp5000"), ("two", "range"), ("ulp1024", "constant")])
def test_prompts_around_the_cached_length(cuda_lib, kinds):
    rng = np.random.default_rng(9)
    lens = [1, 511, 1536, 2047, 2048, 2049, 2560, 4097]
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    H = np.concatenate([_values(kinds[0], n, rng) for n in lens])
    S = np.concatenate([_values(kinds[1], n, rng) for n in lens])
    ctx = cuda_lib.Context(0)
    dev = [torch.from_numpy(x).cuda() for x in (H, S, cu)]
    for pct in (1, 40, 49, 50):
        got = ctx.misalignment(*dev, pct)
        ctx.sync_status()
        ref = oracle.misalignment(H, S, cu, pct)
        assert np.array_equal(got.cpu().numpy().astype(np.int64), ref), pct

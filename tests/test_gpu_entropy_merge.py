"""Rows of the entropy kernel cut into pieces: the merge with one thread, a few lanes, a warp
and a block a row, against the oracle (GPU)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import assert_entropy
from synth import device as sd
from synth import workloads as W

pytestmark = pytest.mark.gpu


# pieces a row on 152 SMs (3648 pieces in all): 3648, 64.0, 64 + a bit, 32.3, 15, 2, 1
@pytest.mark.parametrize("rows,V", [(1, 152064), (57, 32000), (56, 32003), (113, 16001),
                                    (243, 9001), (1824, 4003), (4001, 1030)])
def test_cut_rows(cuda_lib, rows, V):
    w = W.Workload("ent", seed=31, B=1, T_lo=1, T_hi=1, dtype=synth.BF16, V=V, n_layers_model=1,
                   layers_used=1, Hq=1, Hkv=1, d=64, D=8, spike_prob=0.2)
    ld = (V + 7) // 8 * 8
    ctx = cuda_lib.Context(0)
    x = sd.logits(w, 0, rows, ld=ld, pad_val=1e4)
    H = ctx.token_entropy(x, V=V)
    assert torch.equal(H, ctx.token_entropy(x, V=V))
    ctx.sync_status()
    assert_entropy(H.cpu().numpy(), oracle.token_entropy(W.host_logits(w, np.arange(rows), ld=ld), V=V))

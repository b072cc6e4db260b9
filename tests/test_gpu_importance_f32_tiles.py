"""fp32 row normalisers and column sums at the edges of their tiles, in each split of the work
(64 or 128 fixed rows, chunks of 1 to 8 query tiles, items per head or per KV group, prompts in
batch order or in order of length), against the oracle (GPU)."""
import math

import numpy as np
import pytest
import torch

import oracle
import synth
from test_gpu_importance import _qk, _run, _wl

pytestmark = pytest.mark.gpu

CASES = {
    # 64 rows, one query tile per item, a head per item
    "one": ([1], 1, 1, 64),
    "edges64": ([63, 64, 65, 0, 127], 2, 1, 128),
    "edges128": ([128, 129, 191, 192, 193], 4, 2, 64),
    # more items than blocks: prompts in order of length
    "sorted": ([0, 700, 1, 0, 640, 300, 640, 900], 8, 8, 64),
    # column sums with 128 rows and one query tile per item
    "edges256": ([255, 256, 257, 320, 385, 448, 511, 640], 8, 2, 64),
    # 128 rows for both, items per KV group, chunks of 8 query tiles
    "many": ([1 + (37 * i) % 200 for i in range(160)], 16, 8, 64),
    "long": ([1153, 1025, 1100, 1217] * 2, 16, 16, 64),
}


@pytest.mark.parametrize("exclude_self", [False, True])
@pytest.mark.parametrize("name", list(CASES))
def test_f32_tiles(cuda_lib, name, exclude_self):
    lens, Hq, Hkv, d = CASES[name]
    w, cu = _wl(synth.F32, lens, Hq, Hkv, d)
    S, ref = _run(cuda_lib, w, cu, [0], exclude_self=exclude_self)
    # fp32 scores (sums of d terms of size 1: below 1e-5) move a probability by as much, and
    # a column's fp32 sum of positive terms adds less than that
    np.testing.assert_allclose(S, ref, rtol=3e-5, atol=1e-12)


@pytest.mark.parametrize("name", list(CASES))
def test_f32_row_normalisers(cuda_lib, name):
    lens, Hq, Hkv, d = CASES[name]
    w, cu = _wl(synth.F32, lens, Hq, Hkv, d)
    Qh, Kh, Qd, Kd = _qk(w, cu, 0)
    ctx = cuda_lib.Context(0)
    lse = ctx.attn_lse(Qd, Kd, torch.as_tensor(cu, device="cuda"), max(lens))
    ctx.sync_status()
    ref = oracle.attn_lse(Qh, Kh, cu, 1 / math.sqrt(d))
    np.testing.assert_allclose(lse.cpu().numpy(), ref, rtol=0, atol=1e-5)

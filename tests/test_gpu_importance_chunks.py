"""Column sums of bf16 inputs in items of one and of two pairs of query tiles, on either side of
the rule that picks between them (items of one pair fit the SMs), against the oracle (GPU).

Tolerance: the scores are fp32 sums of d products of bf16 values (below 1e-5), which moves a
probability by as much; a column's fp32 sum of positive terms and its normalisers add less."""
import numpy as np
import pytest

import synth
from test_gpu_importance import _run, _wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exclude_self", [False, True])
@pytest.mark.parametrize("lens,Hq,Hkv,d", [
    ([1500], 7, 1, 128),          # one pair an item: 6 pairs of key tiles, 12 items of two pairs
    ([257, 512, 513, 1], 4, 2, 64),
    ([600, 513, 770] * 7, 8, 8, 64),  # two pairs an item
    ([300] * 40, 4, 4, 128),
    ([1000], 16, 16, 64),         # two pairs: 96 items of them, 160 of one
    ([900, 1100], 8, 8, 128),     # one pair would make 160 items
])
def test_pairs_per_item(cuda_lib, lens, Hq, Hkv, d, exclude_self):
    w, cu = _wl(synth.BF16, lens, Hq, Hkv, d)
    S, ref = _run(cuda_lib, w, cu, [0], exclude_self=exclude_self)
    np.testing.assert_allclose(S, ref, rtol=3e-5, atol=1e-12)

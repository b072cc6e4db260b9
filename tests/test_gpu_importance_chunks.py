"""Column sums of bf16 inputs in items of one and of two pairs of query tiles, on either side of
the rule that picks between them (fewer items than SMs), against the oracle (GPU)."""
import pytest

import synth
from gpu_util import assert_importance
from test_gpu_importance import _run, _wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exclude_self", [False, True])
@pytest.mark.parametrize("lens,Hq,Hkv,d", [
    ([1500], 7, 1, 128),          # one pair an item: 6 pairs of key tiles, 12 items of two pairs
    ([257, 512, 513, 1], 4, 2, 64),
    ([600, 513, 770] * 7, 8, 8, 64),  # two pairs an item
    ([300] * 40, 4, 4, 128),
])
def test_pairs_per_item(cuda_lib, lens, Hq, Hkv, d, exclude_self):
    w, cu = _wl(synth.BF16, lens, Hq, Hkv, d)
    S, ref = _run(cuda_lib, w, cu, [0], exclude_self=exclude_self)
    assert_importance(S, ref)

"""Importance with a bound on the prompt lengths far above them (GPU): the same bits as with the
tight bound wherever the work is cut the same way, the oracle's values where it is not, and no more
workspace than the batch itself can need."""
import numpy as np
import pytest
import torch

import oracle
import synth
from test_gpu_importance import _qk, _wl

pytestmark = pytest.mark.gpu


def _importance(ctx, Qd, Kd, cu, bound):
    ctx.attn_importance(Qd, Kd, torch.as_tensor(cu, device="cuda"), bound)
    S = ctx.attn_importance_finalize(1, int(cu[-1]))
    ctx.sync_status()
    return S


@pytest.mark.parametrize("dtype", [synth.F32, synth.BF16])
@pytest.mark.parametrize("lens,Hq,Hkv", [([300, 17, 129], 8, 2), ([1], 1, 1), ([700], 4, 4)])
def test_same_bits(cuda_lib, dtype, lens, Hq, Hkv):
    w, cu = _wl(dtype, lens, Hq, Hkv, 64)
    _, _, Qd, Kd = _qk(w, cu, 0)
    ctx = cuda_lib.Context(0)
    tight = _importance(ctx, Qd, Kd, cu, max(lens))
    for bound in ((max(lens) + sum(lens)) // 2, sum(lens)):
        assert torch.equal(_importance(ctx, Qd, Kd, cu, bound), tight), bound


def test_workspace_of_many_short_prompts(cuda_lib):
    """1000 prompts of 128 tokens in fp32, one head, fewer items than the SMs want: with slots for
    every 64 queries of the bound the partial sums would take 1 GB."""
    w, cu = _wl(synth.F32, [128] * 1000, 1, 1, 64)
    Qh, Kh, Qd, Kd = _qk(w, cu, 0)
    ctx = cuda_lib.Context(0)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    S = _importance(ctx, Qd, Kd, cu, 128000)
    assert free - torch.cuda.mem_get_info()[0] < 256 << 20
    C = np.zeros(int(cu[-1]))
    oracle.attn_colsum(Qh, Kh, cu, 1 / 8, out=C)
    ref = oracle.importance(C, cu, 1, 1)
    np.testing.assert_allclose(S.cpu().numpy(), ref, rtol=3e-5, atol=1e-12)  # as the fp32 tile tests

"""Rows of the entropy kernel cut into pieces: the merge with one thread, a few lanes, a warp
and a block a row, against the oracle (GPU).

Tolerance: 1e-5 of H (of 1 nat for rows below that).  The sums are fp32, of terms of one sign, in
chains of at most a few hundred additions: below 1e-5 at the worst, ~1e-6 as roundings fall.  A
piece lost or counted twice moves H by more: one of the 3648 pieces of a near-flat row of 152064
entries by ln(1 + 1/3648) = 2.7e-4 nats, 2.3e-5 of H, and one that holds one of three equal large
logits by 0.05 nats or more."""
import numpy as np
import pytest
import torch

import oracle
import synth
from synth import device as sd
from synth import workloads as W

pytestmark = pytest.mark.gpu


def _close(H, ref):
    err = np.abs(H.cpu().numpy() - ref) / np.maximum(ref, 1.0)
    assert err.max() <= 1e-5, f"entropy error {err.max():.2e} of max(H, 1)"


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
    _close(H, oracle.token_entropy(W.host_logits(w, np.arange(rows), ld=ld), V=V))


@pytest.mark.parametrize("rows,V", [(1, 152064), (2, 152064), (57, 32000), (56, 32003), (113, 16001), (243, 9001)])
def test_every_piece_counts(cuda_lib, rows, V):
    """Near-flat rows, and rows whose mass lies on three logits in the first, a middle and the last
    columns."""
    g = torch.Generator(device="cuda").manual_seed(rows)
    ld = (V + 7) // 8 * 8
    x = (torch.randn(rows, ld, generator=g, device="cuda") * 0.1).bfloat16()
    if rows > 1:
        for r in range(1, rows, 2):
            x[r, [r % 8, V // 2 - r, V - 1 - r % 8]] = 30.0
    ctx = cuda_lib.Context(0)
    H = ctx.token_entropy(x, V=V)
    ctx.sync_status()
    z = x[:, :V].double()
    logp = torch.log_softmax(z, dim=1)
    _close(H, -(logp.exp() * logp).sum(dim=1).cpu().numpy())

"""Misalignment counts where the threshold selection can go wrong (GPU), exactly equal to the
oracle: constant prompts, two values, keys that span the whole exponent range and both signs,
neighbouring floats (spans under, at and over one pass of 1024 bins), ties cut by index across
the scan's boundaries."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def _values(kind, n, rng):
    if kind == "constant":
        return np.full(n, 3.25, np.float32)
    if kind == "two":
        return rng.choice(np.asarray([-1.0, 2.0], np.float32), n)
    if kind == "range":
        return (rng.choice([-1.0, 1.0], n) * 10.0 ** rng.uniform(-37, 38, n)).astype(np.float32)
    span = {"ulp1023": 1023, "ulp1024": 1024, "ulp5000": 5000}[kind]
    bits = np.float32(1.5).view(np.uint32) + rng.integers(0, span + 1, n).astype(np.uint32)
    bits[:2] = np.float32(1.5).view(np.uint32) + np.asarray([0, span], np.uint32)[: min(2, n)]
    return bits.view(np.float32)


@pytest.mark.parametrize("kind", ["constant", "two", "range", "ulp1023", "ulp1024", "ulp5000"])
def test_misalignment_threshold_ties(cuda_lib, kind):
    rng = np.random.default_rng(5)
    lens = [2, 31, 512, 513, 1025, 9000]
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    H = np.concatenate([_values(kind, n, rng) for n in lens])
    S = np.concatenate([_values(kind, n, rng) for n in lens])
    ctx = cuda_lib.Context(0)
    dev = [torch.from_numpy(x).cuda() for x in (H, S, cu)]
    for pct in (3, 40, 50):
        got = ctx.misalignment(*dev, pct)
        ctx.sync_status()
        ref = oracle.misalignment(H, S, cu, pct)
        assert np.array_equal(got.cpu().numpy().astype(np.int64), ref), pct

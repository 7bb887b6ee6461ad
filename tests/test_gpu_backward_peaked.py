"""The tiled gradients of the fp32 read on the GPU (needs a GB300) where heads of one call take
different ways: plain heads, heads with priors so peaked that pairs' weights vanish, at small
and at large beta, and heads most of whose channels are too wide for the factors.

fp32 throughout: 1e-4 of each gradient's largest entry against the float64 oracle.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_07160_gb300 import build, fem
from paper_2602_07160_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    return fem.load()


@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("T,d", [(64, 16), (130, 64), (100, 128), (300, 40), (700, 24)])
def test_heads_of_one_call(T, d, causal):
    q, k, v, beta = W.make_custom(1, 4, T, d, dtype="f32", seed=T)
    peaked = torch.tensor([1.0, 5.0, 5.0, 1.0]).reshape(1, 4, 1, 1)
    q, k = q * peaked, k * peaked
    beta[1] = beta[1].clamp(max=4.0)
    beta[3] = 20.0 + 10.0 * beta[3]
    dout = torch.randn(q.shape, generator=torch.Generator().manual_seed(T)) * 1e-3
    x = [a.cuda() for a in (q, k, v, beta)]
    out, lse = fem.fem_fwd_f32(*x, causal=causal)
    got = fem.fem_bwd_f32(*x, out, lse, dout.cuda(), causal=causal)
    fem.check_device_error()
    ref = oracle.fem_backward(q, k, v, beta, dout, causal)
    for g, r in zip(got, ref):
        for h in range(4):  # head by head: dq, dk, dv [B, H, T, d], dbeta [H, d]
            a, b = (g[:, h], r[:, h]) if g.dim() == 4 else (g[h], r[h])
            assert np.abs(a.cpu().double().numpy() - b).max() <= 1e-4 * np.abs(b).max()


def test_same_bits_from_call_to_call():
    """dq and dk in any head, dv in channels that no head counts as wide (the wide ones' dv and dbeta
    are summed with atomics)."""
    q, k, v, beta = W.make_custom(1, 3, 400, 64, dtype="f32", seed=1)
    beta[1, ::7] = 60.0
    q[:, 2], k[:, 2] = 6 * q[:, 2], 6 * k[:, 2]
    x = [a.cuda() for a in (q, k, v, beta)]
    dout = torch.randn(q.shape, generator=torch.Generator().manual_seed(2)).cuda()
    out, lse = fem.fem_fwd_f32(*x)
    first = fem.fem_bwd_f32(*x, out, lse, dout)
    plain = beta * (v.amax(2) - v.amin(2))[0] < 150.0
    for _ in range(3):
        again = fem.fem_bwd_f32(*x, out, lse, dout)
        assert torch.equal(first[0], again[0]) and torch.equal(first[1], again[1])
        for h in range(3):
            assert torch.equal(first[2][:, h, :, plain[h].cuda()], again[2][:, h, :, plain[h].cuda()])

"""The tiled gradients of the fp32 read on the GPU (needs a GB300): edges of the 64-row
and 64-key tiles and of the channel tiles, clusters sharing a tile, channels too wide for
the factored exponentials, and priors peaked enough to go pair by pair.

fp32 throughout: 1e-4 of each gradient's scale against the float64 oracle, as the
pair-by-pair kernels.  The gradients take exp(beta (v - o)) of the forward's rounded
output, an error of beta |o| 2^-24: 5e-5 at beta = 200, |o| <= 4.
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


def _check(B, H, T, d, causal, beta_hi=20.0, scale=1.0, tol=1e-4):
    q, k, v, beta = W.make_custom(B, H, T, d, dtype="f32", seed=T + d, beta_hi=beta_hi)
    q, k = q * scale, k * scale
    beta[:, 0] = 0.0
    dout = torch.randn(q.shape, generator=torch.Generator().manual_seed(T), dtype=torch.float32)
    dev = torch.device("cuda", 0)
    x = [a.to(dev) for a in (q, k, v, beta)]
    out, lse = fem.fem_fwd_f32(*x, causal=causal)
    got = fem.fem_bwd_f32(*x, out, lse, dout.to(dev), causal=causal)
    fem.check_device_error()
    ref = oracle.fem_backward(q, k, v, beta, dout, causal)
    for g, r in zip(got, ref):
        r = np.asarray(r)
        assert np.isfinite(g.cpu().numpy()).all()
        assert np.abs(g.cpu().double().numpy() - r).max() <= tol * max(1.0, np.abs(r).max())


@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("B,H,T,d", [(1, 1, 64, 16), (2, 2, 65, 33), (1, 2, 127, 64), (1, 1, 129, 100), (1, 2, 96, 128),
                                     (1, 1, 200, 1), (2, 1, 257, 48), (1, 1, 700, 64)])
def test_tiled_gradients_match_oracle(B, H, T, d, causal):
    _check(B, H, T, d, causal)


@pytest.mark.parametrize("causal", [True, False])
def test_wide_channels(causal):
    _check(1, 2, 150, 40, causal, beta_hi=200.0)


@pytest.mark.parametrize("d", [32, 128])
def test_peaked_prior(d):
    _check(1, 2, 140, d, True, scale=4.0)

"""The tiled fp32 read on the GPU (needs a GB300): edges of its 64-row and 64-key
tiles, widths that fill no channel tile, both bank forms, and entries it evaluates
again key by key.

fp32 products and sums throughout: the fp32 read's bound, 1e-4 against the float64
oracle (values of unit spread).
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


def _run(q, k, v, beta, causal):
    dev = torch.device("cuda", 0)
    out = torch.full(q.shape, float("nan"), dtype=torch.float32, device=dev)
    out, lse = fem.fem_fwd_f32(*(x.to(dev) for x in (q, k, v, beta)), causal=causal, out=out)
    fem.check_device_error()
    return out.cpu().double().numpy(), lse.cpu().double().numpy()


@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("B,H,T,d", [(1, 1, 80, 16), (1, 2, 63, 34), (64, 1, 64, 1), (1, 3, 65, 64), (1, 2, 129, 33),
                                     (2, 1, 200, 100), (1, 2, 300, 128), (64, 1, 32, 17)])
def test_tile_matches_oracle(B, H, T, d, causal):
    q, k, v, beta = W.make_custom(B, H, T, d, dtype="f32", seed=T + d)
    beta[:, 0] = 0.0
    out, lse = _run(q, k, v, beta, causal)
    ref, ref_lse = oracle.fem_read(q, k, v, beta, causal)
    assert np.abs(out - ref).max() <= 1e-4
    assert np.abs(lse - ref_lse).max() <= 1e-4


def test_tile_wide_tilt_and_peaked_prior():
    """beta up to 1000 and scores spread over tens of nats: most early rows of a tile see no key
    near the bank's shift, and the prior's heavy key lies far below the largest value."""
    q, k, v, beta = W.make_custom(1, 2, 160, 32, dtype="f32", beta_lo=1.0, beta_hi=1000.0, seed=3)
    for scale in (1.0, 4.0):
        out, _ = _run(q * scale, k * scale, v, beta, True)
        ref, _ = oracle.fem_read(q * scale, k * scale, v, beta, True)
        assert np.abs(out - ref).max() <= 1e-4


def test_tile_row_ignores_infinite_value_of_a_later_key():
    q, k, v, beta = W.make_custom(1, 1, 128, 16, dtype="f32", seed=5)
    ref, _ = oracle.fem_read(q, k, v, beta, True)
    v[0, 0, 100, 3] = float("inf")
    out, _ = _run(q, k, v, beta, True)
    assert np.abs(out[0, 0, :100] - ref[0, 0, :100]).max() <= 1e-4


def test_tile_bf16_narrow_heads():
    q, k, v, beta = W.make_custom(2, 2, 150, 32, seed=9)
    dev = torch.device("cuda", 0)
    out, _ = fem.fem_fwd(*(x.to(dev) for x in (q, k, v, beta)), causal=True)
    ref, _ = oracle.fem_read(q, k, v, beta, True)
    assert np.abs(out.cpu().double().numpy() - ref).max() <= 1e-4

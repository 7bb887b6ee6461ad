"""The fp32 read on the GPU (needs a GB300) where a prior's weights and the tilt leave fp32's
range on either side: the key with the largest value has a weight that underflows, and the
keys with weight lie below it by more nats than fp32 holds.

The fp32 read's bound, 1e-4, against the float64 oracle.
"""
import numpy as np
import pytest

import oracle
from paper_2602_07160_gb300 import build, fem
from paper_2602_07160_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    return fem.load()


def _check(B, H, T, d, causal):
    q, k, v, beta = W.make_custom(B, H, T, d, dtype="f32", beta_lo=2.0, beta_hi=1000.0, seed=T + d)
    q, k = q * 6, k * 6  # scores spread over some hundreds of nats
    beta[:, 0] = 0.0
    out, lse = fem.fem_fwd_f32(*(x.cuda() for x in (q, k, v, beta)), causal=causal)
    fem.check_device_error()
    ref, ref_lse = oracle.fem_read(q, k, v, beta, causal)
    assert np.abs(out.cpu().double().numpy() - ref).max() <= 1e-4
    assert np.abs(lse.cpu().double().numpy() - ref_lse).max() <= 1e-4


@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("T,d", [(3, 1), (33, 16), (64, 20), (128, 40), (70, 64)])
def test_short_rows(T, d, causal):
    _check(1, 2, T, d, causal)


@pytest.mark.parametrize("B,H,T,d", [(1, 2, 33, 200), (3, 1, 128, 129), (1, 1, 130, 256), (80, 1, 28, 33), (300, 1, 9, 100)])
@pytest.mark.parametrize("causal", [True, False])
def test_rows_by_warps(B, H, T, d, causal):
    _check(B, H, T, d, causal)


@pytest.mark.parametrize("T,first,last,causal", [(192, 64, 128, False), (200, 0, 64, False), (300, 70, 300, True), (60, 10, 30, True)])
def test_keys_with_a_score_of_minus_infinity(T, first, last, causal):
    """Keys masked by a score of -inf, whole tiles of them among those: no weight, for the read and
    for its log-normaliser (in the oracle their scores are some -1e5)."""
    q, k, v, beta = W.make_custom(1, 1, T, 16, dtype="f32", seed=T)
    q = q.abs() + 0.1
    far = k.clone()
    far[:, :, first:last] = -1e5
    k[:, :, first:last] = -float("inf")
    out, lse = fem.fem_fwd_f32(*(x.cuda() for x in (q, k, v, beta)), causal=causal)
    fem.check_device_error()
    ref, ref_lse = oracle.fem_read(q, far, v, beta, causal)
    assert np.abs(out.cpu().double().numpy() - ref).max() <= 1e-4
    assert np.abs(lse.cpu().double().numpy() - ref_lse).max() <= 1e-4


@pytest.mark.parametrize("B,H,T,d", [(1, 2, 129, 16), (1, 1, 200, 128), (2, 1, 90, 64), (1, 1, 333, 33), (1, 1, 700, 60)])
@pytest.mark.parametrize("causal", [True, False])
def test_tiles(B, H, T, d, causal):
    _check(B, H, T, d, causal)


def test_tiles_of_bf16_narrow_heads():
    q, k, v, beta = W.make_custom(1, 2, 300, 32, beta_lo=2.0, beta_hi=1000.0, seed=4)
    q, k = q * 6, k * 6
    out, _ = fem.fem_fwd(*(x.cuda() for x in (q, k, v, beta)), causal=True)
    ref, _ = oracle.fem_read(q, k, v, beta, True)
    assert np.abs(out.cpu().double().numpy() - ref).max() <= 1e-4

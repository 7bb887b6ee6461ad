"""The fp32 GLA-prior read in chunks (fem_gla_fwd; needs a GB300) at chunk and channel-block
remainders, with values of wide spread (rows that don't see the chunk's largest value), with
resets (a step's decay -inf), and over several runs of chunks and groups of heads.

The fp32 read's bound against the float64 oracle, 1e-4 times the values' spread.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_07160_gb300 import build, fem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    return fem.load()


def _inputs(seed, B, H, T, m, d, v_scale=1.0):
    dev = torch.device("cuda", 0)
    g = torch.Generator(device=dev).manual_seed(seed)
    qf = torch.relu(torch.randn((B, H, T, m), generator=g, device=dev)) + 0.05
    kf = torch.relu(torch.randn((B, H, T, m), generator=g, device=dev)) + 0.05
    v = torch.randn((B, H, T, d), generator=g, device=dev) * v_scale
    logdecay = -0.3 * torch.rand((B, H, T), generator=g, device=dev)
    beta = torch.exp(torch.empty((H, d), device=dev).uniform_(np.log(0.05), np.log(20.0), generator=g))
    beta[0, : min(3, d)] = 0.0
    return qf, kf, v, logdecay, beta


@pytest.mark.parametrize("B,H,T,m,d,v_scale,reset", [(1, 1, 1, 16, 1, 1.0, False), (1, 2, 64, 16, 24, 1.0, False),
                                                     (2, 1, 65, 32, 64, 1.0, True), (1, 2, 128, 64, 65, 6.0, False),
                                                     (1, 1, 129, 64, 128, 1.0, True), (1, 1, 577, 32, 155, 6.0, True)])
def test_chunks_match_oracle(B, H, T, m, d, v_scale, reset):
    qf, kf, v, logdecay, beta = _inputs(T + d, B, H, T, m, d, v_scale)
    finite = logdecay.clone()
    if reset:
        logdecay[..., 10::37] = -float("inf")
        finite[..., 10::37] = -1e5
    out = torch.full(v.shape, float("nan"), dtype=torch.float32, device=v.device)
    out, logz = fem.fem_gla_fwd(qf, kf, v, logdecay, beta, out=out)
    fem.check_device_error()
    ref, ref_lz = oracle.gla_read(*(x.cpu() for x in (qf, kf, v, finite, beta)))
    err = np.abs(out.cpu().double().numpy() - ref)
    assert np.isfinite(err).all() and err.max() <= 1e-4 * v_scale
    assert np.abs(logz.cpu().double().numpy() - ref_lz).max() <= 1e-4


def test_runs_of_chunks_continue_the_state():
    """More chunks than a workspace holds: from a later first step on, chunks and runs fall
    elsewhere and the state before that step has decayed away."""
    qf, kf, v, logdecay, beta = _inputs(3, 1, 1, 350000, 64, 155)
    whole, _ = fem.fem_gla_fwd(qf, kf, v, logdecay, beta)
    rest, _ = fem.fem_gla_fwd(*(x[:, :, 1000:].contiguous() for x in (qf, kf, v, logdecay)), beta)
    fem.check_device_error()
    assert (whole[:, :, 2000:] - rest[:, :, 1000:]).abs().max().item() <= 1e-4


def test_groups_of_heads():
    """More heads than a workspace holds: the last ones by themselves give the same."""
    qf, kf, v, logdecay, beta = _inputs(4, 84, 1, 4096, 64, 155)
    whole, _ = fem.fem_gla_fwd(qf, kf, v, logdecay, beta)
    part, _ = fem.fem_gla_fwd(*(x[-3:].contiguous() for x in (qf, kf, v, logdecay)), beta)
    fem.check_device_error()
    assert torch.equal(whole[-3:], part)

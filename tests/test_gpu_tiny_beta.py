"""The fp32 read at beta near and below the normal range on the GPU (needs a GB300), in each
of its kernels: the read there is the prior mean up to beta times the squared spread.

The fp32 read's bound, 1e-4, against the float64 oracle at beta = 0.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_07160_gb300 import build, fem
from paper_2602_07160_gb300 import workloads as W

pytestmark = pytest.mark.gpu

BETAS = [1e-45, 1e-44, 1e-41, 2.9e-39, 1.2e-38, 1e-37, 1e-20, 1e-12]


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    return fem.load()


@pytest.mark.parametrize("dtype,T,d", [("f32", 200, 64), ("f32", 70, 128), ("f32", 64, 16), ("f32", 20, 200), ("f32", 300, 150),
                                       ("bf16", 200, 32), ("bf16", 40, 16)])
def test_tiny_beta_reads_the_mean(dtype, T, d):
    q, k, v, _ = W.make_custom(1, 2, T, d, dtype=dtype, seed=T)
    beta = W.beta_grid(2, d, BETAS)
    read = fem.fem_fwd_f32 if dtype == "f32" else fem.fem_fwd
    out, lse = read(*(x.cuda() for x in (q, k, v, beta)), causal=True)
    fem.check_device_error()
    ref, ref_lse = oracle.fem_read(q, k, v, torch.zeros_like(beta), True)
    assert np.abs(out.cpu().double().numpy() - ref).max() <= 1e-4
    assert np.abs(lse.cpu().double().numpy() - ref_lse).max() <= 1e-4


@pytest.mark.parametrize("T", [200, 640])
def test_tiny_beta_on_the_tensor_core_gla_read(T):
    """The tensor-core GLA read's bound, 2e-2 at unit spread, on both its forms."""
    g = torch.Generator().manual_seed(T)
    qf, kf = (torch.relu(torch.randn((1, 1, T, 64), generator=g)) + 0.05 for _ in range(2))
    v = torch.randn((1, 1, T, 64), generator=g)
    logdecay = -0.02 * torch.rand((1, 1, T), generator=g)
    beta = W.beta_grid(1, 64, BETAS)
    out, _ = fem.fem_gla_fwd_tc(*(x.cuda() for x in (qf, kf, v, logdecay, beta)))
    fem.check_device_error()
    ref, _ = oracle.gla_read(qf, kf, v, logdecay, torch.zeros_like(beta))
    assert np.abs(out.cpu().double().numpy() - ref).max() <= 2e-2

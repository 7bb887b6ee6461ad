"""The fp32 GLA-prior read with values so wide that most rows lie under fp32's range of their
chunk's largest (needs a GB300): chunk and channel remainders, resets, and values and outputs
that are not 16-byte aligned.

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


@pytest.mark.parametrize("T,m,d,scale,shift", [(3, 16, 5, 30.0, 0), (64, 64, 64, 30.0, 0), (65, 32, 70, 5.0, 0), (200, 16, 130, 100.0, 0),
                                               (333, 64, 36, 10.0, 1), (40, 32, 64, 3.0, 3)])
def test_wide_values(T, m, d, scale, shift):
    g = torch.Generator().manual_seed(T)
    qf, kf = (torch.relu(torch.randn((1, 2, T, m), generator=g)) + 0.05 for _ in range(2))
    v = torch.randn((1, 2, T, d), generator=g) * scale
    decay = -0.3 * torch.rand((1, 2, T), generator=g)
    decay[..., 9::31] = -1e5
    beta = torch.exp(torch.empty((2, d)).uniform_(np.log(0.05), np.log(200.0), generator=g))
    beta[:, 0] = 0.0
    # `shift` floats past a 16-byte boundary
    vd = torch.empty(v.numel() + 4, device="cuda")[shift:shift + v.numel()].view(v.shape).copy_(v)
    out = torch.full((v.numel() + 4,), float("nan"), device="cuda")[shift:shift + v.numel()].view(v.shape)
    out, logz = fem.fem_gla_fwd(qf.cuda(), kf.cuda(), vd, decay.cuda(), beta.cuda(), out=out)
    fem.check_device_error()
    ref, ref_lz = oracle.gla_read(qf, kf, v, decay, beta)
    assert np.abs(out.cpu().double().numpy() - ref).max() <= 1e-4 * scale
    assert np.abs(logz.cpu().double().numpy() - ref_lz).max() <= 1e-4

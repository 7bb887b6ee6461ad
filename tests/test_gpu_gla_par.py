"""The chunk-parallel GLA-prior read (fem_gla_fwd_tc from three chunks on; needs a GB300)
at chunk remainders, more chunks than one prefix scan's 32 lanes, several heads' anchors
and scales, strong decay (the state underflows between chunks) and values of wide spread.

The bf16 read's bounds against the float64 oracle, max abs 2e-2 and mean abs 2e-3, times
the values' spread; its mean error grows like 2^-9 over the square root of the keys a row
sees, and with decay at most 2 a step a row sees two or three.
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


@pytest.mark.parametrize("B,H,T,g_scale,v_scale", [(1, 1, 257, 0.3, 1.0), (2, 3, 383, 0.3, 1.0), (1, 2, 384, 0.02, 1.0),
                                                   (1, 1, 4225, 0.1, 1.0), (1, 2, 500, 2.0, 1.0), (1, 2, 640, 0.05, 3.0)])
def test_parallel_chunks_match_oracle(B, H, T, g_scale, v_scale):
    g = torch.Generator().manual_seed(T)
    qf = torch.relu(torch.randn((B, H, T, 64), generator=g)) + 0.05
    kf = torch.relu(torch.randn((B, H, T, 64), generator=g)) + 0.05
    v = torch.randn((B, H, T, 64), generator=g) * v_scale
    logdecay = -g_scale * torch.rand((B, H, T), generator=g)
    beta = torch.exp(torch.empty((H, 64)).uniform_(np.log(0.05), np.log(20.0), generator=g))
    beta[:, :3] = 0.0
    dev = torch.device("cuda", 0)
    out = torch.full(v.shape, float("nan"), dtype=torch.float32, device=dev)
    out, logz = fem.fem_gla_fwd_tc(*(x.to(dev) for x in (qf, kf, v, logdecay, beta)), out=out)
    fem.check_device_error()
    ref, ref_logz = oracle.gla_read(qf, kf, v, logdecay, beta)
    err = np.abs(out.cpu().double().numpy() - ref)
    assert np.isfinite(err).all()
    assert err.max() <= 2e-2 * v_scale and err.mean() <= 2e-3 * v_scale
    assert np.abs(logz.cpu().double().numpy() - ref_logz).max() <= 1e-2

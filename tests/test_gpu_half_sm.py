"""The d = 64 read in its two-CTAs-per-SM form (grids of more CTAs than SMs; needs a GB300).

The same heads read in a small batch (one CTA per SM at most) run the other form of the
kernel: the two perform the same operations, up to the order of the two factors of a
rescale, so they agree to fp32 rounding (a few ulp of |o| <= 8 and, through 1/beta, 1e-5).
A sample of heads is checked against the float64 oracle at the bf16 read's bounds.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_07160_gb300 import build, fem
from paper_2602_07160_gb300 import workloads as W

pytestmark = pytest.mark.gpu

B, H = 40, 8  # 320 heads: more CTAs than SMs from the first query tile on


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    return fem.load()


@pytest.mark.parametrize("T,causal,scale", [(1, True, 1.0), (127, True, 1.0), (128, False, 1.0), (129, True, 1.0),
                                            (256, True, 1.0), (385, True, 1.0), (300, False, 1.0), (640, True, 1.0),
                                            (300, True, 2.0), (450, True, 2.0)])
def test_two_ctas_per_sm(T, causal, scale):
    q, k, v, beta = W.make_custom(B, H, T, 64, seed=T, beta_hi=50.0 if scale > 1 else 20.0)
    q, k = q * scale, k * scale
    beta[:, 0] = 0.0
    dev = torch.device("cuda", 0)
    d = [x.to(dev) for x in (q, k, v, beta)]
    out = torch.full(q.shape, float("nan"), dtype=torch.float32, device=dev)
    out, lse = fem.fem_fwd(*d, causal=causal, out=out)
    fem.check_device_error()
    for b in (0, 17, B - 1):
        part, part_lse = fem.fem_fwd(*(x[b:b + 1].contiguous() for x in d[:3]), d[3], causal=causal)
        fem.check_device_error()
        assert (out[b] - part[0]).abs().max().item() <= 1e-5
        assert (lse[b] - part_lse[0]).abs().max().item() <= 1e-5
    ref, ref_lse = oracle.fem_read(q[17:18], k[17:18], v[17:18], beta, causal)
    err = np.abs(out[17].cpu().double().numpy() - ref[0])
    assert err.max() <= 2e-2 and err.mean() <= 2e-3
    assert np.abs(lse[17].cpu().double().numpy() - ref_lse[0]).max() <= (2e-3 if scale == 1.0 else 2e-2)

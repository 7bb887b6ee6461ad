"""The decode read of the shorter caches in one launch (a cluster of CTAs per head; needs a GB300)
at the edges of its chunks, its cluster sizes and its rule, against the float64 oracle.

The decode read's bounds, max abs 1e-3 and mean abs 1e-4 (fp32 arithmetic on bf16 inputs).
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


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,H,T", [(1, 1, 1), (2, 1, 64), (1, 3, 65), (1, 2, 129), (1, 1, 512), (1, 1, 513),
                                   (1, 2, 1000), (1, 1, 1024), (1, 1, 1025), (76, 1, 260), (77, 1, 260)])
def test_cluster_matches_oracle(B, H, T, d):
    g = torch.Generator().manual_seed(T + d)
    q = torch.randn((B, H, d), generator=g).bfloat16()
    k = torch.randn((B, H, T, d), generator=g).bfloat16()
    v = torch.randn((B, H, T, d), generator=g).bfloat16()
    beta = torch.exp(torch.empty((H, d)).uniform_(np.log(0.05), np.log(20.0), generator=g))
    beta[0, :3] = 0.0
    dev = torch.device("cuda", 0)
    out, lse = fem.fem_decode(*(x.to(dev) for x in (q, k, v, beta)))
    fem.check_device_error()
    for b in {0, B - 1}:
        ref, ref_lse = oracle.decode_read(q[b : b + 1], k[b : b + 1], v[b : b + 1], beta)
        err = np.abs(out[b : b + 1].cpu().double().numpy() - ref)
        assert err.max() <= 1e-3 and err.mean() <= 1e-4
        assert np.abs(lse[b : b + 1].cpu().double().numpy() - ref_lse).max() <= 1e-4

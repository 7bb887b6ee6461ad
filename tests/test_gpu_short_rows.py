"""The fp32 read of few rows of few keys (a block per row; needs a GB300) at the edges of its keys,
channels and shared memory, against the float64 oracle at the fp32 read's bound, max abs 1e-4 for
values of unit spread (times the spread for wider ones); bf16 inputs at d = 16 and 32 likewise.
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


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("B,H,T,d,causal,scale", [(1, 1, 1, 16, True, 1.0), (1, 1, 64, 16, True, 1.0), (2, 3, 79, 32, False, 1.0),
                                                  (1, 2, 33, 1, True, 1.0), (1, 2, 47, 17, False, 1.0), (1, 2, 40, 128, True, 1.0),
                                                  (1, 2, 47, 128, True, 1.0), (1, 1, 20, 256, False, 1.0), (1, 2, 31, 130, True, 1.0),
                                                  (1, 2, 64, 16, True, 8.0), (1, 1, 128, 16, True, 1.0), (1, 8, 100, 32, True, 1.0),
                                                  (1, 1, 87, 64, False, 1.0)])
def test_short_rows(B, H, T, d, causal, scale, dtype):
    if dtype == "bf16" and d not in (16, 32):
        pytest.skip("the bf16 read takes d 16 and 32 here")
    q, k, v, beta = W.make_custom(B, H, T, d, seed=T + d)
    q, k, v = (x.float() for x in (q, k, v))
    v = (v * scale).bfloat16().float()
    beta[:, 0] = 0.0
    dev = torch.device("cuda", 0)
    cast = (lambda x: x.bfloat16()) if dtype == "bf16" else (lambda x: x)
    out = torch.full(q.shape, float("nan"), dtype=torch.float32, device=dev)
    call = fem.fem_fwd if dtype == "bf16" else fem.fem_fwd_f32
    out, lse = call(cast(q).to(dev), cast(k).to(dev), cast(v).to(dev), beta.to(dev), causal=causal, out=out)
    fem.check_device_error()
    ref, ref_lse = oracle.fem_read(q, k, v, beta, causal)
    assert np.abs(out.cpu().double().numpy() - ref).max() <= 1e-4 * scale
    assert np.abs(lse.cpu().double().numpy() - ref_lse).max() <= 1e-4

"""The one-launch pre-pass (needs a GB300) at the edges of its key tiles, of its two instances
(one or two tiles a warp) and of the rule beyond it: the bf16 read, whose bank it makes, against
the float64 oracle at the read's bounds, max abs 2e-2 and mean abs 2e-3.
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


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("T,causal", [(1, True), (128, False), (129, True), (256, True), (257, False), (384, True),
                                      (385, True), (511, True), (512, False), (513, True)])
def test_prepass_tiles(T, causal, d):
    q, k, v, beta = W.make_custom(2, 2, T, d, seed=T + d)
    beta[:, :2] = 0.0
    dev = torch.device("cuda", 0)
    out = torch.full(q.shape, float("nan"), dtype=torch.float32, device=dev)
    out, lse = fem.fem_fwd(*(x.to(dev) for x in (q, k, v, beta)), causal=causal, out=out)
    fem.check_device_error()
    ref, ref_lse = oracle.fem_read(q, k, v, beta, causal)
    err = np.abs(out.cpu().double().numpy() - ref)
    assert err.max() <= 2e-2 and err.mean() <= 2e-3
    assert np.abs(lse.cpu().double().numpy() - ref_lse).max() <= 2e-3

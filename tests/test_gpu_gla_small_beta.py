"""The fp32 GLA-prior read at small beta on the GPU (needs a GB300): down to zero the read tends
to the prior mean, in lone chunks, over several, and where only some channels of a block are
small; at the same small beta with values of size 1 / beta it is a tilted read like any other.

Against the float64 oracle (beta = 0 below 1e-8, where its own logarithms end): 1e-5 at unit
spread for the small form's ratio of sums of a few hundred terms and its logarithm; the log
form's two logarithms, 1e-6 / beta, for values of size 1 / beta.
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


def _inputs(T, m, d):
    g = torch.Generator().manual_seed(T + d)
    qf, kf = (torch.relu(torch.randn((1, 2, T, m), generator=g)) + 0.05 for _ in range(2))
    v = torch.randn((1, 2, T, d), generator=g)
    return qf, kf, v, -0.3 * torch.rand((1, 2, T), generator=g)


@pytest.mark.parametrize("T,m,d", [(5, 16, 24), (64, 64, 64), (65, 32, 100), (300, 64, 155), (1000, 16, 3)])
def test_small_beta_tends_to_the_mean(T, m, d):
    qf, kf, v, g = _inputs(T, m, d)
    beta = W.beta_grid(2, d, [0.0, 2.0, 1e-2, 1e-4, 1e-6, 1e-12, 1e-22, 1e-37, 1e-41])
    out, _ = fem.fem_gla_fwd(*(x.cuda() for x in (qf, kf, v, g, beta)))
    fem.check_device_error()
    ref, _ = oracle.gla_read(qf, kf, v, g, torch.where(beta < 1e-8, 0.0, beta))
    assert np.abs(out.cpu().double().numpy() - ref).max() <= 1e-5


@pytest.mark.parametrize("T", [40, 200])
def test_small_beta_with_large_values(T):
    qf, kf, v, g = _inputs(T, 32, 64)
    beta = W.beta_grid(2, 64, [1e-3, 1e-6, 1e-9])
    scale = 3.0 / beta[None, :, None, :]
    out, _ = fem.fem_gla_fwd(*(x.cuda() for x in (qf, kf, v * scale, g, beta)))
    fem.check_device_error()
    ref, _ = oracle.gla_read(qf, kf, v * scale, g, beta)
    assert (np.abs(out.cpu().double().numpy() - ref) * beta.double().numpy()[None, :, None, :]).max() <= 3e-6

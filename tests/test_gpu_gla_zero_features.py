"""The GLA-prior reads with features that are zero (ReLU without an offset) on the GPU (needs
a GB300): rows whose features meet no key of their own chunk read the state alone, also where
the chunk's values lie far above the state's.

Bounds against the float64 oracle: fp32 1e-4 times the values' spread; tensor cores 2^-8 of the
spread (the linear bank's entries) or 2^-8 / beta (the shifted ones').
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


@pytest.mark.parametrize("entry", ["fem_gla_fwd", "fem_gla_fwd_tc"])
@pytest.mark.parametrize("T", [200, 384, 700])
def test_rows_without_a_key_of_their_chunk(entry, T):
    g = torch.Generator().manual_seed(T)
    qf, kf = (torch.relu(torch.randn((1, 2, T, 64), generator=g)) for _ in range(2))
    v = torch.randn((1, 2, T, 64), generator=g).clamp(-2.0, 2.0)
    c0 = (T - 1) // 128 * 128  # the last chunk: feature 0 has no key there, its largest value lies far above
    kf[:, :, :4, 0] = 1.0
    kf[:, :, c0:, 0] = 0.0
    qf[:, :, c0::3] = 0.0
    qf[:, :, c0::3, 0] = 0.7
    v[:, :, T - 2] = 4.2
    g_t = -0.02 * torch.rand((1, 2, T), generator=g)
    beta = torch.tensor([50.0, 20.0, 1.0, 0.1, 0.0])[torch.arange(128) % 5].reshape(2, 64)
    out, logz = getattr(fem, entry)(*(x.to("cuda") for x in (qf, kf, v, g_t, beta)))
    fem.check_device_error()
    ref, ref_lz = oracle.gla_read(qf, kf, v, g_t, beta)
    assert np.isfinite(ref).all()
    spread = float(v.max() - v.min())
    b = beta.double().numpy()[None, :, None, :]
    tol = 1e-4 * spread if entry == "fem_gla_fwd" else np.where(b < 0.25, 2.0**-8 * spread, 2.0**-8 / np.maximum(b, 0.25) + 2e-3)
    assert (np.abs(out.cpu().double().numpy() - ref) <= tol).all()
    assert np.abs(logz.cpu().double().numpy() - ref_lz).max() <= (1e-4 if entry == "fem_gla_fwd" else 2.0**-7)

"""The tiled gradients of the fp32 read are linear in the cotangent on the GPU (needs a
GB300): small and large cotangents, rows of very different ones, and channels whose
spread times beta lies on both sides of the factored exponentials' bound.

Each gradient within 1e-4 of its own largest entry (the fp32 gradients' bound, without a
floor, so that small cotangents count); dq also row by row, within 1e-4 of the row's
cotangent times the largest key entry.
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


def _inputs(kind, T, d, beta, heads=1):
    g = torch.Generator().manual_seed(T + d)
    q, k = (torch.randn((1, heads, T, d), generator=g) for _ in range(2))
    v = torch.rand((1, heads, T, d), generator=g) * 2 - 1  # half the spread is 1
    if kind == "low":  # one value far below the others, seen alone by the first row that sees it
        v[:, :, 0] = -21.0
    b = torch.tensor(beta)[torch.arange(heads * d) % len(beta)].reshape(heads, d)
    return q, k, v, b, torch.randn((1, heads, T, d), generator=g)


@pytest.mark.parametrize("kind,T,d,beta", [("uniform", 512, 16, [60.0, 70.0, 71.5, 74.0, 84.0]), ("low", 200, 40, [6.0, 7.0, 7.7]),
                                           ("uniform", 130, 128, [0.0, 5.0, 68.0])])
@pytest.mark.parametrize("scale", [1.0, 1e-8, 1e-30, 1e6, "rows"])
def test_gradients_scale_with_the_cotangent(kind, T, d, beta, scale):
    q, k, v, b, dout = _inputs(kind, T, d, beta)
    if scale == "rows":
        dout = dout * 10.0 ** (-10 * torch.rand((1, 1, T, 1), generator=torch.Generator().manual_seed(T)))
        dout[:, :, 5::9] = 0.0
    else:
        dout = dout * scale
    dev = torch.device("cuda", 0)
    x = [a.to(dev) for a in (q, k, v, b)]
    out, lse = fem.fem_fwd_f32(*x, causal=True)
    got = [g.cpu().double().numpy() for g in fem.fem_bwd_f32(*x, out, lse, dout.to(dev), causal=True)]
    fem.check_device_error()
    ref = oracle.fem_backward(q, k, v, b, dout, True)
    for g, r in zip(got, ref):
        assert np.abs(g - r).max() <= 1e-4 * np.abs(r).max()
    row = np.abs(dout.double().numpy()).max(-1) * float(k.abs().max())
    assert (np.abs(got[0] - ref[0]).max(-1) <= 1e-4 * row).all()

"""The gated read's two banks from one plan and one bank launch (needs a GB300): against the two
plain reads it is made of, lambda picking each, at the first length with separate plan and bank
launches, at ragged tiles, and where V is large enough for the bank pass to run backwards.

o = g (mu + lambda (F - mu)) in fp32 with g = 1: for lambda in {0, 1} a rounding or two of values
of unit size (mean abs 1e-5), except at entries that one of the calls completes exactly and the
other does not, which differ by the bf16 read's error (max abs 2e-2).
"""
import pytest
import torch

from paper_2602_07160_gb300 import build, fem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    return fem.load()


@pytest.mark.parametrize("B,H,T,d", [(1, 1, 513, 64), (2, 3, 700, 128), (1, 2, 640, 64), (1, 17, 16384, 128)])
def test_gated_read_is_its_two_reads(B, H, T, d):
    dev = torch.device("cuda", 0)
    g = torch.Generator(device=dev).manual_seed(T + d)
    q, k, v = (torch.randn((B, H, T, d), generator=g, device=dev).bfloat16() for _ in range(3))
    beta = 0.05 + 3.0 * torch.rand((H, d), generator=g, device=dev)
    one = torch.ones((B, H, T, d), device=dev)
    for lam, b in ((one, beta), (torch.zeros_like(one), torch.zeros_like(beta))):
        out, lse = fem.fem_fwd_gated(q, k, v, beta, lam, one)
        ref, ref_lse = fem.fem_fwd(q, k, v, b)
        fem.check_device_error()
        err = (out - ref).abs()
        assert err.max().item() <= 2e-2 and err.mean().item() <= 1e-5
        assert (lse - ref_lse).abs().max().item() <= 1e-5

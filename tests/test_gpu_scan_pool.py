"""The GLA reads' memory pool on the GPU (needs a GB300): a call whose workspace is larger than
the pool keeps leaves no more than that behind.
"""
import pytest
import torch

from paper_2602_07160_gb300 import build, fem

pytestmark = pytest.mark.gpu

KEEP = 320 << 20


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    return fem.load()


def test_pool_returns_what_is_beyond_its_bound():
    T = 900_000  # one head: 66 KB a chunk of 128 steps, 460 MB
    qf, kf = (torch.rand((1, 1, T, 64), device="cuda") for _ in range(2))
    v, out = torch.randn((1, 1, T, 64), device="cuda"), torch.empty((1, 1, T, 64), device="cuda")
    g, logz = torch.zeros((1, 1, T), device="cuda"), torch.empty((1, 1, T), device="cuda")
    beta = torch.ones((1, 64), device="cuda")

    def call(n):
        fem.fem_gla_fwd_tc(*(x[:, :, :n].contiguous() for x in (qf, kf, v, g)), beta, out=out[:, :, :n].contiguous(),
                           logz=logz[:, :, :n].contiguous())
        fem.check_device_error()
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    before = call(1000)  # the kernels are loaded
    assert before - call(T) <= KEEP + (32 << 20)

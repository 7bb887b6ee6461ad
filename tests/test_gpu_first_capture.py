"""Calls recorded into a graph as the first of a process (needs a GB300): the workspace pool is
created under the capture, and a replay gives what the same call gives directly."""
import os
import subprocess
import sys

import pytest

from paper_2602_07160_gb300 import build

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CALLS = {
    "gla_tc": "fem.fem_gla_fwd_tc(qf, qf, v, -0.1 * qf[..., 0].contiguous(), beta)",
    "backward": "fem.fem_bwd_f32(qf, qf, v, beta, out, lse, v)",
}
PROGRAM = """
import torch
from paper_2602_07160_gb300 import fem
dev = torch.device("cuda", 0)
g = torch.Generator().manual_seed(1)
qf = torch.rand((1, 2, 600, 64), generator=g).to(dev)
v = torch.randn((1, 2, 600, 64), generator=g).to(dev)
beta = torch.full((2, 64), 0.5, device=dev)
out, lse = fem.fem_fwd_f32(qf, qf, v, beta)  # no workspace
def call():
    return {call}
torch.cuda.synchronize()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph):
    held = call()
graph.replay()
graph.replay()
direct = call()
torch.cuda.synchronize()
fem.check_device_error()
assert all(torch.isfinite(a).all() for a in direct)
assert all(torch.allclose(a, b, rtol=1e-5, atol=1e-5 * b.abs().max().item()) for a, b in zip(held, direct))
"""


@pytest.mark.parametrize("name", sorted(CALLS))
def test_first_call_under_capture(name):
    build.build()
    done = subprocess.run([sys.executable, "-c", PROGRAM.replace("{call}", CALLS[name])], cwd=ROOT, capture_output=True,
                          text=True, timeout=240)
    assert done.returncode == 0, done.stderr[-2000:]

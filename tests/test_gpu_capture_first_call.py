"""The first call of a process recorded by a stream capture: products and the gradient allocate
stream-ordered scratch, and what their first call sets up must not end the capture.  Each case
runs in a process of its own; the replays give what the same call gives outside a capture."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = """
import sys
import torch
import paper_1309_0302_gb300 as G
g = torch.Generator(device="cuda").manual_seed(3)
def randn(*s):
    return torch.randn(*s, generator=g, device="cuda")
Z, B, C, gL, A1 = randn(300, 260), randn(260, 8), randn(300, 8), randn(300, 260), randn(260, 4)
call = {"mul_ZB": lambda: G.mul_ZB(Z, B), "mul_ZtC": lambda: G.mul_ZtC(Z, C),
        "unaligned": lambda: G.mul_ZB(Z[:, 1:258], B[:257]),
        "backward": lambda: G.backward(Z, A1, 1, [], gL=gL)}[sys.argv[1]]
G.library()
torch.cuda.synchronize()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph):
    Y = call()
for _ in range(2):
    Y.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(Y, call())
print("captured")
"""


@pytest.mark.parametrize("call", ["mul_ZB", "mul_ZtC", "unaligned", "backward"])
def test_first_call_under_capture(call):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    run = subprocess.run([sys.executable, "-c", CHILD, call], cwd=root, capture_output=True, text=True, timeout=300)
    assert run.returncode == 0 and "captured" in run.stdout, run.stderr[-2000:]

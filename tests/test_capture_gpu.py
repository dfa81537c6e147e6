"""The controller's calls under stream capture, as the first calls of a process and after
others: replaying the graph gives what the calls give outside it, bit for bit (the sums have
a fixed order)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import sys; sys.path.insert(0, %r)
import numpy as np, torch
from paper_1305_1293_gb300 import pch
rng = np.random.default_rng(5)
n = %d
p = torch.from_numpy((rng.normal(size=pch.mlp_num_params()) * 0.15).astype(np.float32)).cuda()
x = torch.from_numpy(rng.uniform(-1, 1, (n, pch.mlp_num_features())).astype(np.float32)).cuda()
t = torch.from_numpy(rng.normal(size=n).astype(np.float32)).cuda()

def state():
    return [p.clone(), torch.zeros_like(p), torch.zeros_like(p), torch.zeros_like(p), torch.zeros(1, device='cuda'),
            torch.zeros(n, device='cuda')]

def step(s, stream):
    w, g, m, v, loss, y = s
    pch.mlp_forward(w, x, y, stream=stream)
    pch.mlp_backward(w, x, t, g, loss, stream=stream)
    pch.mlp_adam(w, g, m, v, 3, 1e-3, stream=stream)

a, b = state(), state()
torch.cuda.synchronize()
if %r:
    step(state(), torch.cuda.current_stream())
    torch.cuda.synchronize()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph):
    step(a, torch.cuda.current_stream())
for _ in range(3):
    graph.replay()
    step(b, torch.cuda.current_stream())
torch.cuda.synchronize()
assert a[4].item() > 0 and all(torch.equal(q, r) for q, r in zip(a, b))
print('captured')
"""


@pytest.mark.parametrize("n,warm", [(1000, False), (1000, True), (20000, False)])
def test_training_step_in_a_graph(n, warm):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    r = subprocess.run([sys.executable, "-c", CODE % (ROOT, n, warm)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "captured" in r.stdout, r.stdout + r.stderr

"""The library's device memory is given back when the last mesh is destroyed.

Memory is compared as the driver reports it for the device, in a process of its own; 32 MB
of slack for what the driver itself keeps."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def pch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1305_1293_gb300 import pch as p
    return p


RETURNED = """
import sys; sys.path.insert(0, %r)
import torch
from paper_1305_1293_gb300 import pch, meshgen as mg
free = lambda: torch.cuda.mem_get_info()[0]
m = mg.icosphere(3, 0.02, seed=7)
for turn in range(3):
    a, b = pch.Mesh(m.vertices, m.faces), pch.Mesh(m.vertices, m.faces)
    _, st = pch.solve(a, 3, stats=True)
    pch.solve(b, 3)
    held = free()
    a.close()
    b.close()
    got = free() - held
    assert got >= 2 * st['bytes_workspace'] - (32 << 20), (turn, got, st['bytes_workspace'])
print('returned')
"""


def test_all_memory_returned_with_the_last_mesh(pch):
    r = subprocess.run([sys.executable, "-c", RETURNED % ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "returned" in r.stdout, r.stdout + r.stderr


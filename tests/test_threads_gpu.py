"""Threads that create, solve, contour and destroy meshes at the same time, each on a stream
of its own: one thread's destruction or growing workspace must not disturb the graph that
another is building.  Parity bar 1e-9 against the oracle."""
import threading

import numpy as np
import pytest

from paper_1305_1293_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1305_1293_gb300 import pch as p
    return p


def test_threads_and_streams(pch, oracle_lib):
    import torch
    meshes = [mg.geodesic_sphere(9, 0.05, seed=81), mg.terrain(40, 30, seed=82), mg.torus(30, 14, seed=83),
              mg.geodesic_sphere(71, 0.02, seed=84)]
    refs = [oracle_lib.geodesic(m.vertices, m.faces, 11)[0] for m in meshes]
    failed = []

    def work(which):
        try:
            torch.cuda.set_device(0)
            stream = torch.cuda.Stream()
            m, ref = meshes[which % len(meshes)], refs[which % len(meshes)]
            for turn in range(6):
                h = pch.Mesh(m.vertices, m.faces)
                out = torch.empty(m.nv, dtype=torch.float64, device="cuda")
                for _ in range(2):
                    out.fill_(-1.0)
                    torch.cuda.current_stream().synchronize()
                    pch.solve(h, 11, out=out, stream=stream)
                    stream.synchronize()
                    got = out.cpu().numpy()
                    assert np.max(np.abs(got - ref) / np.maximum(ref, 1e-300)) < 1e-9, turn
                pch.iso_contours(h, got, [float(ref.max()) / 2])
                h.close()
        except BaseException as e:                      # reported by the main thread
            failed.append((which, repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed

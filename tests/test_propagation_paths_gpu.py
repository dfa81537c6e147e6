"""The two forms of the propagation kernel (a lane or a pair of lanes a window) around the
line where one takes over from the other: 16 windows a warp, set here through the number
of fresh windows that a warp takes at least.

Tolerance: the parity bar 1e-9 against the oracle; labels equal where unique."""
import numpy as np
import pytest

from paper_1305_1293_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu
TOL = 1e-9


@pytest.fixture(scope="module")
def pch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1305_1293_gb300 import pch as p
    return p


MESHES = {"sphere": lambda: mg.geodesic_sphere(11, 0.05, seed=61), "terrain": lambda: mg.terrain(33, 29, seed=62),
          "flat": lambda: mg.flat_patch(20, jitter=0.0, seed=63), "torus": lambda: mg.torus(40, 14, seed=64)}


@pytest.mark.parametrize("take", [1, 15, 16, 17, 32])
@pytest.mark.parametrize("name", list(MESHES))
def test_take_sizes(pch, oracle_lib, monkeypatch, name, take):
    m = MESHES[name]()
    monkeypatch.setenv("PCH_TAKE_MIN", str(take))
    mesh = pch.Mesh(m.vertices, m.faces)
    for s in (0, m.nv // 2):
        ref, _ = oracle_lib.geodesic(m.vertices, m.faces, s)
        for kw in ({}, {"k": 200, "hops": 3}, {"hops": 1}):
            got = pch.solve(mesh, s, **kw)
            assert np.array_equal(np.isfinite(got), np.isfinite(ref))
            assert float(np.max(np.abs(got - ref) / np.maximum(ref, 1e-300))) < TOL, (s, kw)
    mesh.close()


@pytest.mark.parametrize("take", [1, 32])
def test_batch_and_labels(pch, oracle_lib, monkeypatch, take):
    monkeypatch.setenv("PCH_TAKE_MIN", str(take))
    ms = [f() for f in MESHES.values()]
    meshes = [pch.Mesh(m.vertices, m.faces) for m in ms]
    for m, got in zip(ms, pch.solve_batch(meshes, [5] * len(ms))):
        ref, _ = oracle_lib.geodesic(m.vertices, m.faces, 5)
        assert float(np.max(np.abs(got - ref) / np.maximum(ref, 1e-300))) < TOL
    m, srcs = ms[0], [3, 400, 777]
    fields = np.array([oracle_lib.geodesic(m.vertices, m.faces, s)[0] for s in srcs])
    two = np.sort(fields, axis=0)[:2]
    unique = two[1] > two[0] * (1 + 1e-9)
    labels, dist = pch.voronoi(meshes[0], srcs)
    assert float(np.max(np.abs(dist - fields.min(0)) / np.maximum(fields.min(0), 1e-300))) < TOL
    assert np.array_equal(labels[unique], fields.argmin(0)[unique])
    for x in meshes:
        x.close()

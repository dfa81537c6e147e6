"""Where the propagation kernel's FP32 order tests can go wrong: units far from 1 (the FP32
images are scaled by the mesh's mean edge length), rays that pass exactly through
vertices (undecided in FP32), edges of very different lengths, and ends of windows at
vertices, whose events are made once.

Tolerance: the parity bar 1e-9 against the oracle; 1e-12 of the patch against the plane."""
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


def field(pch, v, f, s, **kw):
    mesh = pch.Mesh(v, f)
    try:
        return pch.solve(mesh, s, **kw)
    finally:
        mesh.close()


def max_rel(got, ref):
    assert np.array_equal(np.isfinite(got), np.isfinite(ref))
    return float(np.max(np.abs(got - ref) / np.maximum(ref, 1e-300)))


@pytest.mark.parametrize("exponent", [-100, -41, 0, 40, 100])
@pytest.mark.parametrize("hops", [1, 32])
def test_units(pch, oracle_lib, exponent, hops):
    m = mg.geodesic_sphere(9, 0.05, seed=41)
    ref, _ = oracle_lib.geodesic(m.vertices, m.faces, 17)
    got = field(pch, m.vertices * 2.0 ** exponent, m.faces, 17, hops=hops)
    assert max_rel(got * 2.0 ** -exponent, ref) < TOL


@pytest.mark.parametrize("n,source", [(16, 0), (24, 12 * 25 + 12), (33, 34 * 16 + 5)])
def test_rays_through_vertices(pch, n, source):
    m = mg.flat_patch(n, jitter=0.0, seed=5)
    got = field(pch, m.vertices, m.faces, source)
    assert np.max(np.abs(got - np.linalg.norm(m.vertices - m.vertices[source], axis=1))) < 1e-12


@pytest.mark.parametrize("stretch", [1.0, 40.0])
def test_uneven_edges(pch, oracle_lib, stretch):
    """A height field whose columns grow geometrically along x (edges from 1 to `stretch`)."""
    m = mg.terrain(22, 18, seed=43)
    v = m.vertices.copy()
    q = stretch ** (1.0 / 22)
    v[:, 0] = np.cumsum(np.concatenate([[0.0], q ** np.arange(22)]))[v[:, 0].astype(int)]
    for s in (0, mg.terrain_center(22, 18)):
        ref, _ = oracle_lib.geodesic(v, m.faces, s)
        assert max_rel(field(pch, v, m.faces, s), ref) < TOL


@pytest.mark.parametrize("n_inst", [1, 3])
def test_instances_of_different_units(pch, oracle_lib, n_inst):
    """One launch sequence over meshes of different scales: each has its own FP32 scale."""
    ms = [mg.icosphere(2, 0.05, seed=50 + i) for i in range(n_inst)]
    scale = [1.0, 2.0 ** 60, 2.0 ** -60][:n_inst]
    meshes = [pch.Mesh(m.vertices * c, m.faces) for m, c in zip(ms, scale)]
    got = pch.solve_batch(meshes, [3] * n_inst)
    for m, c, g in zip(ms, scale, got):
        ref, _ = oracle_lib.geodesic(m.vertices, m.faces, 3)
        assert max_rel(g / c, ref) < TOL
    for m in meshes:
        m.close()

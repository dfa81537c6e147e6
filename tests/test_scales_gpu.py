"""Meshes in units far from 1: a field scales with its mesh, also where lengths, or products
of two of them, are beyond single precision (2^+-128).

Against the oracle on the mesh as generated, times the scale (a power of two: the scaled mesh
is the same one, exactly); tolerance the parity bar 1e-9."""
import numpy as np
import pytest

from paper_1305_1293_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu
TOL = 1e-9

MESHES = {"sphere": lambda: mg.geodesic_sphere(11, 0.05, seed=61), "terrain": lambda: mg.terrain(33, 29, seed=62),
          "flat": lambda: mg.flat_patch(20, jitter=0.2, seed=63), "torus": lambda: mg.torus(40, 14, seed=64)}


@pytest.fixture(scope="module")
def pch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1305_1293_gb300 import pch as p
    return p


@pytest.mark.parametrize("exponent", [-400, -130, 130, 400])
@pytest.mark.parametrize("name", list(MESHES))
def test_field_scales_with_the_mesh(pch, oracle_lib, name, exponent):
    m = MESHES[name]()
    mesh = pch.Mesh(np.ldexp(m.vertices, exponent), m.faces)
    for s in (0, m.nv // 2, m.nv - 1):
        ref, _ = oracle_lib.geodesic(m.vertices, m.faces, s)
        for kw in ({}, {"k": 200, "hops": 3}):
            got = np.ldexp(pch.solve(mesh, s, **kw), -exponent)
            assert np.isfinite(got).all(), (s, kw)
            assert float(np.max(np.abs(got - ref) / np.maximum(ref, 1e-300))) < TOL, (s, kw)
    mesh.close()

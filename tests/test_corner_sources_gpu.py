"""Face-point sources on a corner of their face and within a few tolerances (2^-40 of the edge)
of it, where the windows through the face's edges are edge-on: the field is that of the
corner's vertex, up to the point's distance from it; every vertex is reached.  Also beside a
vertex source at the same corner, in either order, and in labels and paths.

Tolerance: the parity bar 1e-9 against the oracle's field of the vertex, plus twice the
offset of the point (triangle inequality: the two fields differ by at most the offset)."""
import ctypes

import numpy as np
import pytest

from paper_1305_1293_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu
TOL = 1e-9

MESHES = {"sphere": lambda: mg.geodesic_sphere(11, 0.05, seed=61), "terrain": lambda: mg.terrain(33, 29, seed=62),
          "ico": lambda: mg.icosphere(3, 0.1, seed=5)}


@pytest.fixture(scope="module")
def pch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1305_1293_gb300 import pch as p
    return p


def weights(corner, eps):
    b = np.full(3, eps / 2)
    b[corner] = 1.0 - eps
    return b


def check(got, ref, offset, what):
    assert np.isfinite(got).all(), (what, int((~np.isfinite(got)).sum()))
    assert np.all(np.abs(got - ref) <= TOL * ref + offset), (what, float(np.max(np.abs(got - ref))))


@pytest.mark.parametrize("name", list(MESHES))
def test_near_a_corner(pch, oracle_lib, name):
    m = MESHES[name]()
    longest = max(np.linalg.norm(m.vertices[m.faces[:, i]] - m.vertices[m.faces[:, i - 1]], axis=1).max() for i in range(3))
    mesh = pch.Mesh(m.vertices, m.faces)
    for f in (0, m.nf // 2, m.nf - 1):
        for c in range(3):
            ref, _ = oracle_lib.geodesic(m.vertices, m.faces, int(m.faces[f, c]))
            for eps in (0.0, 1e-16, 1e-13, 1e-12, 3e-12):
                got = pch.solve(mesh, face=f, bary=weights(c, eps))
                check(got, ref, 2 * eps * longest, (f, c, eps))
    mesh.close()


@pytest.mark.parametrize("order", [0, 1])
def test_beside_a_vertex_source(pch, oracle_lib, order):
    m = MESHES["terrain"]()
    mesh = pch.Mesh(m.vertices, m.faces)
    for v in (0, m.nv // 2, m.nv - 1):
        ref, _ = oracle_lib.geodesic(m.vertices, m.faces, v)
        faces, corners = np.nonzero(m.faces == v)
        points = [pch.make_source(face=int(f), bary=np.eye(3)[c]) for f, c in zip(faces, corners)] * 40
        srcs = [pch.make_source(vertex=v)] + points if order == 0 else points + [pch.make_source(vertex=v)]
        arr, out = (pch.Source * len(srcs))(*srcs), np.empty(m.nv)
        assert pch.lib.pch_solve_multi(mesh.handle, arr, len(srcs), None, out.ctypes.data, None) == pch.PCH_OK
        check(out, ref, 0.0, (v, order))
    mesh.close()


def test_labels_and_paths(pch, oracle_lib):
    import pathcheck
    m = MESHES["sphere"]()
    mesh = pch.Mesh(m.vertices, m.faces)
    f, g = 17, m.nf - 40
    ends = [int(m.faces[f, 1]), int(m.faces[g, 2])]
    fields = np.array([oracle_lib.geodesic(m.vertices, m.faces, v)[0] for v in ends])
    labels, dist = pch.voronoi(mesh, None, faces=[f, g], barys=[np.eye(3)[1], np.eye(3)[2]])
    check(dist, fields.min(0), 0.0, "labels")
    unique = np.abs(fields[0] - fields[1]) > 1e-9 * fields.min(0)
    assert np.array_equal(labels[unique], fields.argmin(0)[unique])
    targets = np.arange(0, m.nv, 53)
    d, paths = pch.trace_paths(mesh, None, targets, face=f, bary=np.eye(3)[1])
    check(d, fields[0], 0.0, "paths")
    for t, p in zip(targets, paths):
        assert p is not None and p[1][0] == t
        x = pathcheck.path_xyz(m.vertices, m.faces, p)
        assert np.allclose(x[-1], m.vertices[ends[0]], atol=1e-12)
        length = np.linalg.norm(np.diff(x, axis=0), axis=1).sum()
        assert abs(length - fields[0][t]) <= 1e-9 * max(fields[0][t], 1e-300)
    mesh.close()

"""Meshes of 2^19 faces and more are kept in Morton order inside the library; face and
half-edge ids at the boundary stay the caller's.  One mesh, given with its faces as
generated and shuffled: every answer refers to the caller's own numbering.

Tolerances: fields of the two orders differ by rounding only (1e-12 relative); paths must
pass the geometric checks; contour segments equal the linear interpolation exactly."""
import numpy as np
import pytest

import pathcheck
from paper_1305_1293_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu
OPTS = {"k": 1572864, "hops": 32}


@pytest.fixture(scope="module")
def case():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1305_1293_gb300 import pch
    m = mg.geodesic_sphere(163, 0.02, seed=77)
    assert m.nf >= 1 << 19
    order = np.random.default_rng(7).permutation(m.nf)
    shuffled = np.ascontiguousarray(m.faces[order])
    a, b = pch.Mesh(m.vertices, m.faces), pch.Mesh(m.vertices, shuffled)
    yield pch, m, shuffled, order, a, b
    a.close()
    b.close()


def test_face_point_source(case):
    pch, m, shuffled, order, a, b = case
    assert a.info() == b.info()
    for fb in (0, 131071, m.nf - 1):
        da = pch.solve(a, face=int(order[fb]), bary=(0.2, 0.3, 0.5), **OPTS)
        db = pch.solve(b, face=fb, bary=(0.2, 0.3, 0.5), **OPTS)
        p = (0.2, 0.3, 0.5) @ m.vertices[shuffled[fb]]
        corner = np.linalg.norm(m.vertices[shuffled[fb]] - p, axis=1)
        assert np.max(np.abs(db[shuffled[fb]] - corner)) < 1e-12
        assert np.max(np.abs(da - db) / np.maximum(da, 1e-300)) < 1e-12


def test_paths(case):
    pch, m, shuffled, order, a, b = case
    targets = [1, 77777, m.nv - 1]
    dist, paths = pch.trace_paths(b, [12345], targets, max_points=8192, **OPTS)
    for t, path in zip(targets, paths):
        xyz = pathcheck.path_xyz(m.vertices, shuffled, path)
        length = np.linalg.norm(np.diff(xyz, axis=0), axis=1).sum()
        assert int(path[1][0]) == t and int(path[1][-1]) == 12345
        assert abs(length - dist[t]) <= 1e-9 * dist[t]


def test_contours(case):
    pch, m, shuffled, order, a, b = case
    field = np.linalg.norm(m.vertices - m.vertices[5], axis=1)
    levels = [0.5, 1.25]
    got = pch.iso_contours(b, field, levels)
    d = field[shuffled]
    want = []
    for l, lev in enumerate(levels):
        inside = d < lev
        for f in np.nonzero(inside.any(1) & ~inside.all(1))[0]:
            k = [i for i in range(3) if inside[f, i] and not inside[f, (i + 1) % 3]]
            k += [i for i in range(3) if not inside[f, i] and inside[f, (i + 1) % 3]]
            want.append((f, l, 3 * f + k[0], 3 * f + k[1],
                         *((lev - d[f, i]) / (d[f, (i + 1) % 3] - d[f, i]) for i in k)))
    want.sort(key=lambda r: r[:2])
    assert len(want) == len(got)
    assert np.array_equal(got["face"], [r[0] for r in want]) and np.array_equal(got["level"], [r[1] for r in want])
    assert np.array_equal(got["half_edge"], [r[2:4] for r in want])
    assert np.array_equal(got["t"], [r[4:] for r in want])

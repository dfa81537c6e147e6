"""Contours where the order tests on integer images, the tile lists and the two ways of
allocating the segments can go wrong: signed zeros, negative and infinite distances, NaN,
more segments in a tile of faces than its list holds, more possible segments than are
allocated at once.  Exact equality with the interpolation written out in numpy."""
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


def expected(faces, field, levels):
    d = field[faces]
    rows = []
    with np.errstate(invalid="ignore", over="ignore"):
        usable = ~np.isnan(d).any(1) & ~(d == np.inf).any(1)
        for l, lev in enumerate(levels):
            inside = d < lev
            for f in np.nonzero(usable & inside.any(1) & ~inside.all(1))[0]:
                k = [i for i in range(3) if inside[f, i] and not inside[f, (i + 1) % 3]]
                k += [i for i in range(3) if not inside[f, i] and inside[f, (i + 1) % 3]]
                t = [(lev - d[f, i]) / (d[f, (i + 1) % 3] - d[f, i]) for i in k]
                rows.append((f, l, 3 * f + k[0], 3 * f + k[1], t[0], t[1]))
    return sorted(rows, key=lambda r: r[:2])


def check(got, rows):
    assert len(got) == len(rows)
    assert np.array_equal(got["face"], [r[0] for r in rows]) and np.array_equal(got["level"], [r[1] for r in rows])
    assert np.array_equal(got["half_edge"], np.array([r[2:4] for r in rows]).reshape(-1, 2))
    assert np.array_equal(got["t"], np.array([r[4:] for r in rows]).reshape(-1, 2), equal_nan=True)


def test_special_values(pch):
    m = mg.geodesic_sphere(6, 0.02, seed=3)
    rng = np.random.default_rng(4)
    field = np.round(rng.normal(size=m.nv), 1)
    for value in (0.0, -0.0, np.inf, -np.inf, np.nan, 1e308, -1e308, 5e-324, -5e-324):
        field[rng.integers(m.nv, size=6)] = value
    levels = [0.0, -0.0, 0.1, -0.3, 1e308, 5e-324, -5e-324, -1e308]
    mesh = pch.Mesh(m.vertices, m.faces)
    with np.errstate(all="ignore"):
        check(pch.iso_contours(mesh, field, levels), expected(m.faces, field, levels))
    mesh.close()


@pytest.mark.parametrize("n_levels,capacity", [(40, None), (40, 1000), (700, 1 << 22)])
def test_many_segments(pch, n_levels, capacity):
    """Every face crosses most levels (a tile of 256 faces holds more than 2,048); 4 Mi segments
    of capacity are more than are allocated before the count is known."""
    m = mg.geodesic_sphere(9, 0.02, seed=5)
    field = np.random.default_rng(6).uniform(0.0, 1.0, m.nv)
    levels = np.linspace(0.02, 0.98, n_levels)
    mesh = pch.Mesh(m.vertices, m.faces)
    rows = expected(m.faces, field, levels)
    check(pch.iso_contours(mesh, field, levels, capacity=capacity), rows[:capacity])
    mesh.close()

"""Selection at distances of 2^17 mean edge lengths and more, where a step of the keys' FP32
images is wider than the first bin of the selection's histogram: the threshold still reaches
the nearest window, so every iteration makes progress.

The mesh is a flat strip of unit squares beside a separate fine grid that makes the mean edge
length small against the strip.  The strip is convex and flat: distances are straight lines,
relative tolerance the parity bar 1e-9.  The iteration limit turns a stall into a timeout: two
iterations select or drop at least one window, and these strips make some 10^5 of them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
MOST = 2 * 100000 + 50000


@pytest.fixture(scope="module")
def pch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1305_1293_gb300 import pch as p
    return p


def grid(nx, ny, step, origin):
    """nx x ny squares of side `step` in the plane, two triangles each."""
    y, x = np.mgrid[0:ny + 1, 0:nx + 1]
    v = np.stack([origin[0] + step * x.ravel(), origin[1] + step * y.ravel(), np.zeros(x.size)], 1)
    a = (np.arange(ny)[:, None] * (nx + 1) + np.arange(nx)[None, :]).ravel()
    f = np.concatenate([np.stack([a, a + 1, a + nx + 2], 1), np.stack([a, a + nx + 2, a + nx + 1], 1)])
    return v, f


def strip_and_grid(length, width, fine):
    v, f = grid(length, width, 1.0, (0.0, 0.0))
    v2, f2 = grid(fine, fine, 1e-6, (0.0, -5.0))
    return np.concatenate([v, v2]), np.concatenate([f, f2 + len(v)]).astype(np.int32), len(v)


@pytest.mark.parametrize("width,fine,k", [(2, 1024, 1), (2, 1024, 2), (3, 700, 1), (3, 700, 4)])
def test_far_windows_are_selected(pch, width, fine, k):
    v, f, n = strip_and_grid(200, width, fine)
    p = v[f]
    mean_edge = np.mean([np.linalg.norm(p[:, i] - p[:, (i + 1) % 3], axis=1).mean() for i in range(3)])
    assert 200.0 / mean_edge > 2 ** 17
    mesh = pch.Mesh(v, f)
    d = pch.solve(mesh, 0, k=k, max_iters=MOST)
    want = np.linalg.norm(v[:n] - v[0], axis=1)
    assert np.all(np.abs(d[:n] - want) <= 1e-9 * np.maximum(want, 1e-300))
    assert np.all(np.isinf(d[n:]))
    mesh.close()


def test_far_windows_in_a_batch(pch):
    """Instances of their own thresholds: the far strip beside a plain grid."""
    v, f, n = strip_and_grid(200, 2, 1024)
    v2, f2 = grid(9, 7, 1.0, (0.0, 0.0))
    f2 = f2.astype(np.int32)
    meshes = [pch.Mesh(v, f), pch.Mesh(v2, f2)]
    far, near = pch.solve_batch(meshes, [0, 3], k=1, max_iters=MOST)
    want = np.linalg.norm(v[:n] - v[0], axis=1)
    assert np.all(np.abs(far[:n] - want) <= 1e-9 * np.maximum(want, 1e-300))
    want = np.linalg.norm(v2 - v2[3], axis=1)
    assert np.all(np.abs(near - want) <= 1e-9 * np.maximum(want, 1e-300))
    for m in meshes:
        m.close()

"""Fields on either side of the size at which children's records are no longer prefetched
(512 MB of half-edge records, 96 bytes each: 1,864,135 faces): a jittered grid in the plane, whose
distances are Euclidean.

Tolerance: a vertex is reached through at most about 2,000 unfolded edges, each of which
rounds the pseudo-source's position a few times (2^-53 of the edge or of the distance): below
2,000 * 4 * 1.2e-16 = 1e-12 of the distance, and ten times that is allowed.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,control", [(966, "plain"), (967, "plain"), (967, "learned")])
def test_planar_distances(n, control):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1305_1293_gb300 import pch

    rng = np.random.default_rng(n)
    y, x = np.meshgrid(np.arange(n, dtype=np.float64), np.arange(n, dtype=np.float64), indexing="ij")
    inner = (x > 0) & (x < n - 1) & (y > 0) & (y < n - 1)
    x = x + np.where(inner, rng.uniform(-0.2, 0.2, x.shape), 0.0)
    y = y + np.where(inner, rng.uniform(-0.2, 0.2, y.shape), 0.0)
    v = np.stack([x.ravel(), y.ravel(), np.zeros(n * n)], axis=1)
    a = (np.arange(n - 1)[:, None] * n + np.arange(n - 1)[None, :]).ravel()
    f = np.concatenate([np.stack([a, a + 1, a + n + 1], axis=1), np.stack([a, a + n + 1, a + n], axis=1)]).astype(np.int32)
    assert (len(f) * 3 * 96 < 1 << 29) == (n == 966)
    source = (n // 3) * n + n // 2
    mesh = pch.Mesh(v, f)
    d = pch.solve(mesh, source, k=1 << 19, control=pch.CONTROL_LEARNED if control == "learned" else pch.CONTROL_PLAIN)
    mesh.close()
    want = np.linalg.norm(v - v[source], axis=1)
    assert np.all(np.abs(d - want) <= 1e-11 * want)

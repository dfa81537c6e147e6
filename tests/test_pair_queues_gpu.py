"""Pairs of lanes a window with full queues: lists of 9 to 16 windows for each of few resident
warps, where more windows continue than a pair queue holds (16), the buffer of 16 children
fills several times in a round, and chains stop at the arena's limit; and the same inputs
with whole warps (17 windows a warp at least).

Tolerance: the parity bar 1e-9 against the oracle or straight lines, and between the two
forms (a child of which half is lost or left over is wrong in the leading digits)."""
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


def rel(a, b):
    return float(np.max(np.abs(a - b) / np.maximum(b, 1e-300)))


@pytest.mark.parametrize("per_warp", [9, 13, 16])
def test_full_pair_queues(pch, oracle_lib, monkeypatch, per_warp):
    import torch
    m = mg.geodesic_sphere(30, 0.05, seed=71)                     # 18,000 faces
    ref, _ = oracle_lib.geodesic(m.vertices, m.faces, 7)
    warps = torch.cuda.get_device_properties(0).multi_processor_count
    monkeypatch.setenv("PCH_PROP_BLOCKS_PER_SM", "1")             # one warp an SM
    mesh = pch.Mesh(m.vertices, m.faces)
    for hops in (0, 3):
        got, st = pch.solve(mesh, 7, stats=True, k=per_warp * warps, block=32, hops=hops)
        assert rel(got, ref) < TOL
        assert st["windows_chained"] > st["iterations"] * warps   # chains ran in most warps' rounds
        assert st["children_computed"] > 16 * st["iterations"]
    mesh.close()


@pytest.mark.parametrize("name", ["sphere", "terrain", "flat"])
def test_pairs_and_whole_warps_agree(pch, monkeypatch, name):
    """100,000 faces and more: the form changes nothing but the order of events."""
    m = {"sphere": lambda: mg.geodesic_sphere(71, 0.02, seed=72), "terrain": lambda: mg.terrain(260, 230, seed=73),
         "flat": lambda: mg.flat_patch(240, jitter=0.0, seed=74)}[name]()
    mesh = pch.Mesh(m.vertices, m.faces)
    fields = []
    for take in ("1", "17"):
        monkeypatch.setenv("PCH_TAKE_MIN", take)
        fields.append([pch.solve(mesh, m.nv // 3, k=k) for k in (0, 3000)])
    for a, b in zip(*fields):
        assert np.isfinite(a).all() and rel(a, b) < TOL
    if name == "flat":
        line = np.linalg.norm(m.vertices - m.vertices[m.nv // 3], axis=1)
        assert rel(fields[0][0], line) < TOL
    mesh.close()

"""More contour segments than 2^31 - 1: refused, nothing of the caller's written, also when a
single tile of 256 faces holds more than 32-bit offsets do and room for a few segments was
asked for (the segments of a small room are written before the total is known)."""
import ctypes

import numpy as np
import pytest

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


def test_tile_beyond_32_bits(pch):
    """A strip with the field 0 along one side and 1 along the other: every face crosses every
    level, 256 faces a block of the two kernels (8 blocks an SM), 2^31 + 256 segments a tile."""
    import torch
    faces = 256 * 8 * torch.cuda.get_device_properties(0).multi_processor_count
    n = faces // 2
    x = np.arange(n + 1.0)
    v = np.concatenate([np.stack([x, 0 * x, 0 * x], 1), np.stack([x, 0 * x + 1, 0 * x], 1)])
    a = np.arange(n)
    f = np.concatenate([np.stack([a, a + 1, a + n + 2], 1), np.stack([a, a + n + 2, a + n + 1], 1)]).astype(np.int32)
    field = np.concatenate([np.zeros(n + 1), np.ones(n + 1)])
    levels = np.linspace(0.25, 0.75, 2 ** 31 // 256 + 1)
    mesh = pch.Mesh(v, f)
    out = np.full(64, -7, dtype=np.int64).view(pch.CONTOUR_DTYPE)
    total = ctypes.c_int64(-3)
    st = pch.lib.pch_iso_contours(mesh.handle, field.ctypes.data, 0, levels.ctypes.data, levels.size, out.ctypes.data,
                                  len(out), ctypes.byref(total))
    assert st == pch.PCH_ERR_CAPACITY and "exceed" in pch.lib.pch_last_error().decode()
    assert np.all(out.view(np.int64) == -7) and total.value == -3
    got = pch.iso_contours(mesh, field, levels[:3])          # the mesh is as usable as before
    assert len(got) == 3 * faces and np.array_equal(got["face"], np.repeat(np.arange(faces), 3))
    mesh.close()

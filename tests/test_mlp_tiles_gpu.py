"""The controller's tiled forward and backward kernels at the edges of their tiles (64
samples) and grids, against the FP64 network.

Tolerance: a gradient entry is a sum over n samples of FP32 products of at most 64 x 3
layers' terms; relative to the largest entry its error stays below 4e-6 times a growth of
sqrt(n) < 2^8 rounding steps of 6e-8, so 1e-4 of the largest entry, as the controller's
other GPU tests use."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1305_1293_gb300 import pch
    return torch, pch


@pytest.mark.parametrize("n", [1, 63, 64, 65, 64 * 152, 64 * 152 + 1, 20011])
def test_forward_backward(env, n):
    torch, pch = env
    from oracle import mlp_oracle as mo
    rng = np.random.default_rng(n)
    p = (rng.normal(size=pch.mlp_num_params()) * 0.15).astype(np.float32)
    x = rng.uniform(-1, 1, (n, pch.mlp_num_features())).astype(np.float32)
    t = rng.normal(size=n).astype(np.float32)
    pd, xd, td = (torch.from_numpy(a).cuda() for a in (p, x, t))
    y = torch.full((n,), float("nan"), device="cuda")
    g = torch.full_like(pd, float("nan"))
    loss = torch.full((1,), float("nan"), device="cuda")
    pch.mlp_forward(pd, xd, y)
    pch.mlp_backward(pd, xd, td, g, loss)
    torch.cuda.synchronize()
    p64, x64, t64 = (a.astype(np.float64) for a in (p, x, t))
    y_ref, _ = mo.forward(p64, x64)
    g_ref = mo.grad(p64, x64, t64)
    assert np.max(np.abs(y.cpu().numpy() - y_ref)) <= 1e-4 * max(1.0, np.abs(y_ref).max())
    assert np.max(np.abs(g.cpu().numpy() - g_ref)) <= 1e-4 * max(1e-3, np.abs(g_ref).max())
    want = mo.loss(p64, x64, t64)
    assert abs(loss.item() - want) <= 1e-4 * max(1.0, want)
    g2 = torch.empty_like(g)
    pch.mlp_backward(pd, xd, td, g2, loss)
    assert torch.equal(g, g2)                # a fixed order of every sum

"""Rays and Gaussians at the edges of the 32-bit arithmetic: every traversal blends the same hits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2601_20429_gb300 import render as R
from paper_2601_20429_gb300 import scenes


@pytest.mark.parametrize("traversal", ["restart", "checkpoint", "single"])
@pytest.mark.parametrize("k", [1, 2, 8])
def test_depths_of_both_zeros(traversal, k):
    """Rays that start at the mean of several Gaussians: their depths are 0 of either sign, one depth. Every
    ray blends all 24 whatever k (the products of a ray are taken in the order of the leaf slots)."""
    n = 24
    rng = np.random.default_rng(4)
    q = rng.standard_normal((n, 4))
    mean = np.array([0.25, -0.5, 0.125], np.float32)
    g = scenes.GaussianParams(np.tile(mean, (n, 1)), rng.uniform(-1.5, -1.0, (n, 3)).astype(np.float32),
                              (q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32),
                              np.full(n, np.log(0.1 / 0.9), np.float32), rng.normal(0, 0.3, (n, 1, 3)).astype(np.float32), 0)
    m = 64
    d = rng.standard_normal((m, 3))
    rays = tuple(torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()
                 for x in (np.tile(mean, (m, 1)), d / np.linalg.norm(d, axis=1, keepdims=True), np.full(m, -1.0), np.full(m, 9.0)))
    sc = R.Scene.from_params(g)
    ref = R.render(sc, None, rays=rays, k=32, traversal="restart", want_n_blended=True)
    assert ref["n_blended"].tolist() == [n] * m
    a = R.render(sc, None, rays=rays, k=k, traversal=traversal)["rgbT"]
    b = R.render(sc, None, rays=rays, k=k, traversal=traversal, want_n_blended=True)
    torch.cuda.synchronize()
    assert b["n_blended"].tolist() == [n] * m
    np.testing.assert_array_equal(a[:, 3].cpu().numpy(), ref["rgbT"][:, 3].cpu().numpy())
    sc.close()

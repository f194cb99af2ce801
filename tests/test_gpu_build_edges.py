"""The build's one-launch sort passes and clustering rounds, its gathers and its valid count at the edges
of their tiles, bit for bit against numpy's stable sort and the oracle's clustering."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import oracle as O
from paper_2601_20429_gb300 import native as N
from paper_2601_20429_gb300 import render as R
from paper_2601_20429_gb300 import scenes


@pytest.mark.parametrize("n", [2, 31, 1023, 1024, 1025, 2049, 12_345, 262_145])
@pytest.mark.parametrize("bits,few", [(64, False), (64, True), (13, True), (8, False)])
def test_sort_edges(n, bits, few):
    rng = np.random.default_rng(n + bits)
    keys = rng.integers(0, 40 if few else 1 << 63, n, dtype=np.uint64) << np.uint64(0 if bits < 64 else (3 if few else 0))
    k, v = torch.from_numpy(keys.view(np.int64)).cuda(), torch.arange(n, dtype=torch.int32, device="cuda")
    N.grtx_sort_pairs(k, v, bits)
    torch.cuda.synchronize()
    part = keys & np.uint64((1 << bits) - 1) if bits < 64 else keys
    order = np.argsort(part, kind="stable")
    np.testing.assert_array_equal(v.cpu().numpy(), order)
    np.testing.assert_array_equal(k.cpu().numpy().view(np.uint64), keys[order])


@pytest.mark.parametrize("dups", [False, True])
@pytest.mark.parametrize("n", [15, 16, 17, 33, 255, 256, 257, 1024, 2047, 2048, 2049, 2305, 4097, 33_000])
def test_clustering_edges(n, dups):
    rng = np.random.default_rng(n)
    lo = rng.integers(0, 12, (n, 3)).astype(np.float32) if dups else rng.uniform(-1, 1, (n, 3)).astype(np.float32)
    boxes = np.concatenate([lo, lo + (1.0 if dups else rng.uniform(0.001, 0.1, (n, 3)).astype(np.float32))], 1).astype(np.float32)
    boxes = np.ascontiguousarray(boxes[np.argsort(O.morton_sized64(boxes, O.centroid_bounds(boxes)), kind="stable")])
    left, right = (torch.empty(n - 1, dtype=torch.int32, device="cuda") for _ in range(2))
    parent = torch.empty(2 * n - 1, dtype=torch.int32, device="cuda")
    it = N.grtx_ploc_tree(torch.from_numpy(boxes).cuda(), left, right, parent)
    torch.cuda.synchronize()
    ol, orr, oit = O.ploc(boxes, radius=16)
    assert it == oit
    np.testing.assert_array_equal(left.cpu().numpy().view(np.uint32), ol)
    np.testing.assert_array_equal(right.cpu().numpy().view(np.uint32), orr)


@pytest.mark.parametrize("n,valid", [(1, 1), (2, 0), (33, 32), (33, 1), (1000, 999), (1025, 1024), (5000, 31)])
def test_valid_count(n, valid):
    g = scenes.tiny_scene(seed=n, n=n)
    g.logits[:] = 1.0
    g.logits[np.random.default_rng(n).permutation(n)[: n - valid]] = -9.0
    sc = R.Scene.from_params(g)
    info = sc.info()
    assert info["n_valid"] == valid
    if valid:
        assert sorted(sc.export()[1].cpu().numpy().tolist()) == np.nonzero(g.logits > 0)[0].tolist()
    sc.close()


@pytest.mark.parametrize("deg", [0, 1, 2, 3])
def test_appearance_rows_at_any_alignment(deg):
    """The colours of a scene do not depend on where the caller's SH array starts, at a build or a refit."""
    rng = np.random.default_rng(deg)
    g = scenes.tiny_scene(seed=3, n=777)
    g.sh = rng.normal(0, 0.3, (g.n, (deg + 1) ** 2, 3)).astype(np.float32)
    g.sh_degree = deg
    t = [torch.from_numpy(a).cuda() for a in g.arrays()]
    flat = torch.empty(t[4].numel() + 1, device="cuda")
    odd = flat[1:].view(t[4].shape)
    odd.copy_(t[4])
    assert odd.data_ptr() % 16 == 4
    cam = scenes.pinhole_camera(64, 64, (0.0, 0.0, -3.0))
    a, b = R.Scene(*t, deg), R.Scene(*t[:4], odd, deg)
    ref = R.render(a, cam, k=8)["rgbT"].clone()
    assert torch.equal(ref, R.render(b, cam, k=8)["rgbT"])
    b.update(*t[:4], odd)
    assert torch.equal(ref, R.render(b, cam, k=8)["rgbT"])
    a.close()
    b.close()

"""Rays and Gaussians at the edges of the 32-bit arithmetic: every traversal blends the same hits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2601_20429_gb300 import native as N
from paper_2601_20429_gb300 import render as R
from paper_2601_20429_gb300 import scenes


def _discs(cam, o, n, ratio, size, at, aside, offset, seed):
    """Faint discs of aspect 1:ratio whose planes hold one of the camera's rays: their means lie at depth `at`
    on it (an array), `aside` in the plane beside it and `offset` half-thicknesses off it."""
    rng = np.random.default_rng(seed)
    W, H, th = cam["width"], cam["height"], np.tan(0.5 * cam["fov"])
    p = rng.integers(0, W * H, n)
    u, v = (2 * (p % W + 0.5) / W - 1) * th * W / H, (1 - 2 * (p // W + 0.5) / H) * th
    d = np.asarray(cam["forward"]) + u[:, None] * np.asarray(cam["right"]) + v[:, None] * np.asarray(cam["up"])
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    nrm = np.cross(d, rng.standard_normal((n, 3)))
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    e2 = np.cross(nrm, d)
    M = np.stack([d, e2, nrm], 2)                       # columns: the disc's axes (a rotation)
    w = np.sqrt(np.maximum(1 + np.trace(M, axis1=1, axis2=2), 1e-12)) / 2
    q = np.stack([w, (M[:, 2, 1] - M[:, 1, 2]) / (4 * w), (M[:, 0, 2] - M[:, 2, 0]) / (4 * w),
                  (M[:, 1, 0] - M[:, 0, 1]) / (4 * w)], 1)
    opacity = 0.015
    s = np.tile([size, size, size / ratio], (n, 1)) / np.sqrt(2 * np.log(opacity / 0.01))
    mean = np.asarray(o) + at[:, None] * d + aside[:, None] * e2 + (offset * size / ratio)[:, None] * nrm
    return scenes.GaussianParams(mean.astype(np.float32), np.log(s).astype(np.float32), q.astype(np.float32),
                                 np.full(n, np.log(opacity / (1 - opacity)), np.float32),
                                 rng.normal(0, 0.3, (n, 1, 3)).astype(np.float32), 0)


def _equal_transmittance(g, cam, **opts):
    sc = R.Scene.from_params(g)
    a = R.render(sc, cam, T_min=0.0, **opts)["rgbT"]
    b = R.render(sc, cam, T_min=0.0, traversal="restart", **opts)["rgbT"]
    torch.cuda.synchronize()
    np.testing.assert_array_equal(a[:, 3].cpu().numpy(), b[:, 3].cpu().numpy())
    sc.close()


@pytest.mark.parametrize("seed", range(4))
@pytest.mark.parametrize("ratio", [1e2, 1e3, 1e4, 1e5])
def test_camera_inside_thin_discs(ratio, seed):
    """A wide tile whose camera lies in the discs' planes, within the discs: the walk filters no hit out (the same
    transmittances, bit for bit, as rounds that test every leaf that a ray's boxes reach)."""
    o = (0.1, 0.2, -0.3)
    cam = scenes.pinhole_camera(8, 4, o, (0.4, 0.1, 1.0), 100.0)
    rng = np.random.default_rng(seed + 50)
    n = 400
    g = _discs(cam, o, n, ratio, 3.0, 10 ** rng.uniform(-3, -0.5, n), 10 ** rng.uniform(-4, -1, n), rng.uniform(-0.99, 0.99, n),
               seed)
    _equal_transmittance(g, cam, k=16)


@pytest.mark.parametrize("seed", range(3))
@pytest.mark.parametrize("ratio", [1e4, 1e6, 3e6])
def test_thin_discs_behind_t_near(ratio, seed):
    """Depths just behind t_near (within 2 %) of discs seen along their planes: none is taken for one before it."""
    o = (0.1, 0.2, -0.3)
    cam = scenes.pinhole_camera(8, 4, o, (0.4, 0.1, 1.0), 60.0, t_near=1.0)
    rng = np.random.default_rng(seed + 70)
    n = 1500
    g = _discs(cam, o, n, ratio, 0.3, 1.0 + rng.uniform(0.0, 0.02, n), rng.uniform(-0.1, 0.1, n), np.zeros(n), seed)
    _equal_transmittance(g, cam, k=16)


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


@pytest.mark.parametrize("opts", [dict(ckpt_capacity=2, evict_capacity=1), dict(ckpt_capacity=1, evict_capacity=8)])
@pytest.mark.parametrize("form,width", [("sphere", 2), ("sphere", 4), ("ico20", 2), ("proxy20", 2)])
def test_a_ray_falls_back_once(form, width, opts):
    """A ray whose lists are too small for a packet's round leaves them for restarted rounds at once: one fallback
    a ray, and the image of restarted rounds. (500 faint overlapping Gaussians, dozens of hits a ray.)"""
    n = 500
    rng = np.random.default_rng(2)
    q = rng.standard_normal((n, 4))
    g = scenes.GaussianParams(rng.uniform(-1, 1, (n, 3)).astype(np.float32), np.log(rng.uniform(0.1, 0.4, (n, 3))).astype(np.float32),
                              (q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32),
                              np.full(n, np.log(0.05 / 0.95), np.float32), rng.normal(0, 0.3, (n, 1, 3)).astype(np.float32), 0)
    sc = R.Scene.from_params(g, form=form, bvh_width=width)
    cam = scenes.pinhole_camera(40, 24, (0.1, 0.2, -3.0))
    wide = dict(bvh_width=4) if width == 4 else {}
    r = R.render(sc, cam, k=4, want_stats=True, **opts, **wide)
    st = N.stats_dict(r["stats"])
    assert 0 < st["fallbacks"] <= st["rays"] == 40 * 24
    ref = R.render(sc, cam, k=4, traversal="restart", **wide)["rgbT"]
    torch.cuda.synchronize()
    np.testing.assert_allclose(r["rgbT"].cpu().numpy(), ref.cpu().numpy(), rtol=0, atol=1e-5)
    sc.close()


@pytest.mark.parametrize("entry", ["frame", "batch"])
def test_restart_fills_the_multiprocessors(entry):
    """A restarted launch keeps no walk: at k = 32 six of its blocks fit a multiprocessor (32 KB of k-buffers and
    3 KB of packet stacks each, of 228 KB), and the launch takes slots for as many (three 8-byte words each)."""
    g = scenes.tiny_scene(seed=1, n=200)
    sc = R.Scene.from_params(g)
    cam = scenes.pinhole_camera(32, 32, (0.0, 0.0, -3.0))
    if entry == "frame":
        R.render(sc, cam, k=32, traversal="restart")
    else:
        R.render_batch(sc, [(cam, None), (cam, None)], k=32, traversal="restart")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert sc.info()["bytes_workspace"] >= 6 * sms * 128 * 3 * 8
    sc.close()


@pytest.fixture(scope="module")
def big():
    """2^24 + 77 faint Gaussians in a box, about 150 hits a ray: too many leaf slots for a list entry that holds a
    slot and an opacity code."""
    n = (1 << 24) + 77
    gen = torch.Generator("cuda").manual_seed(9)
    means = torch.rand((n, 3), generator=gen, device="cuda") * 2 - 1
    scales = torch.log(torch.rand((n, 3), generator=gen, device="cuda") * 0.002 + 0.0015)
    q = torch.randn((n, 4), generator=gen, device="cuda")
    sh = torch.randn((n, 1, 3), generator=gen, device="cuda") * 0.3
    sc = R.Scene(means, scales, q, torch.full((n,), float(np.log(0.03 / 0.97)), device="cuda"), sh, 0)
    del means, scales, q, sh
    assert sc.info()["n_valid"] == n
    yield sc
    sc.close()
    torch.cuda.empty_cache()


@pytest.mark.parametrize("k,opts", [(8, {}), (16, {}), (16, dict(evict_capacity=100)), (8, dict(T_min=0.2))])
def test_scenes_of_more_slots_than_codes_leave_room_for(big, k, opts):
    cam = scenes.pinhole_camera(40, 24, (0.1, 0.2, -2.5))
    same = {a: v for a, v in opts.items() if a == "T_min"}
    a = R.render(big, cam, k=k, **opts)["rgbT"]
    b = R.render(big, cam, k=k, traversal="restart", **same)["rgbT"]
    torch.cuda.synchronize()
    assert 0.0 < float(b[:, 3].min()) < 0.5
    np.testing.assert_array_equal(a[:, 3].cpu().numpy(), b[:, 3].cpu().numpy())
    np.testing.assert_allclose(a.cpu().numpy(), b.cpu().numpy(), rtol=0, atol=1e-5)


@pytest.mark.parametrize("k", [8, 16])
def test_worlds_of_more_slots_than_codes_leave_room_for(big, k):
    small = R.Scene.from_params(scenes.surface_scene(n=3000, seed=5, n_spheres=4, n_patches=4))
    M = np.eye(4)[:3]
    world = R.World([(big, M), (small, M + [[0, 0, 0, 0.5]] * 3)])
    cam = scenes.pinhole_camera(40, 24, (0.1, 0.2, -2.5))
    a = R.render_world(world, cam, k=k)["rgbT"]
    b = R.render_world(world, cam, k=k, traversal="restart")["rgbT"]
    torch.cuda.synchronize()
    np.testing.assert_array_equal(a[:, 3].cpu().numpy(), b[:, 3].cpu().numpy())
    np.testing.assert_allclose(a.cpu().numpy(), b.cpu().numpy(), rtol=0, atol=1e-5)
    world.close()
    small.close()

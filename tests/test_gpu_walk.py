"""The tile walk (the uninstrumented first round of checkpointed sphere-form traces) against restart
traversal, which walks the tree for each ray and keeps no lists: both blend the same Gaussians in the
same order with the same arithmetic, so transmittances are bitwise equal, and colours agree to the
contraction of the SH polynomials in two kernels (a few ulp of sums of at most about 8: 1e-5)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2601_20429_gb300 import render as R
from paper_2601_20429_gb300 import scenes
from paper_2601_20429_gb300.serve import Server

TOL = 1e-5


def _fog(n=3000, seed=3):
    """Large faint Gaussians around the origin: over a thousand hits per ray, far more than a list holds."""
    rng = np.random.default_rng(seed)
    q = rng.standard_normal((n, 4))
    logits = np.log(0.02 / 0.98) + 0.2 * rng.standard_normal(n)
    return scenes.GaussianParams(rng.uniform(-1, 1, (n, 3)).astype(np.float32),
                                 np.log(rng.uniform(0.3, 0.9, (n, 3))).astype(np.float32),
                                 (q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32),
                                 logits.astype(np.float32), rng.normal(0, 0.3, (n, 4, 3)).astype(np.float32), 1)


def _scene(kind):
    if kind == "fog":
        return _fog()
    if kind == "surface":
        return scenes.surface_scene(n=20000, seed=5, n_spheres=8, n_patches=8)
    if kind == "outdoor":
        return scenes.outdoor_scene(n=20000, seed=6, size=16.0, n_clusters=20)
    return scenes.surface_scene(n=int(kind), seed=7, n_spheres=1, n_patches=1, extent=0.1)


@pytest.fixture(scope="module")
def built():
    cache = {}

    def get(kind):
        if kind not in cache:
            cache[kind] = R.Scene.from_params(_scene(kind))
        return cache[kind]

    yield get
    for sc in cache.values():
        sc.close()


def _same(a, b):
    torch.cuda.synchronize()
    np.testing.assert_array_equal(a[:, 3].cpu().numpy(), b[:, 3].cpu().numpy())
    np.testing.assert_allclose(a.cpu().numpy(), b.cpu().numpy(), rtol=0, atol=TOL)


CAMS = {
    "one": scenes.pinhole_camera(1, 1, (0.0, 0.0, -3.0)),
    "tile": scenes.pinhole_camera(8, 4, (0.1, 0.2, -3.0)),
    "ragged": scenes.pinhole_camera(33, 17, (0.5, -0.4, -2.5), fov_y_deg=80.0),
    "axis": scenes.pinhole_camera(32, 32, (0.0, 0.0, 0.0), (0.0, 0.0, 1.0), 90.0, t_near=0.2, t_far=2.5),
    "fisheye": scenes.fisheye_camera(96, 50, (0.0, 1.7, 0.0), (1.0, 0.0, 0.0), 90.0),
}


@pytest.mark.parametrize("kind", ["surface", "outdoor", "fog", "1", "2", "3"])
@pytest.mark.parametrize("cam", sorted(CAMS))
@pytest.mark.parametrize("k", [1, 8, 16, 32])
def test_walk_equals_restart(built, kind, cam, k):
    sc = built(kind)
    a = R.render(sc, CAMS[cam], k=k)["rgbT"]
    b = R.render(sc, CAMS[cam], k=k, traversal="restart")["rgbT"]
    _same(a, b)


@pytest.mark.parametrize("kind", ["surface", "fog"])
@pytest.mark.parametrize("opts", [dict(evict_capacity=1), dict(evict_capacity=40), dict(evict_capacity=100),
                                  dict(evict_capacity=2000), dict(ckpt_capacity=3), dict(packet_stack=1),
                                  dict(packet_stack=30), dict(T_min=0.0), dict(T_min=0.5),
                                  dict(alpha_max=0.9999999, T_min=1e-6), dict(bg=(0.3, 0.2, 0.1))])
def test_walk_limits(built, kind, opts):
    """Short lists and stacks, no or early termination: the same image whichever way the ray goes on."""
    sc = built(kind)
    same = {k: v for k, v in opts.items() if k in ("T_min", "alpha_max", "bg")}
    _same(R.render(sc, CAMS["ragged"], k=8, **opts)["rgbT"],
          R.render(sc, CAMS["ragged"], k=8, traversal="restart", **same)["rgbT"])


@pytest.mark.parametrize("n", [1, 31, 33, 777])
def test_walk_ray_lists(built, n):
    """Scattered rays (bundles that share nothing), with per-ray ranges, a negative t_near, zero direction
    components and rays that are not finite among them."""
    sc = built("surface")
    rng = np.random.default_rng(n)
    o = rng.uniform(-2, 2, (n, 3)).astype(np.float32)
    d = rng.standard_normal((n, 3)).astype(np.float32)
    d[::5, 0] = 0.0
    d[::7, 1:] = 0.0
    tn = np.where(rng.uniform(size=n) < 0.2, -1.0, 0.01).astype(np.float32)
    tf = rng.uniform(0.5, 9.0, n).astype(np.float32)
    tf[::11] = math.inf
    tf[::13] = -2.0
    if n > 64:
        d[40], d[41, 1], o[42, 2] = math.nan, math.inf, math.nan
    rays = tuple(torch.from_numpy(x).cuda() for x in (o, d, tn, tf))
    a = R.render(sc, None, rays=rays, k=16)["rgbT"]
    b = R.render(sc, None, rays=rays, k=16, traversal="restart")["rgbT"]
    fine = torch.isfinite(rays[1]).all(1) & torch.isfinite(rays[0]).all(1)
    _same(a[fine], b[fine])


@pytest.mark.parametrize("size", [(8, 4), (64, 64), (250, 130), (300, 301), (640, 360)])
def test_walk_of_split_tiles(built, size):
    """Launches of few tiles split them over the resident warps, by up to eight."""
    cam = scenes.pinhole_camera(*size, (0.5, 0.4, -2.5))
    sc = built("surface")
    _same(R.render(sc, cam, k=16)["rgbT"], R.render(sc, cam, k=16, traversal="restart")["rgbT"])


@pytest.mark.parametrize("kind,opts", [("surface", {}), ("fog", {}), ("fog", dict(evict_capacity=40)),
                                       ("surface", dict(packet_stack=2)), ("1", {})])
@pytest.mark.parametrize("shape", [(5000, 1), (40, 30)])
def test_walk_of_scattered_rays(built, kind, opts, shape):
    """Ray lists whose bundles share nothing are traced one ray to a warp."""
    n = shape[0] * shape[1]
    rng = np.random.default_rng(n)
    d = rng.standard_normal((n, 3))
    rays = [torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()
            for x in (rng.uniform(-1, 1, (n, 3)), d, np.zeros(n), np.full(n, math.inf))]
    cam = None if shape[1] == 1 else dict(scenes.pinhole_camera(*shape, (0.0, 0.0, -3.0)))
    sc = built(kind)
    _same(R.render(sc, cam, rays=rays, k=8, **opts)["rgbT"], R.render(sc, cam, rays=rays, k=8, traversal="restart")["rgbT"])


@pytest.mark.parametrize("kind", ["surface", "fog"])
def test_walk_in_batches_and_servers(built, kind):
    sc = built(kind)
    cams = [CAMS["ragged"], CAMS["tile"], CAMS["fisheye"]]
    ref = [R.render(sc, c, k=16, traversal="restart")["rgbT"] for c in cams]
    for a, b in zip(R.render_batch(sc, [(c, None) for c in cams], k=16), ref):
        _same(a, b)
    srv = Server([sc], k=16)
    outs = [torch.empty_like(r) for r in ref]
    srv.render_requests([(0, c, o, i) for i, (c, o) in enumerate(zip(cams, outs))])
    for a, b in zip(outs, ref):
        _same(a, b)
    srv.close()


@pytest.mark.parametrize("n", [1, 33, 900, 5001])
@pytest.mark.parametrize("opts", [{}, dict(evict_capacity=40), dict(packet_stack=2)])
@pytest.mark.parametrize("image", [CAMS["ragged"], scenes.pinhole_camera(701, 401, (0.3, 0.2, -3.5), (0, 0, 0), 60.0)])
def test_walk_of_lists_in_batches(built, n, opts, image):
    """Short ray lists beside an image in one launch (beside one that fills the GPU in smaller bundles;
    scattered ones left to the one-ray kernel)."""
    sc = built("surface")
    rng = np.random.default_rng(n)
    near = rng.uniform(-0.02, 0.02, (n, 3)) + [0.0, 0.0, 1.0]
    lists = [tuple(torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda() for x in (o, d, np.full(n, 1e-3), np.full(n, 9.0)))
             for o, d in ((rng.uniform(-2, 2, (n, 3)), rng.standard_normal((n, 3))), (np.tile([0.1, 0.2, -3.0], (n, 1)), near))]
    views = [(image, None), (None, lists[0]), (None, lists[1])]
    outs = R.render_batch(sc, views, k=8, **opts)
    for (cam, rays), a in zip(views, outs):
        _same(a, R.render(sc, cam, rays=rays, k=8, traversal="restart")["rgbT"])


@pytest.mark.parametrize("kind", ["surface", "fog"])
@pytest.mark.parametrize("save", [0, 16])
def test_walk_backward(built, kind, save):
    """Gradients through the walk against those through restart rounds: the same terms, summed by atomics in
    another order (2-norm within 1e-5 of it)."""
    sc = built(kind)
    cam = CAMS["ragged"]
    up = torch.randn((33 * 17, 4), generator=torch.Generator("cuda").manual_seed(1), device="cuda")
    f = R.render(sc, cam, k=8, save_cap=save)
    r = R.render(sc, cam, k=8, traversal="restart")
    _same(f["rgbT"], r["rgbT"])
    a = R.backward(sc, cam, f["rgbT"], up, k=8, saved=f.get("saved"))
    b = R.backward(sc, cam, r["rgbT"], up, k=8, traversal="restart")
    for name in a:
        assert float((a[name] - b[name]).norm()) <= 1e-5 * float(b[name].norm()), name


@pytest.mark.parametrize("kind", ["surface", "fog", "1"])
@pytest.mark.parametrize("k,opts", [(8, {}), (16, {}), (32, {}), (8, dict(evict_capacity=40)), (8, dict(evict_capacity=1)),
                                    (16, dict(packet_stack=1)), (16, dict(T_min=0.0))])
def test_walk_of_worlds(built, kind, k, opts):
    """Overlapping, rotated, sheared and distant placements, walked object by object, against restart rounds."""
    M = [np.eye(4)[:3], np.array([[0.0, -0.6, 0.0, 0.5], [0.6, 0.0, 0.1, 0.2], [0.0, 0.0, 0.8, 0.3]]),
         np.array([[1.3, 0.0, 0.2, -0.9], [0.0, 0.7, 0.0, 0.1], [0.0, 0.0, 1.0, 1.5]]), np.eye(4)[:3] + [[0, 0, 0, 40.0]] * 3]
    world = R.World([(built(n), m) for n, m in zip((kind, "outdoor", kind, kind), M)])
    same = {a: v for a, v in opts.items() if a == "T_min"}
    for cam in ("ragged", "one", "axis"):
        _same(R.render_world(world, CAMS[cam], k=k, **opts)["rgbT"],
              R.render_world(world, CAMS[cam], k=k, traversal="restart", **same)["rgbT"])
    world.close()

"""The walks' index checks: the first round of the uninstrumented kernels, over the cases where their stacks,
leaf lists, eviction lists and left list fill, without an index outside its array."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2601_20429_gb300 import native as N
from paper_2601_20429_gb300 import render as R
from paper_2601_20429_gb300 import scenes


def _faint(n=3000, seed=3):
    rng = np.random.default_rng(seed)
    q = rng.standard_normal((n, 4))
    return scenes.GaussianParams(rng.uniform(-1, 1, (n, 3)).astype(np.float32),
                                 np.log(rng.uniform(0.3, 0.9, (n, 3))).astype(np.float32),
                                 (q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32),
                                 np.full(n, np.log(0.02 / 0.98), np.float32), rng.normal(0, 0.3, (n, 4, 3)).astype(np.float32), 1)


SCENES = {"surface": lambda: scenes.surface_scene(n=20000, seed=5, n_spheres=8, n_patches=8),
          "outdoor": lambda: scenes.outdoor_scene(n=20000, seed=6, size=16.0, n_clusters=20),
          "fog": _faint, "1": lambda: scenes.surface_scene(n=1, seed=7, n_spheres=1, n_patches=1, extent=0.1)}
CAMS = [scenes.pinhole_camera(64, 40, (0.5, 0.4, -2.5)), scenes.pinhole_camera(701, 401, (0.3, 0.2, -3.5), (0, 0, 0), 60.0),
        scenes.fisheye_camera(96, 50, (0.0, 1.7, 0.0), (1.0, 0.0, 0.0), 90.0)]
OPTS = [{}, dict(evict_capacity=1), dict(evict_capacity=40), dict(packet_stack=1), dict(packet_stack=24), dict(T_min=0.0)]


def _checked(call, cam, rays, opts, **kw):
    n = int(rays[0].shape[0]) if rays else cam["width"] * cam["height"]
    out, errors = torch.empty((n, 4), device="cuda"), torch.zeros(1, dtype=torch.int64, device="cuda")
    call(N.make_camera(cam, rays), R.trace_params(k=16, **opts), out, errors, **kw)
    torch.cuda.synchronize()
    return out, int(errors.item())


def _scattered(n):
    rng = np.random.default_rng(n)
    return tuple(torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).cuda()
                 for x in (rng.uniform(-1, 1, (n, 3)), rng.standard_normal((n, 3)), np.zeros(n), np.full(n, math.inf)))


@pytest.mark.parametrize("kind", sorted(SCENES))
@pytest.mark.parametrize("opts", OPTS)
def test_walks_stay_inside_their_arrays(kind, opts):
    sc = R.Scene.from_params(SCENES[kind]())
    call = lambda *a, **k: N.grtx_trace_self_check(sc.handle, *a, **k)  # noqa: E731
    for cam, rays in [(c, None) for c in CAMS] + [(None, _scattered(33)), (None, _scattered(5000))]:
        out, errors = _checked(call, cam, rays, opts)
        assert errors == 0
        ref = R.render(sc, cam, rays=rays, k=16, **opts)["rgbT"]
        np.testing.assert_allclose(out.cpu().numpy(), ref.cpu().numpy(), rtol=0, atol=1e-5)
    sc.close()


def test_the_check_counts_what_it_leaves_out():
    """With the scene's nodes said to be fewer than they are, the walks count and leave out the others."""
    sc = R.Scene.from_params(SCENES["surface"]())
    call = lambda *a, **k: N.grtx_trace_self_check(sc.handle, *a, **k)  # noqa: E731
    for cam, rays in ((CAMS[0], None), (None, _scattered(5000))):
        assert _checked(call, cam, rays, {}, max_nodes=sc.info()["n_nodes"])[1] == 0
        out, errors = _checked(call, cam, rays, {}, max_nodes=100)
        assert errors > 0 and bool(torch.isfinite(out).all())
    sc.close()


@pytest.mark.parametrize("kind", ["surface", "fog", "1"])
@pytest.mark.parametrize("opts", OPTS)
def test_world_walks_stay_inside_their_arrays(kind, opts):
    a, b = R.Scene.from_params(SCENES[kind]()), R.Scene.from_params(SCENES["outdoor"]())
    M = [np.eye(4)[:3], np.array([[0.0, -0.6, 0.0, 0.5], [0.6, 0.0, 0.1, 0.2], [0.0, 0.0, 0.8, 0.3]]),
         np.eye(4)[:3] + [[0, 0, 0, 40.0]] * 3]
    world = R.World([(a, M[0]), (b, M[1]), (a, M[2])])
    for cam in CAMS:
        out, errors = _checked(lambda *x: N.grtx_world_self_check(world.handle, *x), cam, None, opts)
        assert errors == 0
        ref = R.render_world(world, cam, k=16, **opts)["rgbT"]
        np.testing.assert_allclose(out.cpu().numpy(), ref.cpu().numpy(), rtol=0, atol=1e-5)
    world.close()


def test_self_check_arguments():
    sc = R.Scene.from_params(SCENES["1"]())
    out, errors = torch.empty((64 * 40, 4), device="cuda"), torch.zeros(1, dtype=torch.int64, device="cuda")
    for bad in (dict(k=8), dict(k=16, traversal="restart")):
        with pytest.raises(N.GrtxError):
            N.grtx_trace_self_check(sc.handle, N.make_camera(CAMS[0]), R.trace_params(**bad), out, errors)
    with pytest.raises(N.GrtxError):
        N.grtx_trace_self_check(sc.handle, N.make_camera(CAMS[0]), R.trace_params(k=16), out, None)
    sc.close()

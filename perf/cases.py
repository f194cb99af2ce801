"""What a user of this framework has it do, as cases that can be timed and compared.

A case is a dict of plain values. `prepare` makes from a seed what a user's program holds before the
call (Gaussians, cameras, a built scene, a world, a server), `run` is one pass through the public
entry points, `work` the bytes and operations the pass cannot do without, and `exact` the same
outputs from plain torch in 64 bits. Sizes follow the framework's own configurations
(paper_2601_20429_gb300/scenes.py, bench.py and the tests): scenes of 1,000 to 6,000,000 Gaussians,
images from 64x64 to 1920x1080, k of 8, 16 and 32, spherical harmonics of degree 0 to 3.
"""
import math

import numpy as np
import torch

from paper_2601_20429_gb300 import render as R
from paper_2601_20429_gb300 import scenes
from paper_2601_20429_gb300.serve import Server

ALPHA_MIN, ALPHA_MAX, T_MIN = 0.01, 0.99, 1e-3
BG = (0.05, 0.1, 0.2)


# ------------------------------------------------------------------------------------------
# Cases
# ------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: an image of the tiny configuration, where launch and latency count
        dict(name="tiny_frame", kind="frame", scene="tiny", n=1000, sh=0, width=64, height=64, k=8, dist=3.0,
             traversal="checkpoint"),
        # a preview or a small request: too few tiles to fill the GPU for long
        dict(name="preview_256", kind="frame", scene="surface", n=500_000, sh=3, width=256, height=256, k=16, dist=5.0,
             traversal="checkpoint"),
        # the configuration the headline metric is quoted on: one frame of a 1M surface scene
        dict(name="frame_1080p", kind="frame", scene="surface", n=1_000_000, sh=3, width=1920, height=1080, k=16,
             dist=4.0, traversal="checkpoint"),
        # a close serving view of a large scene: many Gaussians per ray, early termination matters
        dict(name="view_720p_deep", kind="frame", scene="surface", n=2_000_000, sh=3, width=1280, height=720, k=16,
             dist=3.0, traversal="checkpoint"),
        # the large outdoor configuration: 6M Gaussians, fisheye primary rays and the bounce rays of a mirror and
        # a glass ball, traced in one launch
        dict(name="outdoor_bounce", kind="bounce", scene="outdoor", n=6_000_000, sh=3, width=1920, height=1080, k=16,
             traversal="checkpoint"),
        # an explicit list of rays without order (secondary or probe rays), ragged, at the larger k
        dict(name="rays_scattered", kind="rays", scene="surface", n=1_000_000, sh=3, rays=20_011, k=32,
             traversal="checkpoint"),
        # several placed objects (multi-level instancing)
        dict(name="world_8", kind="world", scene="surface", n=250_000, sh=3, width=1280, height=720, k=16, places=8,
             traversal="checkpoint"),
        # the training step: the scene kept across steps and refitted, forward and backward
        dict(name="train_refit", kind="train", scene="surface", n=262_144, sh=3, width=800, height=800, k=16, keep=1,
             save=0),
        # a training step that saves the blend lists, on an odd image and an odd number of Gaussians
        dict(name="train_saved", kind="train", scene="surface", n=65_537, sh=3, width=401, height=299, k=8, keep=1,
             save=64),
        # the plain differentiable call: a tree built anew at every step, small scene, degree 1
        dict(name="train_rebuild", kind="train", scene="surface", n=20_000, sh=1, width=128, height=128, k=16, keep=0,
             save=0),
        # loading a scene: the whole acceleration structure, and its arrays exported
        dict(name="build_1m", kind="build", scene="surface", n=1_000_000, sh=3, builder="ploc"),
        # a burst of mixed requests to the server
        dict(name="serve_burst", kind="serve", scene="surface", n=500_000, sh=3, k=16, requests=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "train", "train", "build", "rays", "world", "bounce", "serve"])
    sh = rng.choice([3, 3, 3, 2, 1, 0])
    k = rng.choice([8, 16, 16, 32])
    trav = rng.choice(["checkpoint", "checkpoint", "checkpoint", "restart", "single"])
    px = _log(rng, 64 * 64, 1280 * 720)
    width = max(16, int(math.sqrt(px * rng.uniform(0.8, 2.0))))
    height = max(16, px // width)
    if kind == "frame":
        return dict(kind=kind, scene="surface", n=_log(rng, 1000, 2_000_000), sh=sh, width=width, height=height, k=k,
                    dist=round(rng.uniform(3.0, 8.0), 3), traversal=trav)
    if kind == "train":
        px = _log(rng, 64 * 64, 800 * 800)
        width = max(16, int(math.sqrt(px * rng.uniform(0.8, 2.0))))
        return dict(kind=kind, scene="surface", n=_log(rng, 2000, 262_144), sh=sh, width=width,
                    height=max(16, px // width), k=k, keep=rng.choice([1, 1, 0]), save=rng.choice([0, 0, 64, 24]))
    if kind == "build":
        return dict(kind=kind, scene=rng.choice(["surface", "outdoor"]), n=_log(rng, 2000, 2_000_000), sh=sh,
                    builder=rng.choice(["ploc", "ploc", "lbvh"]))
    if kind == "rays":
        return dict(kind=kind, scene="surface", n=_log(rng, 10_000, 1_000_000), sh=sh, rays=_log(rng, 500, 50_000), k=k,
                    traversal=rng.choice(["checkpoint", "checkpoint", "restart"]))
    if kind == "world":
        return dict(kind=kind, scene="surface", n=_log(rng, 5000, 500_000), sh=sh, width=width, height=height, k=k,
                    places=rng.randint(2, 12), traversal=rng.choice(["checkpoint", "checkpoint", "restart"]))
    if kind == "bounce":
        return dict(kind=kind, scene="outdoor", n=_log(rng, 100_000, 3_000_000), sh=sh, width=width, height=height, k=k,
                    traversal="checkpoint")
    return dict(kind=kind, scene="surface", n=_log(rng, 50_000, 500_000), sh=sh, k=k, requests=rng.randint(3, 16))


# ------------------------------------------------------------------------------------------
# Inputs. The scene generators draw the distributions of scenes.py on the GPU.
# ------------------------------------------------------------------------------------------
class _Draw:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda").manual_seed(int(seed))

    def u(self, lo, hi, *shape):
        return torch.rand(shape, generator=self.g, device="cuda") * (hi - lo) + lo

    def n(self, mean, std, *shape):
        return torch.randn(shape, generator=self.g, device="cuda") * std + mean

    def unit(self, n):
        return torch.nn.functional.normalize(self.n(0.0, 1.0, n, 3), dim=1)

    def pick(self, n, weights):
        c = torch.cumsum(weights.double(), 0)
        at = torch.rand(n, generator=self.g, device="cuda", dtype=torch.float64) * c[-1]
        return torch.searchsorted(c, at).clamp_(max=weights.numel() - 1)


def _quat_z_to(normal, twist):
    """Quaternion (w, x, y, z) that takes +z to `normal` after a twist about +z."""
    w, x, y = 1.0 + normal[:, 2], -normal[:, 1], normal[:, 0]
    flip = w < 1e-6
    w = torch.where(flip, torch.zeros_like(w), w)
    x = torch.where(flip, torch.ones_like(x), x)
    inv = torch.rsqrt(w * w + x * x + y * y)
    w, x, y = w * inv, x * inv, y * inv
    c, s = torch.cos(0.5 * twist), torch.sin(0.5 * twist)
    return torch.stack([w * c, x * c + y * s, y * c - x * s, w * s], 1)


def _on_surfaces(r, pts, nrm, sh, noise):
    n = pts.shape[0]
    st = torch.exp(r.n(math.log(0.01), 0.3, n, 2))
    sn = st.amin(1, keepdim=True) * torch.exp(-r.u(0.0, math.log(100.0), n, 1))
    o = torch.sin(r.u(0.0, 0.5 * math.pi, n)).square().clamp(0.0105, 1 - 1e-6)    # Beta(1/2, 1/2), ...
    o[torch.topk(o, n // 16, largest=False).indices] = 0.004                      # ... and n / 16 below alpha_min
    return [pts + r.n(0.0, noise, n, 3), torch.log(torch.cat([st, sn], 1)), _quat_z_to(nrm, r.u(0.0, 2 * math.pi, n)),
            torch.logit(o), r.n(0.0, 0.3, n, (sh + 1) ** 2, 3)]


def _gaussians(scene, n, sh, seed):
    """[means, log_scales, quats, logits, sh], float32 on the GPU."""
    r = _Draw(seed)
    if scene == "tiny":
        q = torch.nn.functional.normalize(r.n(0.0, 1.0, n, 4), dim=1)
        return [r.u(-1.0, 1.0, n, 3), r.u(-4.5, -2.5, n, 3), q, r.n(0.0, 1.0, n),
                (r.u(0.0, 1.0, n, (sh + 1) ** 2, 3) - 0.5) * scenes.TWO_SQRT_PI]
    if scene == "surface":                      # 100 noisy spheres and 100 square patches
        sc, pc = r.u(-2.0, 2.0, 100, 3), r.u(-2.0, 2.0, 100, 3)
        rad, side = r.u(0.1, 0.6, 100), r.u(0.3, 1.5, 100)
        pn = r.unit(100)
        pu = torch.nn.functional.normalize(torch.linalg.cross(pn, r.unit(100)), dim=1)
        pv = torch.linalg.cross(pn, pu)
        at = r.pick(n, torch.cat([4 * math.pi * rad * rad, side * side]))
        s, p = at.clamp(max=99), (at - 100).clamp(min=0)
        u = r.unit(n)
        ab = r.u(-0.5, 0.5, n, 2) * side[p, None]
        ball = (at < 100)[:, None]
        pts = torch.where(ball, sc[s] + rad[s, None] * u, pc[p] + ab[:, :1] * pu[p] + ab[:, 1:] * pv[p])
        return _on_surfaces(r, pts, torch.where(ball, u, pn[p]), sh, 0.01)
    half = n // 2                               # outdoor: a 100 m ground plane, and 500 clusters on it
    ground = torch.stack([r.u(-50.0, 50.0, half), torch.zeros(half, device="cuda"), r.u(-50.0, 50.0, half)], 1)
    rad = torch.exp(r.u(math.log(0.2), math.log(5.0), 500))
    cen = torch.stack([r.u(-50.0, 50.0, 500), rad, r.u(-50.0, 50.0, 500)], 1)
    shell = r.u(0.0, 1.0, 500) < 0.5
    c = r.pick(n - half, torch.ones(500, device="cuda"))
    u = r.unit(n - half)
    far = torch.where(shell[c], rad[c], rad[c] * r.n(0.0, 0.5, n - half).abs())
    up = torch.tensor([[0.0, 1.0, 0.0]], device="cuda").expand(half, 3)
    g = _on_surfaces(r, torch.cat([ground, cen[c] + far[:, None] * u]), torch.cat([up, u]), sh, 0.0)
    base = torch.exp(r.n(math.log(0.03), 1.0, n)).clamp(0.005, 5.0)
    g[1] = g[1] - math.log(0.01) + torch.log(base)[:, None]
    return g


def _pose(rng, dist):
    v = rng.standard_normal(3)
    v = v / np.linalg.norm(v)
    return tuple(float(x) for x in dist * v)


def _camera(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] == "bounce":
        return scenes.fisheye_camera(case["width"], case["height"], (0.0, 1.7, 0.0), (1.0, 0.0, 0.0), 90.0)
    return scenes.pinhole_camera(case["width"], case["height"], _pose(rng, case.get("dist", 4.0)), (0.0, 0.0, 0.0), 60.0)


def _camera_rays64(cam):
    """Origins and unit directions of a camera in 64 bits, from its float32 description, in pixel order."""
    f = lambda v: torch.tensor(np.asarray(v, np.float32).astype(np.float64), device="cuda")  # noqa: E731
    W, H, fov = cam["width"], cam["height"], float(np.float32(cam["fov"]))
    y, x = torch.meshgrid(torch.arange(H, device="cuda", dtype=torch.float64) + 0.5,
                          torch.arange(W, device="cuda", dtype=torch.float64) + 0.5, indexing="ij")
    x, y = x.reshape(-1, 1), y.reshape(-1, 1)
    if cam["type"] == scenes.PINHOLE:
        u, v = (2 * x / W - 1) * math.tan(0.5 * fov) * W / H, (1 - 2 * y / H) * math.tan(0.5 * fov)
        d = f(cam["forward"]) + u * f(cam["right"]) + v * f(cam["up"])
    else:
        ex, ey = x - 0.5 * W, 0.5 * H - y
        r = torch.sqrt(ex * ex + ey * ey)
        th, ri = r / (0.5 * W / fov), 1.0 / r.clamp(min=1e-300)
        d = torch.sin(th) * (ex * ri * f(cam["right"]) + ey * ri * f(cam["up"])) + torch.cos(th) * f(cam["forward"])
    return f(cam["pos"]).expand(W * H, 3), torch.nn.functional.normalize(d, dim=1)


def _bounce_rays(cam):
    """Primary rays clipped at a mirror, and its reflected rays: (o, d, tnear, tfar) lists."""
    m = scenes.outdoor_mirror()
    o, d = _camera_rays64(cam)
    f = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda")  # noqa: E731
    dn = (d * f(m["normal"])).sum(1)
    t = ((f(m["center"]) - o) * f(m["normal"])).sum(1) / dn
    p = o + t[:, None] * d
    q = p - f(m["center"])
    hit = (t > 0) & ((q * f(m["axis_u"])).sum(1).abs() <= m["half_u"]) & ((q * f(m["axis_v"])).sum(1).abs() <= m["half_v"])
    n = o.shape[0]
    tf = torch.where(hit, t, torch.full_like(t, math.inf))
    s = torch.cat([hit.nonzero()[:, 0], torch.zeros(1, dtype=torch.long, device="cuda")])   # (never empty)
    d2 = d[s] - 2 * dn[s, None] * f(m["normal"])
    prim = (o, d, torch.zeros(n, device="cuda"), tf)
    sec = (torch.where(hit[s, None], p[s], o[s]), torch.nn.functional.normalize(d2, dim=1),
           torch.full((s.numel(),), 1e-3, device="cuda"), torch.full((s.numel(),), math.inf, device="cuda"))
    return [tuple(v.float().contiguous() for v in r) for r in (prim, sec)]


def _scattered_rays(case, g, seed):
    """Rays from points of the scene in random directions (as diffuse bounces are)."""
    r = _Draw(seed + 77)
    n = case["rays"]
    at = r.pick(n, torch.ones(case["n"], device="cuda"))
    d = r.unit(n)
    return (g[0][at] + 0.05 * d).contiguous(), d.contiguous(), torch.full((n,), 1e-3, device="cuda"), \
        torch.full((n,), math.inf, device="cuda")


def _placements(case, seed):
    rng = np.random.default_rng(seed)
    out = []
    for i in range(case["places"]):
        a, b, s = rng.uniform(0, 2 * math.pi), rng.uniform(-0.5, 0.5), rng.uniform(0.5, 1.0)
        ra = np.array([[math.cos(a), 0, math.sin(a)], [0, 1, 0], [-math.sin(a), 0, math.cos(a)]])
        rb = np.array([[1, 0, 0], [0, math.cos(b), -math.sin(b)], [0, math.sin(b), math.cos(b)]])
        M = np.zeros((3, 4))
        M[:, :3] = s * ra @ rb
        M[:, 3] = [5.0 * math.cos(2 * math.pi * i / case["places"]), rng.uniform(-0.5, 0.5),
                   5.0 * math.sin(2 * math.pi * i / case["places"])]
        out.append((i % 2, M.astype(np.float32).astype(np.float64)))
    return out


SERVE_SIZES = ((256, 256), (512, 512), (1280, 720), (611, 357))


def _requests(case, seed):
    rng = np.random.default_rng(seed)
    reqs = []
    for i in range(case["requests"]):
        w, h = SERVE_SIZES[i % len(SERVE_SIZES)]
        reqs.append((i % 2, scenes.pinhole_camera(w, h, _pose(rng, rng.uniform(3.0, 8.0)), (0.0, 0.0, 0.0), 60.0)))
    return reqs


def _opts(case):
    return dict(k=case["k"], traversal=case.get("traversal", "checkpoint"), bg=BG)


def prepare(case, seed):
    kind, s = case["kind"], dict(case=case)
    g = _gaussians(case["scene"], case["n"], case["sh"], seed)
    if kind in ("world", "serve"):
        two = [g, _gaussians(case["scene"], 2 * case["n"], case["sh"], seed + 1)]
        s["scenes"] = [R.Scene(*x, case["sh"]) for x in two]
        if kind == "world":
            s["world"] = R.World([(s["scenes"][i], M) for i, M in _placements(case, seed)])
            s["cam"] = scenes.pinhole_camera(case["width"], case["height"], (0.0, 3.0, -9.0), (0.0, 0.0, 0.0), 60.0)
        else:
            s["server"] = Server(s["scenes"], k=case["k"], bg=BG)
            s["reqs"] = [(i, cam, torch.empty((cam["width"] * cam["height"], 4), device="cuda"), tag)
                         for tag, (i, cam) in enumerate(_requests(case, seed))]
        return s
    s["g"] = g
    if kind == "build":
        return s
    if kind == "train":
        s["cam"] = _camera(case, seed)
        s["params"] = [t.requires_grad_(True) for t in g]
        if case["keep"]:
            s["scene"] = R.Scene(*[t.detach() for t in g], case["sh"])
        s["upstream"] = _Draw(seed + 5).n(0.0, 1.0, case["width"] * case["height"], 4)
        return s
    s["scene"] = R.Scene(*g, case["sh"])
    if kind == "frame":
        s["cam"] = _camera(case, seed)
    elif kind == "bounce":
        s["cam"] = _camera(case, seed)
        s["views"] = _bounce_rays(s["cam"])
    else:
        s["rays"] = _scattered_rays(case, g, seed)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "frame":
        return R.render(s["scene"], s["cam"], **_opts(case))["rgbT"]
    if kind == "rays":
        return R.render(s["scene"], None, rays=s["rays"], **_opts(case))["rgbT"]
    if kind == "bounce":
        return R.render_batch(s["scene"], [(s["cam"], s["views"][0]), (None, s["views"][1])], **_opts(case))
    if kind == "world":
        return R.render_world(s["world"], s["cam"], **_opts(case))["rgbT"]
    if kind == "serve":
        s["server"].render_requests(s["reqs"])
        return [r[2] for r in s["reqs"]]
    if kind == "build":
        sc = R.Scene(*s["g"], case["sh"], bvh_builder=case["builder"])
        nodes, ids, codes = sc.export()
        sc.close()
        return [nodes[:, :12], nodes[:, 12:14].contiguous().view(torch.int32), ids, codes]
    o = dict(k=case["k"], bg=BG)
    if case["keep"]:
        o["scene"] = s["scene"]
    if case["save"]:
        o["save_cap"] = case["save"]
    img = R.render_differentiable(*s["params"], case["sh"], s["cam"], **o)
    grads = torch.autograd.grad(img, s["params"], s["upstream"])
    return [img.detach(), *grads]


# ------------------------------------------------------------------------------------------
# The work of one pass
# ------------------------------------------------------------------------------------------
def work(case):
    """Bytes: the Gaussians' parameters read once, the outputs written once. Operations: about 25 Gaussians
    composited per ray, each with its exact test (100), its colour (6 per coefficient and 20 for the basis) and the
    blend (10); a training step composites them twice and differentiates once (300 more)."""
    nk = (case["sh"] + 1) ** 2
    par = 4 * (11 + 3 * nk)
    blend = 130 + 6 * nk
    kind = case["kind"]
    if kind == "build":
        return dict(bytes=case["n"] * (par + 64 + 12), flops=case["n"] * 300)
    if kind in ("frame", "bounce"):
        px = case["width"] * case["height"]
        return dict(bytes=case["n"] * par + 16 * px, flops=25 * px * blend)
    if kind == "rays":
        return dict(bytes=case["n"] * par + (32 + 16) * case["rays"], flops=25 * case["rays"] * blend)
    if kind == "train":
        px = case["width"] * case["height"]
        return dict(bytes=2 * case["n"] * par + 32 * px, flops=25 * px * (2 * blend + 300))
    px = case["width"] * case["height"] if kind == "world" else sum(
        SERVE_SIZES[i % 4][0] * SERVE_SIZES[i % 4][1] for i in range(case["requests"]))
    return dict(bytes=3 * case["n"] * par + 16 * px, flops=25 * px * blend)


# ------------------------------------------------------------------------------------------
# The same outputs in 64 bits, from the definitions: alpha = o exp(-d^2/2) at the point of the ray nearest to the
# mean in the Gaussian's own metric, hits alpha >= ALPHA_MIN sorted by depth, front-to-back compositing that stops
# right after the Gaussian that takes the transmittance below T_MIN.
# ------------------------------------------------------------------------------------------
def _rot(q):
    w, x, y, z = torch.nn.functional.normalize(q, dim=-1).unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).unflatten(-1, (3, 3))


def _basis(n, deg):
    x, y, z = n.unbind(-1)
    p = math.pi
    Y = [torch.full_like(x, 0.5 / math.sqrt(p))]
    if deg >= 1:
        c = math.sqrt(3 / (4 * p))
        Y += [c * y, c * z, c * x]
    if deg >= 2:
        c = 0.5 * math.sqrt(15 / p)
        Y += [c * x * y, c * y * z, 0.25 * math.sqrt(5 / p) * (3 * z * z - 1), c * x * z, 0.5 * c * (x * x - y * y)]
    if deg >= 3:
        a, b, c = 0.25 * math.sqrt(35 / (2 * p)), 0.5 * math.sqrt(105 / p), 0.25 * math.sqrt(21 / (2 * p))
        Y += [a * y * (3 * x * x - y * y), b * x * y * z, c * y * (5 * z * z - 1),
              0.25 * math.sqrt(7 / p) * z * (5 * z * z - 3), c * x * (5 * z * z - 1), 0.5 * b * z * (x * x - y * y),
              a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, -1)


class _Field:
    """Gaussians in 64 bits, with the maps of placed objects where there are any."""

    def __init__(self, g, sh, at=None, maps=None):
        self.g, self.sh = [t.detach().double() for t in g], sh
        self.at, self.maps = at, maps                       # object of each Gaussian, its object-to-world map
        mu, ls, q, lo = self.g[:4]
        self.o = torch.sigmoid(lo)
        self.kap = torch.sqrt(2 * torch.log((self.o / ALPHA_MIN).clamp(min=1.0)))
        A = torch.exp(-ls)[:, :, None] * _rot(q).transpose(1, 2)      # whitening map of the offset from the mean
        size = torch.exp(ls).amax(1)
        self.mu = mu
        if at is not None:
            L = maps[:, :, :3]
            self.inv = torch.linalg.inv(L)
            A = A @ self.inv[at]
            self.mu = (L[at] @ mu[:, :, None])[:, :, 0] + maps[at, :, 3]
            size = size * torch.linalg.matrix_norm(L, 2)[at]
        self.A = A
        self.size = torch.where(self.o > ALPHA_MIN, self.kap * size, torch.full_like(size, -1.0))

    def near(self, o, d):
        """Gaussians that some ray of a common origin can hit: those that meet the cone around the rays."""
        ax = torch.nn.functional.normalize(d.mean(0), dim=0)
        half = torch.acos((d @ ax).clamp(-1, 1)).amax() + 1e-6
        v = self.mu - o[0]
        far = v.norm(dim=1)
        ang = torch.acos(((v @ ax) / far.clamp(min=1e-12)).clamp(-1, 1))
        wide = torch.asin((self.size / far.clamp(min=1e-12)).clamp(-1, 1))
        return ((self.size > 0) & ((far <= self.size) | (ang <= half + wide + 1e-6))).nonzero()[:, 0]

    def hits(self, o, d, tn, tf, at):
        """(R, H) ids of each ray's hits in depth order up to termination, and which of them are real."""
        A, mu = self.A[at], self.mu[at]
        dl = [d @ A[:, j].T for j in range(3)]
        if bool((o == o[0]).all()):
            w = (o[0] - mu)[:, :, None]
            ol = [(A[:, j:j + 1] @ w)[:, 0, 0][None, :] for j in range(3)]
        else:
            ol = [o @ A[:, j].T - (A[:, j] * mu).sum(1)[None, :] for j in range(3)]
        aa = dl[0] * dl[0] + dl[1] * dl[1] + dl[2] * dl[2]
        t = -(ol[0] * dl[0] + ol[1] * dl[1] + ol[2] * dl[2]) / aa
        D2 = sum((ol[j] + t * dl[j]).square() for j in range(3))
        ok = (D2 <= self.kap[at].square()) & (t > tn[:, None]) & (t <= tf[:, None]) & (self.size[at] > 0)
        t = torch.where(ok, t, torch.full_like(t, math.inf))
        H = max(1, int(ok.sum(1).amax()))
        t, j = torch.topk(t, H, dim=1, largest=False, sorted=True)
        al = (self.o[at][j] * torch.exp(-0.5 * torch.gather(D2, 1, j))).clamp(max=ALPHA_MAX)
        real = torch.isfinite(t)
        T = torch.cumprod(1 - torch.where(real, al, torch.zeros_like(al)), 1)
        real = real & (torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1) >= T_MIN)
        H = max(1, int(real.sum(1).amax()))
        return at[j[:, :H]], real[:, :H]

    def shade(self, g, o, d, ids, real):
        """(C + T bg, T) of the rays from their blend lists; differentiable in g."""
        mu, ls, q, lo, sh = g
        n = d
        if self.at is not None:
            w = self.inv[self.at[ids]]
            M = self.maps[self.at[ids]]
            oo = (w @ (o[:, None, :] - M[..., 3])[..., None])[..., 0]
            d = n = (w @ d[:, None, :, None])[..., 0]
            n = torch.nn.functional.normalize(n, dim=-1)
        else:
            oo, d, n = o[:, None, :], d[:, None, :], torch.nn.functional.normalize(n, dim=-1)[:, None, :]
        W = torch.exp(-ls[ids])[..., None] * _rot(q[ids]).transpose(-1, -2)
        ol, dl = (W @ (oo - mu[ids])[..., None])[..., 0], (W @ d[..., None])[..., 0]
        t = -(ol * dl).sum(-1) / dl.square().sum(-1)
        al = torch.sigmoid(lo[ids]) * torch.exp(-0.5 * (ol + t[..., None] * dl).square().sum(-1))
        al = torch.where(real, al.clamp(max=ALPHA_MAX), torch.zeros_like(al))
        T = torch.cumprod(1 - al, 1)
        w = al * torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1)
        c = (torch.einsum("...k,...kc->...c", _basis(n, self.sh).expand(*ids.shape, -1), sh[ids]) + 0.5).clamp(min=0.0)
        bg = torch.tensor(np.asarray(BG, np.float32).astype(np.float64), device="cuda")
        return torch.cat([(w[..., None] * c).sum(1) + T[:, -1:] * bg, T[:, -1:]], 1)


def _chunks(cam, count, n, side=32):
    """Groups of ray indices: square tiles of a camera, or as many rays as all Gaussians fit with."""
    if cam is None:
        step = max(1, 60_000_000 // n)
        return [torch.arange(a, min(a + step, count), device="cuda") for a in range(0, count, step)]
    W, H = cam["width"], cam["height"]
    i = torch.arange(W * H, device="cuda").reshape(H, W)
    return [i[y:y + side, x:x + side].reshape(-1) for y in range(0, H, side) for x in range(0, W, side)]


def _exact_image(F, o, d, tn, tf, cam, upstream=None):
    """The image, and with `upstream` the gradients of its inner product with it."""
    out = torch.empty((o.shape[0], 4), dtype=torch.float64, device="cuda")
    grads = [torch.zeros_like(t) for t in F.g] if upstream is not None else None
    every = (F.size > 0).nonzero()[:, 0]
    for c in _chunks(cam, o.shape[0], max(1, every.numel())):
        at = F.near(o[c], d[c]) if cam is not None else every
        if not at.numel():
            out[c] = torch.tensor(np.asarray(BG + (1.0,), np.float32).astype(np.float64), device="cuda")
            continue
        small = max(1, 60_000_000 // at.numel())
        for b in c.split(small):
            ids, real = F.hits(o[b], d[b], tn[b], tf[b], at)
            for p in range(0, b.numel(), 1024):
                q = b[p:p + 1024]
                if upstream is None:
                    out[q] = F.shade(F.g, o[q], d[q], ids[p:p + 1024], real[p:p + 1024])
                    continue
                used, local = torch.unique(ids[p:p + 1024], return_inverse=True)
                g = [t[used].requires_grad_(True) for t in F.g]
                img = F.shade(g, o[q], d[q], local, real[p:p + 1024])
                out[q] = img.detach()
                for G, x in zip(grads, torch.autograd.grad(img, g, upstream[q])):
                    G[used] += x
    return out, grads


def _limits(n):
    return torch.zeros(n, dtype=torch.float64, device="cuda"), torch.full((n,), math.inf, dtype=torch.float64, device="cuda")


def exact(case, seed):
    kind = case["kind"]
    if kind == "build":
        return None                              # a tree has no such values
    g = _gaussians(case["scene"], case["n"], case["sh"], seed)
    if kind == "serve":
        with torch.no_grad():
            F = [_Field(g, case["sh"]), _Field(_gaussians(case["scene"], 2 * case["n"], case["sh"], seed + 1), case["sh"])]
            return [_exact_image(F[i], *_camera_rays64(cam), *_limits(cam["width"] * cam["height"]), cam)[0]
                    for i, cam in _requests(case, seed)]
    with torch.no_grad():
        if kind == "world":
            two = [g, _gaussians(case["scene"], 2 * case["n"], case["sh"], seed + 1)]
            pl = _placements(case, seed)
            at = torch.cat([torch.full((two[i][3].numel(),), j, dtype=torch.long, device="cuda")
                            for j, (i, _) in enumerate(pl)])
            F = _Field([torch.cat([two[i][k] for i, _ in pl]) for k in range(5)], case["sh"], at,
                       torch.tensor(np.stack([M for _, M in pl]), device="cuda"))
            cam = scenes.pinhole_camera(case["width"], case["height"], (0.0, 3.0, -9.0), (0.0, 0.0, 0.0), 60.0)
        else:
            F = _Field(g, case["sh"])
            cam = None if kind == "rays" else _camera(case, seed)
    if kind == "rays":
        o, d, tn, tf = (t.double() for t in _scattered_rays(case, g, seed))
    elif kind == "bounce":                       # the bounce rays have no common origin: too many pairs
        o, d, tn, tf = (t.double() for t in _bounce_rays(cam)[0])
        with torch.no_grad():
            return [_exact_image(F, o, d, tn, tf, cam)[0], None]
    else:
        (o, d), (tn, tf) = _camera_rays64(cam), _limits(case["width"] * case["height"])
    if kind != "train":
        with torch.no_grad():
            return _exact_image(F, o, d, tn, tf, cam)[0]
    up = _Draw(seed + 5).n(0.0, 1.0, case["width"] * case["height"], 4).double()
    img, grads = _exact_image(F, o, d, tn, tf, cam, up)
    return [img, *grads]

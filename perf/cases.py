"""What is timed when the traversal library is made faster.

Every case is one pass of work that a program using this library has it do,
through its public entry points (paper_1912_12786_gb300.vsr and .autograd).
The scenes are the repository's workloads -- random alpha-masked quads in the
unit cube, the billboard forest, the displaced sphere -- made on the GPU from
a seed, with sizes from a handful of picking rays to a 1080p frame over a
million triangles.

  listed()           the cases
  draw(rng)          one more case of the same ranges
  prepare(c, seed)   scene, BVH, rays, buffers and the plans a program keeps
  run(state)         one pass; its outputs
  work(c)            bytes and operations no implementation can do without
  exact(c, seed)     the outputs in 64 bits, where that is feasible

Hit records come back as their t, u, v and, apart, the primitive ids, since a
record's fourth word holds an integer.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1912_12786_gb300 import autograd as A
from paper_1912_12786_gb300 import vsr as V
from paper_1912_12786_gb300.inputs import _lib as L
from paper_1912_12786_gb300.inputs import scenes as S

DEV = "cuda"
INF = float("inf")


def listed():
    return [
        # A tool's picking or line-of-sight queries: a few hundred rays at a
        # time against a small scene, where a call's latency is all there is.
        {"name": "picks", "op": "trace", "scene": "quads", "tris": 4096, "rays": "camera",
         "n": 777, "isect": "default", "query": "closest", "dispatch": "static"},
        # A preview frame with an alpha mask: the repository's small workload.
        {"name": "preview_frame", "op": "frame", "scene": "quads", "tris": 4096, "w": 256,
         "h": 256, "isect": "alpha_tex", "query": "closest", "dispatch": "static"},
        # The main workload: a 1080p frame of the forest, primary visibility
        # through the foliage textures and one shadow ray per pixel, at the
        # configuration tuned for the scene.
        {"name": "forest_frame", "op": "lit", "scene": "forest", "tris": 1_000_002, "w": 1920,
         "h": 1080, "isect": "alpha_tex"},
        # The heat map of traversal costs over an oddly sized frame.
        {"name": "heat_map", "op": "frame", "scene": "forest", "tris": 200_002, "w": 1283,
         "h": 719, "isect": "count", "query": "closest", "dispatch": "static"},
        # Incoherent closest hit: rays leaving surfaces, as a light baker or
        # an acoustic simulation traces them, in no particular order.
        {"name": "diffuse_closest", "op": "tuned", "scene": "quads", "tris": 200_000,
         "rays": "diffuse", "n": 1_000_003, "isect": "alpha_tex", "query": "closest"},
        # Short incoherent any-hit rays: ambient occlusion over a large scene
        # with the procedural mask.
        {"name": "occlusion_any", "op": "tuned", "scene": "quads", "tris": 2_000_000,
         "rays": "ao", "n": 1_200_000, "isect": "proc_alpha", "query": "any"},
        # Many small scenes of uneven size in one launch (a training set of
        # scenes, or the tiles of a distributed render).
        {"name": "batch_any", "op": "batch", "scenes": 40, "tris": 60_000, "n": 400_000,
         "isect": "alpha_tex", "query": "any"},
        # The first eight hits along every camera ray: order-independent
        # transparency.
        {"name": "multi_hit", "op": "multi", "scene": "forest", "tris": 200_002, "w": 640,
         "h": 360, "hits": 8, "isect": "alpha_tex"},
        # One mesh placed many times under a top-level BVH.
        {"name": "instances", "op": "instances", "tris": 15_624, "copies": 64, "w": 960,
         "h": 540, "isect": "alpha_tex", "query": "closest"},
        # Diffuse path tracing, three bounces.
        {"name": "path_trace", "op": "path", "scene": "forest", "tris": 200_002, "w": 960,
         "h": 540, "bounces": 3, "isect": "alpha_tex"},
        # One step of inverse rendering: vertices and texels pushed into the
        # scene, rendered, and the image's gradient taken back to both.
        {"name": "inverse_render", "op": "train", "freq": 57, "w": 512, "h": 512, "tex": 512},
        # The same for an ambient-occlusion render and its texels.
        {"name": "occlusion_render", "op": "train_ao", "scene": "quads", "tris": 200_000,
         "w": 480, "h": 270, "spp": 4, "tex": 512},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["trace", "frame", "frame", "lit", "tuned", "tuned", "batch", "multi",
                     "instances", "path", "train", "train_ao"])
    isect = rng.choice(["default", "alpha_tex", "proc_alpha"])
    scene = rng.choice(["quads", "forest"])
    tris = 2 * _log_int(rng, 500, 250_000)
    w, h = _log_int(rng, 64, 1500), _log_int(rng, 64, 800)
    query = rng.choice(["closest", "any"])
    if op == "trace":
        return {"op": op, "scene": scene, "tris": tris, "rays": "camera",
                "n": _log_int(rng, 33, 100_000), "isect": isect, "query": query,
                "dispatch": "static"}
    if op == "frame":
        kind = rng.choice([isect, isect, "count"])
        return {"op": op, "scene": scene, "tris": tris, "w": w, "h": h, "isect": kind,
                "query": query, "dispatch": rng.choice(["static", "static", "dynamic"])}
    if op == "lit":
        return {"op": op, "scene": scene, "tris": tris, "w": w, "h": h, "isect": isect}
    if op == "tuned":
        return {"op": op, "scene": "quads", "tris": tris, "rays": rng.choice(["diffuse", "ao"]),
                "n": _log_int(rng, 20_000, 1_000_000), "isect": isect, "query": query}
    if op == "batch":
        return {"op": op, "scenes": rng.randint(3, 40), "tris": _log_int(rng, 2_000, 60_000),
                "n": _log_int(rng, 5_000, 300_000), "isect": isect, "query": query}
    w, h = _log_int(rng, 50, 800), _log_int(rng, 50, 500)
    if op == "multi":
        return {"op": op, "scene": scene, "tris": tris, "w": w, "h": h,
                "hits": rng.randint(1, 16), "isect": isect}
    if op == "instances":
        return {"op": op, "tris": 2 * _log_int(rng, 200, 8_000), "copies": rng.randint(2, 64),
                "w": w, "h": h, "isect": isect, "query": query}
    if op == "path":
        return {"op": op, "scene": scene, "tris": tris, "w": w, "h": h,
                "bounces": rng.randint(1, 4), "isect": isect}
    if op == "train":
        return {"op": op, "freq": rng.randint(6, 60), "w": _log_int(rng, 50, 512),
                "h": _log_int(rng, 50, 512), "tex": rng.choice([64, 200, 512])}
    return {"op": op, "scene": "quads", "tris": tris, "w": w // 2, "h": h // 2,
            "spp": rng.randint(1, 8), "tex": rng.choice([64, 200, 512])}


# ---------------------------------------------------------------------------
# geometry, textures and rays, on the GPU from a generator


def _gen(seed, salt):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 1_000_003 + salt)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _noise(g, size, base, octaves):
    """Smooth noise in [0, 1], float64 [size, size]."""
    out = torch.zeros(size, size, device=DEV, dtype=torch.float64)
    amp = total = 0.0
    for o in range(octaves):
        amp = 0.5 ** o
        lat = _rand(g, 1, 1, base * 2 ** o + 1, base * 2 ** o + 1)
        out += amp * torch.nn.functional.interpolate(lat, (size, size), mode="bicubic",
                                                     align_corners=True)[0, 0]
        total += amp
    return (out / total).clamp_(0.0, 1.0)


def _foliage(g, size):
    """RGBA8 with alpha 255 on about 45% of the texels."""
    n = _noise(g, size, 16, 4)
    thr = torch.quantile(n[::4, ::4].reshape(-1), 0.55)
    col = _noise(g, size, 16, 3)
    tex = torch.stack([30 + 70 * col, 90 + 150 * col, 20 + 50 * col,
                       torch.where(n > thr, 255.0, 0.0)], -1)
    return S.Texture("rgba8", size, size, tex.clamp(0, 255).to(torch.uint8).cpu().numpy())


def _float_texture(g, size, alpha):
    """RGBA32F: smooth colour; alpha from uniform noise, or 1."""
    tex = torch.stack([_noise(g, size, 8, 3) for _ in range(3)]
                      + [_rand(g, size, size) if alpha == "noise"
                         else torch.ones(size, size, device=DEV, dtype=torch.float64)], -1)
    return tex.to(torch.float32)


def _quad_soup(corners):
    """corners [q, 4, 3] float64 -> verts [4q, 3], idx [2q, 3], uvs [2q, 3, 2]."""
    q = corners.shape[0]
    base = 4 * torch.arange(q, device=DEV)[:, None, None]
    idx = (base + torch.tensor([[0, 1, 2], [0, 2, 3]], device=DEV)).reshape(-1, 3)
    uv = torch.tensor([[[0, 0], [1, 0], [1, 1]], [[0, 0], [1, 1], [0, 1]]], device=DEV,
                      dtype=torch.float32).repeat(q, 1, 1)
    return corners.reshape(-1, 3).to(torch.float32), idx, uv


def _quads(g, tris):
    """Randomly turned squares in the unit cube; their side shrinks with
    their number so that a ray meets about as many of them at every size."""
    q = max(1, tris // 2)
    side = (0.02 + 0.08 * _rand(g, q)) * math.sqrt(4096.0 / max(tris, 4096))
    x = torch.randn(q, 4, generator=g, device=DEV, dtype=torch.float64)
    w, x, y, z = (x / x.norm(dim=1, keepdim=True)).unbind(1)
    a = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y + z * w), 2 * (x * z - y * w)], 1)
    b = torch.stack([2 * (x * y - z * w), 1 - 2 * (x * x + z * z), 2 * (y * z + x * w)], 1)
    c = _rand(g, q, 3)
    a, b = 0.5 * side[:, None] * a, 0.5 * side[:, None] * b
    return torch.stack([c - a - b, c + a - b, c + a + b, c - a + b], 1)


def _billboards(g, q, extent):
    """Upright billboards on a jittered grid over extent x extent."""
    m = math.ceil(math.sqrt(q))
    cell = torch.randperm(m * m, generator=g, device=DEV)[:q]
    px = (cell % m + _rand(g, q)) * (extent / m)
    pz = (cell // m + _rand(g, q)) * (extent / m)
    h = 0.5 + 2.5 * _rand(g, q)
    wd = h * (0.5 + 0.5 * _rand(g, q))
    yaw = 2 * math.pi * _rand(g, q)
    o = torch.zeros_like(px)
    base = torch.stack([px, o, pz], 1)
    ax = 0.5 * wd[:, None] * torch.stack([yaw.cos(), o, yaw.sin()], 1)
    up = torch.stack([o, h, o], 1)
    return torch.stack([base - ax, base + ax, base + ax + up, base - ax + up], 1)


def _ground(extent):
    e = float(extent)
    return torch.tensor([[[0, 0, 0], [e, 0, 0], [e, 0, e], [0, 0, e]]], device=DEV,
                        dtype=torch.float64)


def _geometry(c, seed):
    """(verts, idx, uvs, geom, textures, extent) of the case's scene."""
    g = _gen(seed, 1)
    if c["scene"] == "forest":
        # the forest's density: half a million billboards on 100 x 100
        q = max(1, (c["tris"] - 2) // 2)
        extent = 100.0 * math.sqrt(q / 500_000)
        v, i, uv = _quad_soup(torch.cat([_ground(extent), _billboards(g, q, extent)]))
        geom = (torch.arange(len(i), device=DEV) // 2 - 1) % 4
        geom[:2] = S.NONE
        return v, i, uv, geom, [_foliage(g, 1024) for _ in range(4)], extent
    v, i, uv = _quad_soup(_quads(g, c["tris"]))
    geom = torch.zeros(len(i), device=DEV, dtype=torch.int64)
    if c["op"] == "train_ao":
        t = _float_texture(g, c["tex"], "one").cpu().numpy()
        tex = S.Texture("rgba32f", c["tex"], c["tex"], t)
    else:
        tex = S.disc_alpha_u8(256, 0.4)
    return v, i, uv, geom, [tex], 1.0


def _upload(v, i, uv, geom, textures):
    verts, idx = v.cpu().numpy(), i.to(torch.int32).cpu().numpy().view(np.uint32)
    s = V.vsr_scene_create_indexed(verts, idx, uv.cpu().numpy(),
                                   (geom & 0xFFFFFFFF).cpu().numpy().astype(np.uint32), textures)
    V.vsr_bvh_load(s, L.bvh_build(verts, idx))
    return s


def _rays(o, d, tmin, tmax):
    r = torch.empty(d.shape[0], 8, device=DEV, dtype=torch.float32)
    r[:, 0:3] = o.to(torch.float32)
    r[:, 3] = tmin
    r[:, 4:7] = (d / d.norm(dim=1, keepdim=True)).to(torch.float32)
    r[:, 7] = tmax
    return r


def _camera(eye, target, sx, sy, fovy=60.0):
    """Directions through image-plane points (sx, sy), |sy| <= 1."""
    eye = torch.tensor(eye, device=DEV, dtype=torch.float64)
    f = torch.tensor(target, device=DEV, dtype=torch.float64) - eye
    f = f / f.norm()
    r = torch.linalg.cross(torch.tensor([0.0, 1.0, 0.0], device=DEV, dtype=torch.float64), f)
    r = r / r.norm()
    u = torch.linalg.cross(f, r)
    th = math.tan(math.radians(fovy) / 2)
    return eye, f[None] + th * (sx[:, None] * r[None] + sy[:, None] * u[None])


def _view(c, extent, g):
    """The scene's camera, moved a little by the seed."""
    j = (_rand(g, 3) - 0.5).tolist()
    if c.get("scene") == "forest" or c["op"] == "instances":
        return ((0.5 + 0.02 * j[0]) * extent, 1.7 + 0.2 * j[1], -2.0 + 0.2 * j[2]), \
            (0.5 * extent, 1.0, 0.5 * extent)
    return (0.5 + 0.1 * j[0], 0.5 + 0.1 * j[1], -1.0 + 0.1 * j[2]), (0.5, 0.5, 0.5)


def _frame_rays(c, view, fovy=60.0):
    w, h = c["w"], c["h"]
    x = (2 * (torch.arange(w, device=DEV, dtype=torch.float64) + 0.5) / w - 1) * (w / h)
    y = 1 - 2 * (torch.arange(h, device=DEV, dtype=torch.float64) + 0.5) / h
    eye, d = _camera(view[0], view[1], x.repeat(h), y.repeat_interleave(w), fovy)
    return _rays(eye, d, 0.0, INF)


def _cosine_dirs(g, n):
    """Cosine-distributed unit vectors about +z."""
    x1, x2 = _rand(g, n), _rand(g, n)
    r = x1.sqrt()
    return torch.stack([r * (2 * math.pi * x2).cos(), r * (2 * math.pi * x2).sin(),
                        (1 - x1).sqrt()], 1)


def _surface_rays(g, v, i, n, tmin, tmax):
    """Rays leaving random points of random triangles, cosine-distributed."""
    t = v.double()[i[torch.randint(len(i), (n,), generator=g, device=DEV)]]
    a, b = _rand(g, n, 1).sqrt(), _rand(g, n, 1)
    e1, e2 = t[:, 1] - t[:, 0], t[:, 2] - t[:, 0]
    p = t[:, 0] + a * (1 - b) * e1 + a * b * e2
    nrm = torch.linalg.cross(e1, e2)
    nrm = nrm / nrm.norm(dim=1, keepdim=True)
    t1 = e1 / e1.norm(dim=1, keepdim=True)
    t2 = torch.linalg.cross(nrm, t1)
    m = _cosine_dirs(g, n)
    sign = torch.where(_rand(g, n, 1) < 0.5, -1.0, 1.0)
    return _rays(p, m[:, :1] * t1 + m[:, 1:2] * t2 + sign * m[:, 2:] * nrm, tmin, tmax)


def _sphere(freq, g):
    """Displaced sphere with about 20 freq^2 triangles: a latitude-longitude
    grid, smooth noise along the normal, texture coordinates over the square."""
    nv, nu = 2 * freq + 2, 5 * freq
    j = torch.arange(nv + 1, device=DEV, dtype=torch.float64)
    k = torch.arange(nu + 1, device=DEV, dtype=torch.float64)
    th = (j / nv * (math.pi - 0.02) + 0.01)[:, None]
    ph = (k / nu * 2 * math.pi)[None]
    p = torch.stack([th.sin() * ph.cos(), th.cos().expand(-1, nu + 1), th.sin() * ph.sin()], -1)
    d = _noise(g, 256, 8, 3)[(j / nv * 255).long()][:, ((k % nu) / nu * 255).long()]
    verts = (p * (1 + 0.15 * (d - 0.5))[..., None]).reshape(-1, 3).float()
    a = (j[:-1, None].long() * (nu + 1) + k[None, :-1].long()).reshape(-1)
    idx = torch.stack([torch.stack([a, a + 1, a + nu + 2], 1),
                       torch.stack([a, a + nu + 2, a + nu + 1], 1)], 1).reshape(-1, 3)
    uv = torch.stack([(k / nu)[None].expand(nv + 1, -1), (j / nv)[:, None].expand(-1, nu + 1)],
                     -1).reshape(-1, 2).float()[idx]
    return verts, idx, uv


# ---------------------------------------------------------------------------


class _State:
    """The scenes, tensors and plans of one case."""


def _buffers(s, n, per=1):
    s.hits = torch.empty(n * per, 4, device=DEV, dtype=torch.float32)


def prepare(c, seed):
    s = _State()
    s.c = c
    op = c["op"]
    g = _gen(seed, 2)
    if op == "batch":
        return _prepare_batch(s, c, seed)
    if op == "instances":
        return _prepare_instances(s, c, seed, g)
    if op == "train":
        return _prepare_train(s, c, seed, g)
    v, i, uv, geom, tex, extent = _geometry(c, seed)
    s.eps = 1e-4 * float((v.amax(0) - v.amin(0)).double().norm())
    s.scene = _upload(v, i, uv, geom, tex)
    s.isect = V.intersector(c.get("isect", "proc_alpha"), c.get("dispatch", "static"))
    if op == "trace":
        eye, d = _camera(*_view(c, extent, g), 2 * _rand(g, c["n"]) - 1, 2 * _rand(g, c["n"]) - 1)
        s.rays = _rays(eye, d, 0.0, INF)
        s.params = V.trace_params()
    elif op == "tuned":
        s.rays = _surface_rays(g, v, i, c["n"], s.eps, 0.05 if c["rays"] == "ao" else INF)
    else:
        s.rays = _frame_rays(c, _view(c, extent, g))
        s.params = V.trace_params(image_width=c["w"])
    n = s.rays.shape[0]
    _buffers(s, n, c.get("hits", 1))
    if op == "frame" and c["isect"] == "count":
        s.counts = torch.empty(n, 2, device=DEV, dtype=torch.int32)
    elif op == "tuned":
        V.vsr_trace_tune(s.scene, s.rays, s.isect, c["query"], s.hits)
    elif op == "lit":
        # the program tunes both queries once for the scene
        s.light = S.light_dir_f32()
        s.shadow = torch.empty_like(s.rays)
        s.hits2 = torch.empty_like(s.hits)
        V.vsr_trace_tune(s.scene, s.rays, s.isect, "closest", s.hits, c["w"])
        V.vsr_trace(s.scene, s.rays, s.isect, "closest", s.hits)
        V.vsr_make_shadow_rays(s.rays, s.hits, s.light, s.eps, s.shadow)
        V.vsr_trace_tune(s.scene, s.shadow, s.isect, "any", s.hits2, c["w"])
    elif op == "path":
        s.path = V.path_params(bounces=c["bounces"], eps=s.eps)
        s.dirs = _cosine_dirs(g, n * c["bounces"]).float()
        s.radiance = torch.empty(n, 3, device=DEV, dtype=torch.float32)
        s.segments = torch.empty(n, device=DEV, dtype=torch.int32)
    elif op == "train_ao":
        s.shade = V.shade_params((0.0, 1.0, 0.0), (0.2, 0.3, 0.4), 0)
        s.tex = _float_texture(g, c["tex"], "one").requires_grad_()
        s.xi = _rand(g, n * c["spp"], 2).float().clamp_(max=1 - 2.0 ** -24)
        s.target = _rand(g, n, 3).float()
    return s


def _prepare_batch(s, c, seed):
    s.scenes, s.rays = [], []
    m = c["scenes"]
    for k in range(m):
        # sizes spread over two decades, small and large ones interleaved
        f = 100.0 ** -((k * 7 % m) / max(m - 1, 1))
        f2 = 100.0 ** -((k * 11 % m) / max(m - 1, 1))
        tris, n = 2 * max(32, int(c["tris"] * f / 2)), max(97, int(c["n"] * f2))
        cc = {"op": "batch", "scene": "quads", "tris": tris}
        v, i, uv, geom, tex, extent = _geometry(cc, seed * 64 + k)
        s.scenes.append(_upload(v, i, uv, geom, tex))
        g = _gen(seed * 64 + k, 3)
        h = n // 2
        eye, d = _camera(*_view(cc, extent, g), 2 * _rand(g, h) - 1, 2 * _rand(g, h) - 1)
        s.rays.append(torch.cat([_rays(eye, d, 0.0, INF),
                                 _surface_rays(g, v, i, n - h, 1e-4, INF)]))
    s.hits = [torch.empty(r.shape[0], 4, device=DEV, dtype=torch.float32) for r in s.rays]
    s.batch = V.vsr_batch_create(s.scenes, s.rays, s.hits, V.intersector(c["isect"]), c["query"])
    V.vsr_batch_launch(s.batch)  # a program's warm-up: chooses the launch configuration
    return s


def _prepare_instances(s, c, seed, g):
    q, m = max(1, c["tris"] // 2), c["copies"]
    grid = math.ceil(math.sqrt(m))
    cell = 100.0 * math.sqrt(q / 500_000)
    extent = cell * grid
    v, i, uv = _quad_soup(_billboards(g, q, cell))
    geom = torch.arange(len(i), device=DEV) // 2 % 4
    tile = _upload(v, i, uv, geom, [_foliage(g, 1024) for _ in range(4)])
    gv, gi, guv = _quad_soup(_ground(extent))
    s.meshes = [tile, _upload(gv, gi, guv, torch.full((2,), S.NONE, device=DEV), [])]
    lo, hi = v.amin(0).double().cpu().numpy(), v.amax(0).double().cpu().numpy()
    box = np.array([[x, y, z] for x in (lo[0], hi[0]) for y in (lo[1], hi[1])
                    for z in (lo[2], hi[2])])
    yaw = (2 * math.pi * _rand(g, m)).cpu().numpy()
    w2o = [np.eye(4)[:3]]
    boxes = [[0.0, -1e-3, 0.0, extent, 1e-3, extent]]
    for k in range(m):
        cs, sn = math.cos(yaw[k]), math.sin(yaw[k])
        rot = np.array([[cs, 0, sn], [0, 1, 0], [-sn, 0, cs]])
        centre = np.array([(k % grid + 0.5) * cell, 0.0, (k // grid + 0.5) * cell])
        mid = np.array([0.5 * cell, 0.0, 0.5 * cell])
        w2o.append(np.concatenate([rot.T, (mid - rot.T @ centre)[:, None]], 1))
        wb = (box - mid) @ rot.T + centre
        boxes.append([*(wb.min(0) - 1e-3), *(wb.max(0) + 1e-3)])
    s.inst = V.vsr_instances_create(s.meshes, np.array([1] + [0] * m, np.uint32),
                                    np.array(w2o, np.float32).reshape(-1, 12),
                                    L.bvh_build_boxes(np.array(boxes, np.float32)))
    s.isect = V.intersector(c["isect"])
    s.rays = _frame_rays(c, _view(c, extent, g))
    s.params = V.trace_params(image_width=c["w"])
    n = s.rays.shape[0]
    _buffers(s, n)
    s.ids = torch.empty(n, device=DEV, dtype=torch.int32)
    return s


CUT = 0.3  # alpha cutoff of the inverse-rendering texture


def _train_inputs(c, seed, g):
    v, i, uv = _sphere(c["freq"], _gen(seed, 1))
    tex = _float_texture(g, c["tex"], "noise")
    rays = _frame_rays(c, ((0.1, 0.2, 3.0), (0.0, 0.0, 0.0)), 45.0)
    target = _rand(g, rays.shape[0], 3).float()
    return v, i, uv, tex, rays, target


LIGHT, BACK = (0.48, 0.6, 0.64), (0.2, 0.3, 0.4)


def _prepare_train(s, c, seed, g):
    v, i, uv, tex, s.rays, s.target = _train_inputs(c, seed, g)
    s.scene = _upload(v, i, uv, torch.zeros(len(i), device=DEV, dtype=torch.int64),
                      [S.Texture("rgba32f", c["tex"], c["tex"], tex.cpu().numpy())])
    s.verts, s.tex = v.clone().requires_grad_(), tex.clone().requires_grad_()
    s.isect = V.intersector("alpha_tex", cutoff_f=CUT)
    s.shade = V.shade_params(LIGHT, BACK, 0)
    return s


def _out(hits):
    return {"tuv": hits[:, :3], "prim": hits.view(torch.int32)[:, 3]}


def run(s):
    c = s.c
    op = c["op"]
    if op in ("trace", "frame"):
        counts = getattr(s, "counts", None)
        V.vsr_trace(s.scene, s.rays, s.isect, c["query"], s.hits, counts, s.params)
        return {**_out(s.hits), "counts": counts}
    if op == "tuned":
        V.vsr_trace(s.scene, s.rays, s.isect, c["query"], s.hits)
        return _out(s.hits)
    if op == "lit":
        V.vsr_trace(s.scene, s.rays, s.isect, "closest", s.hits)
        V.vsr_make_shadow_rays(s.rays, s.hits, s.light, s.eps, s.shadow)
        V.vsr_trace(s.scene, s.shadow, s.isect, "any", s.hits2)
        return {"primary": _out(s.hits), "rays": s.shadow, "shadow": _out(s.hits2)}
    if op == "batch":
        V.vsr_batch_launch(s.batch)
        return [h.view(torch.int32) for h in s.hits]
    if op == "multi":
        V.vsr_trace_multi(s.scene, s.rays, s.isect, c["hits"], s.hits, None, s.params)
        return _out(s.hits)
    if op == "instances":
        V.vsr_trace_instances(s.inst, s.rays, s.isect, c["query"], s.hits, s.ids, None, s.params)
        return {**_out(s.hits), "instance": s.ids}
    if op == "path":
        V.vsr_path_trace(s.scene, s.rays, s.isect, s.path, s.dirs, s.radiance, s.segments,
                         s.params)
        return {"radiance": s.radiance, "segments": s.segments}
    if op == "train":
        image = A.render(s.scene, s.rays, s.verts, s.tex, s.isect, s.shade)
        gv, gt = torch.autograd.grad(image, (s.verts, s.tex), image.detach() - s.target)
        return {"image": image.detach(), "verts": gv, "texels": gt}
    image = A.render_ao(s.scene, s.rays, s.tex, s.isect, c["spp"], s.xi, 0.2, s.eps, s.shade)
    gt, = torch.autograd.grad(image, s.tex, image.detach() - s.target)
    return {"image": image.detach(), "texels": gt}


# ---------------------------------------------------------------------------


def work(c):
    """Rays in, records out, and one triangle's corners and texture
    coordinates (60 bytes) per distinct triangle that a ray could end on; one
    descent of a binary tree (two slab tests of 12 operations per level) and
    one triangle test (45) per ray."""
    op = c["op"]
    if op == "batch":
        m = c["scenes"]
        n = sum(max(97, int(c["n"] * 100.0 ** -((k * 11 % m) / max(m - 1, 1)))) for k in range(m))
        tris = sum(c["tris"] * 100.0 ** -((k * 7 % m) / max(m - 1, 1)) for k in range(m))
        depth = math.log2(max(c["tris"] / 10, 2))
    else:
        tris = 20 * c["freq"] ** 2 if op == "train" else c["tris"]
        n = c["n"] if "n" in c else c["w"] * c["h"]
        depth = math.log2(max(tris, 2))
    per_ray = depth * 24 + 45
    geo = 60 * min(tris, n)
    if op == "lit":
        return {"bytes": n * (32 + 16 + 32 + 16) + geo, "flops": 2 * n * per_ray}
    if op == "multi":
        return {"bytes": n * (32 + 16 * c["hits"]) + geo, "flops": n * c["hits"] * per_ray}
    if op == "path":
        return {"bytes": n * (32 + 12 * c["bounces"] + 16) + geo,
                "flops": n * (1 + c["bounces"] / 2) * per_ray}
    if op == "train":
        # vertices and texels in, image out; upstream gradient in, both
        # gradients out
        return {"bytes": n * (32 + 12 + 12) + 2 * (6 * tris + 16 * c["tex"] ** 2) + geo,
                "flops": n * (per_ray + 300)}
    if op == "train_ao":
        return {"bytes": n * (32 + 8 * c["spp"] + 12 + 12) + 2 * 16 * c["tex"] ** 2 + geo,
                "flops": n * (1 + c["spp"]) * per_ray}
    extra = 8 if c.get("isect") == "count" else 4 if op == "instances" else 0
    return {"bytes": n * (32 + 16 + extra) + geo, "flops": n * per_ray}


# ---------------------------------------------------------------------------
# 64-bit results by brute force, where the scene is small enough


def _lerp(uv, u, v):
    return (1 - u - v)[:, None] * uv[:, 0] + u[:, None] * uv[:, 1] + v[:, None] * uv[:, 2]


def _brute(rays, v, i, accept):
    """Closest accepted hit of every ray over all triangles: (prim or -1, t,
    u, v).  accept(ray index, triangle, u, v) -> bool per candidate."""
    tri = v.double()[i]
    a, e1, e2 = tri[:, 0], tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]
    n, m = rays.shape[0], len(i)
    best = torch.full((n,), INF, device=DEV, dtype=torch.float64)
    prim = torch.full((n,), -1, device=DEV, dtype=torch.int64)
    bu, bv = torch.zeros_like(best), torch.zeros_like(best)
    nrm = torch.linalg.cross(e1, e2)
    step = max(1, 60_000_000 // m)
    for k in range(0, n, step):
        o, d = rays[k:k + step, 0:3].double(), rays[k:k + step, 4:7].double()
        # n . d, n . (o - a), and u, v from (d x (o - a)) . e2 and . e1
        dxo = torch.linalg.cross(d, o)
        exa1, exa2 = torch.linalg.cross(a, e1), torch.linalg.cross(a, e2)
        det = -(d @ nrm.T)
        # (o - a) x d . e = o x d . e - a x d . e = -(dxo . e) - d . (e x a)
        u = (-(dxo @ e2.T) + d @ exa2.T) / det
        w = (dxo @ e1.T - d @ exa1.T) / det
        r, p = torch.nonzero((u >= 0) & (w >= 0) & (u + w <= 1), as_tuple=True)
        uu, ww = u[r, p], w[r, p]
        t = ((o[r] - a[p]) * nrm[p]).sum(1) / det[r, p]
        ok = (t > rays[k + r, 3].double()) & (t < rays[k + r, 7].double())
        r, p, t, uu, ww = r[ok], p[ok], t[ok], uu[ok], ww[ok]
        ok = accept(p, uu, ww)
        r, p, t, uu, ww = r[ok], p[ok], t[ok], uu[ok], ww[ok]
        by_t = torch.argsort(t)
        by = by_t[torch.argsort(r[by_t], stable=True)]
        first = torch.ones(len(by), dtype=torch.bool, device=DEV)
        first[1:] = r[by][1:] != r[by][:-1]
        sel = by[first]
        best[k + r[sel]], prim[k + r[sel]] = t[sel], p[sel]
        bu[k + r[sel]], bv[k + r[sel]] = uu[sel], ww[sel]
    return prim, best, bu, bv


def _nearest(size, uv):
    k = (uv.clamp(0, 1) * size).floor().long().clamp(max=size - 1)
    return k[:, 1] * size + k[:, 0]


def exact(c, seed):
    op = c["op"]
    if op == "train" and c["freq"] <= 60:
        return _exact_train(c, seed)
    n = c["n"] if "n" in c else c.get("w", 0) * c.get("h", 0)
    if op in ("trace", "frame") and c["query"] == "closest" and c["isect"] != "proc_alpha" \
            and c["scene"] == "quads" and n * c["tris"] <= 2_000_000_000:
        g = _gen(seed, 2)
        v, i, uv, _, tex, extent = _geometry(c, seed)
        if op == "trace":
            eye, d = _camera(*_view(c, extent, g), 2 * _rand(g, c["n"]) - 1,
                             2 * _rand(g, c["n"]) - 1)
            rays = _rays(eye, d, 0.0, INF)
        else:
            rays = _frame_rays(c, _view(c, extent, g))
        mask = torch.from_numpy(tex[0].texels.reshape(-1).astype(np.int64)).to(DEV)

        def accept(p, u, w):
            if c["isect"] != "alpha_tex":
                return torch.ones_like(p, dtype=torch.bool)
            return mask[_nearest(256, _lerp(uv.double()[p], u, w))] >= 128

        _, t, u, w = _brute(rays, v, i, accept)
        return {"tuv": torch.stack([t, u, w], 1), "prim": None, "counts": None}
    return None


def _exact_train(c, seed):
    """Image and gradients in 64 bits at the visibility that 64 bits give."""
    v, i, uv, tex, rays, target = _train_inputs(c, seed, _gen(seed, 2))
    size = c["tex"]
    alpha = tex[..., 3].reshape(-1)
    cut = torch.tensor(CUT, dtype=torch.float32).item()
    uv = uv.double()
    prim, _, _, _ = _brute(rays, v, i,
                           lambda p, u, w: alpha[_nearest(size, _lerp(uv[p], u, w))] >= cut)
    verts, texels = v.double().requires_grad_(), tex.double().requires_grad_()
    hit = torch.nonzero(prim >= 0)[:, 0]
    o, d = rays[hit, 0:3].double(), rays[hit, 4:7].double()
    tri = verts[i[prim[hit]]]
    a, e1, e2 = tri[:, 0], tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]
    m = torch.stack([-d, e1, e2], 2)
    sol = torch.linalg.solve(m, (o - a)[..., None])[..., 0]
    xy = _lerp(uv[prim[hit]], sol[:, 1], sol[:, 2]) * size - 0.5
    f0 = xy.detach().floor()
    f = xy - f0
    k0, k1 = f0.long().clamp(0, size - 1), (f0.long() + 1).clamp(0, size - 1)
    rgb = texels[..., :3]
    fx, fy = f[:, :1], f[:, 1:]
    alb = (1 - fy) * ((1 - fx) * rgb[k0[:, 1], k0[:, 0]] + fx * rgb[k0[:, 1], k1[:, 0]]) \
        + fy * ((1 - fx) * rgb[k1[:, 1], k0[:, 0]] + fx * rgb[k1[:, 1], k1[:, 0]])
    nrm = torch.linalg.cross(e1, e2)
    nrm = nrm / nrm.norm(dim=1, keepdim=True)
    face = torch.where((nrm.detach() * d).sum(1) < 0, 1.0, -1.0)
    light = torch.tensor(LIGHT, dtype=torch.float32).double().to(DEV)
    lit = (face * (nrm @ light)).clamp(min=0)
    back = torch.tensor(BACK, dtype=torch.float32).double().to(DEV)
    image = back.expand(rays.shape[0], 3).index_put((hit,), alb * lit[:, None])
    gv, gt = torch.autograd.grad(image, (verts, texels), image.detach() - target.double())
    return {"image": image.detach(), "verts": gv, "texels": gt}

"""The octant kernels, which most launches of one ray per thread take, against
the generic kernel (reg_cap_blocks 1; test_gpu_routes.py shows that it is
another one) and, where boxes are not finite, against every triangle tested.
Either side gives every record and count exactly, so the tolerance is zero."""
import numpy as np
import pytest

from kernel_names import kernels_of
from oracle import oracle as O
from paper_1912_12786_gb300.inputs import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CLIP = dict(clip_lo=(-1.0, -1.0, -1.0), clip_hi=(50.0, 1.5, 101.0))


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_12786_gb300 import _build, vsr
    _build.build()
    return vsr


@pytest.fixture(scope="module")
def forest(V):
    sc, rays = scenes.billboard_forest()
    s = V.scene_from_inputs(sc, sc.bvh())
    d = torch.from_numpy(rays).cuda()
    hits = torch.empty(d.shape[0], 4, device="cuda")
    V.vsr_trace(s, d, V.intersector("alpha_tex"), "closest", hits, None,
                V.trace_params(reg_cap_blocks=1, image_width=1920))
    shadow = torch.empty_like(d)
    V.vsr_make_shadow_rays(d, hits, scenes.light_dir_f32(), scenes.shadow_eps(sc), shadow)
    torch.cuda.synchronize()
    yield s, d, shadow
    s.close()


def _both(V, s, rays, kind, query, **kw):
    """(records, counts) of the generic kernel and of `kw`'s launches."""
    n = rays.shape[0]
    out = []
    isect = V.intersector(kind, **(CLIP if kind == "clip" else {}))
    width = kw.get("image_width", 0)
    for p in (V.trace_params(reg_cap_blocks=1, image_width=width),
              V.trace_params(**kw), V.trace_params(octant=1, **kw)):
        h = torch.full((n, 4), 7.0, device="cuda")
        c = torch.zeros(n, 2, dtype=torch.int32, device="cuda") if kind == "count" else None
        V.vsr_trace(s, rays, isect, query, h, c, p)
        out.append((h.view(torch.int32), c))
    torch.cuda.synchronize()
    return out


def _same(out, label):
    for h, c in out[1:]:
        bad = (h != out[0][0]).any(1)
        assert not bad.any(), f"{label}: {int(bad.sum())} rays differ"
        assert c is None or torch.equal(c, out[0][1]), label


@pytest.mark.parametrize("width", [1920, 0])
@pytest.mark.parametrize("kind", ["none", "default", "alpha_tex", "proc_alpha", "count", "clip"])
def test_forest_frame(V, forest, kind, width):
    """Every record and count of a 1080p frame's primary and shadow rays, both
    queries, on pixel tiles and in rows."""
    s, d, shadow = forest
    for name, rays in (("primary", d), ("shadow", shadow)):
        for query in ("closest", "any"):
            _same(_both(V, s, rays, kind, query, image_width=width),
                  f"{name}/{kind}/{query}/{width}")
    assert V.vsr_get_device_error(s) == 0


def test_after_refits(V):
    """Moved vertices, NaN vertices (boxes inverted: the octant kernels fall
    back) and back; with NaN also against all triangles tested one by one,
    which a NaN vertex never lets hit."""
    sc, rays = scenes.small_quads(seed=scenes.SEED_BASE + 46)
    s = V.scene_from_inputs(sc, sc.bvh())
    d = torch.from_numpy(rays).cuda()
    moved = sc.verts + np.random.default_rng(3).normal(0, 0.01, sc.verts.shape).astype(np.float32)
    bad = moved.copy()
    bad[sc.idx[:300].ravel()] = np.nan
    bad[sc.idx[300:340, 1]] = np.nan  # triangles with a single such vertex
    sel = np.sort(np.random.default_rng(4).choice(len(rays), 4000, replace=False))
    for label, verts in (("moved", moved), ("nan", bad), ("back", sc.verts)):
        V.vsr_scene_update(s, torch.from_numpy(np.ascontiguousarray(verts)).cuda())
        ref = scenes.Scene(sc.name, verts, sc.idx, sc.uvs, sc.geom_id, sc.textures)
        for kind in ("default", "alpha_tex", "count"):
            found = {}
            for query in ("closest", "any"):
                out = _both(V, s, d, kind, query, image_width=256)
                _same(out, f"{label}/{kind}/{query}")
                found[query] = out[0][0]
            miss = [f[:, 3] == -1 for f in found.values()]
            assert torch.equal(miss[0], miss[1])
            want, st = O.trace_list(ref, rays[sel], "alpha_tex" if kind == "alpha_tex" else
                                    "default", "closest")
            got = found["closest"].cpu().numpy()[sel].view(np.uint32)
            differ = np.any(got != O.hits_raw(want).view(np.uint32), axis=1) & (st[:, 3] == 0)
            assert not differ.any(), f"{label}/{kind}: {int(differ.sum())} of 4000"
    assert V.vsr_get_device_error(s) == 0
    s.close()


def test_render_and_path(V):
    """Images, adjoints and radiance that rest on the octant kernels' hits."""
    sc, rays = scenes.small_quads()
    s = V.scene_from_inputs(sc, sc.bvh())
    d = torch.from_numpy(rays).cuda()
    n = len(rays)
    shade = V.shade_params(scenes.light_dir_f32())
    dirs = torch.from_numpy(scenes.path_dirs(n, 3)).cuda()
    out = []
    for kw in (dict(reg_cap_blocks=1), dict(), dict(octant=1)):
        p = V.trace_params(image_width=256, **kw)
        img, rad = (torch.empty(n, 3, device="cuda") for _ in range(2))
        hits = torch.empty(n, 4, device="cuda")
        V.vsr_render(s, d, V.intersector("alpha_tex"), shade, img, hits, p)
        V.vsr_path_trace(s, d, V.intersector("alpha_tex"), V.path_params(3), dirs, rad, None, p)
        out.append([x.view(torch.int32) for x in (img, hits, rad)])
    torch.cuda.synchronize()
    for o in out[1:]:
        for a, b in zip(out[0], o):
            assert torch.equal(a, b)
    names = kernels_of(lambda st: V.vsr_path_trace(s, d, V.intersector("alpha_tex"),
                                                   V.path_params(3), dirs, rad, None,
                                                   V.trace_params(reg_cap_blocks=1), st))
    assert names == ["k_trace", "k_path_bounce"] * 4
    s.close()

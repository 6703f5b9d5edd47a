"""The single-scene kernels over the two-level node records (k_trace_wide,
k_trace_wide_persistent) on a tree with long descents, the only kind they are
launched on, against the generic kernel (reg_cap_blocks 1), bit for bit: edge
rays, scales and offsets at which the 16-bit grid changes, leaf sizes, refits,
ragged sizes.  Each launch is shown to be the kernel that is meant."""
import numpy as np
import pytest

from kernel_names import kernels_of
from paper_1912_12786_gb300.inputs import scenes
from test_gpu_records import _rays

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

QUADS = 60_000
SHAPES = [dict(block_size=96, lockstep=1), dict(block_size=256, lockstep=1),
          dict(block_size=64, lockstep=1, persistent=1, refill_threshold=24),
          dict(block_size=32, lockstep=1, persistent=1, refill_threshold=1),
          dict(block_size=64, lockstep=1, ray_order=1), dict()]


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_12786_gb300 import _build, vsr
    _build.build()
    return vsr


def _scene(name):
    rng = np.random.default_rng(QUADS)
    side = 0.08 * (2048 / QUADS) ** 0.5
    v, i, uv = scenes._quads_to_tris(scenes.random_quads(rng, QUADS, 0, 1, 0.2 * side, side))
    v = {"quads": v, "tiny": v * np.float32(1e-9), "huge": v * np.float32(1e9),
         "out_of_range": v * np.float32(1e12), "far": v + np.float32(64.0),
         "flat": v * np.float32([1, 1e-6, 1])}[name].astype(np.float32)
    return scenes.Scene(name, v, i, uv, np.zeros(len(i), np.uint32), [scenes.disc_alpha_u8()])


def _descents(blob):
    """Expected visits of a ray that crosses the root box, and inner nodes per
    leaf, from the boxes' surface areas: what records_limit decides on."""
    n = int(blob[16:20].view(np.uint32)[0])
    nodes = blob[64:64 + 32 * n].reshape(n, 32)
    lo, hi = (np.ascontiguousarray(nodes[:, k:k + 12]).view(np.float32).astype(np.float64)
              for k in (0, 16))
    leaf = np.ascontiguousarray(nodes[:, 28:32]).view(np.uint32)[:, 0] >= 4
    e = hi - lo
    area = e[:, 0] * e[:, 1] + e[:, 1] * e[:, 2] + e[:, 2] * e[:, 0]
    used = np.arange(n) != 1
    inner = area[used & ~leaf].sum()
    return inner / area[0], inner / area[used & leaf].sum()


def _expected(kw):
    if kw.get("ray_order"):
        return "k_trace_wide"  # after the sort's kernels
    return "k_trace_wide_persistent" if kw.get("persistent") else "k_trace_wide"


def _check(V, s, d, kind, query, label, shapes=SHAPES):
    n = d.shape[0]
    isect = V.intersector(kind)
    want = torch.full((n, 4), 7.0, device="cuda")
    V.vsr_trace(s, d, isect, query, want, None, V.trace_params(reg_cap_blocks=1))
    for kw in shapes:
        got = torch.full((n, 4), 7.0, device="cuda")
        p = V.trace_params(watchdog_ms=10_000, **kw)
        V.vsr_trace(s, d, isect, query, got, None, p)
        torch.cuda.synchronize()
        bad = (got.view(torch.int32) != want.view(torch.int32)).any(1)
        assert not bad.any(), f"{label}/{kind}/{query} {kw}: {int(bad.sum())} of {n} rays differ"
    assert V.vsr_get_device_error(s) == 0, label
    return want


@pytest.mark.parametrize("name", ["quads", "tiny", "huge", "out_of_range", "far", "flat"])
@pytest.mark.parametrize("leaf_max", [1, 4, 8])
def test_scenes_and_edge_rays(V, name, leaf_max):
    sc = _scene(name)
    blob = sc.bvh(leaf_max=leaf_max)
    if name != "flat":
        visits, per_leaf = _descents(blob)
        assert visits > 1.2 * 90 and per_leaf > 1.2 * 12, (visits, per_leaf)
    s = V.scene_from_inputs(sc, blob)
    d = torch.from_numpy(_rays(sc)).cuda()
    for kind in ("none", "default", "alpha_tex", "proc_alpha"):
        for query in ("closest", "any"):
            want = _check(V, s, d, kind, query, f"{name}/{leaf_max}")
    if name == "quads":
        assert int((V.prim_ids(want) != 0xFFFFFFFF).sum()) > 2000
    if name not in ("flat", "out_of_range"):  # the latter's boxes need the binary nodes
        for kw in SHAPES:
            names = kernels_of(lambda st: V.vsr_trace(
                s, d, V.intersector("alpha_tex"), "closest", want, None, V.trace_params(**kw), st))
            assert names[-1] == _expected(kw), (kw, names)
    s.close()


def test_refits(V):
    """Moved, out of the grid's range and NaN (both: the binary kernels), a single
    NaN vertex, and back."""
    sc = _scene("quads")
    s = V.scene_from_inputs(sc, sc.bvh())
    rays = torch.from_numpy(_rays(sc)).cuda()
    base = torch.from_numpy(sc.verts).cuda()
    some, one = base.clone(), base.clone()
    some[torch.from_numpy(sc.idx[:400].astype(np.int64).ravel()).cuda()] = float("nan")
    one[7] = float("nan")
    far = rays.clone()
    far[:, 0:3] = far[:, 0:3] * 0.3 + 9.0
    for label, v, d in (("moved", 0.3 * base + 9.0, far), ("range", base * 1e12, rays * 1e12),
                        ("nan", some, rays), ("one", one, rays), ("back", base, rays)):
        V.vsr_scene_update(s, v)
        for kind in ("default", "alpha_tex"):
            for query in ("closest", "any"):
                want = _check(V, s, d.contiguous(), kind, query, label)
        assert int((V.prim_ids(want) != 0xFFFFFFFF).sum()) > 500, label
    s.close()


@pytest.mark.parametrize("n", [1, 31, 33, 4097])
def test_ragged(V, n):
    sc = _scene("quads")
    s = V.scene_from_inputs(sc, sc.bvh())
    d = torch.from_numpy(_rays(sc)[:n].copy()).cuda()
    for query in ("closest", "any"):
        _check(V, s, d, "alpha_tex", query, f"n={n}")
    s.close()

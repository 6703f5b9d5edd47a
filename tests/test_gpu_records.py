"""Lock-step launches over the two-level node records (one ray per thread,
persistent, batched) against the per-lane binary traversal, bit for bit, where
the records' 16-bit boxes, the leaf check or the way back to the binary nodes
could go wrong: planes and edges shared exactly, boxes without extent, trees of
one to a few nodes, leaf sizes 1 and 8, scales and offsets, edge-case rays,
refits, and refits that leave boxes non-finite.  The hits are single records
that either side must give exactly, so the tolerance is zero.
"""
import numpy as np
import pytest

from paper_1912_12786_gb300.inputs import scenes

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_12786_gb300 import _build, vsr
    _build.build()
    return vsr


def _grid(cells):
    """A flat axis-aligned grid at y = 0: every edge is shared exactly."""
    k = np.arange(cells + 1, dtype=np.float64)
    x, z = np.meshgrid(k, k, indexing="ij")
    v = np.stack([x, np.zeros_like(x), z], -1).reshape(-1, 3)
    i = (np.arange(cells)[:, None] * (cells + 1) + np.arange(cells)).reshape(-1)
    idx = np.stack([np.stack([i, i + 1, i + cells + 2], 1),
                    np.stack([i, i + cells + 2, i + cells + 1], 1)], 1).reshape(-1, 3)
    uv = v[idx][:, :, [0, 2]] / cells
    return scenes.Scene("grid", v.astype(np.float32), idx.astype(np.uint32),
                        uv.astype(np.float32), np.zeros(len(idx), np.uint32),
                        [scenes.disc_alpha_u8(64, 0.45)])


def _scene(name):
    if name == "grid":
        return _grid(24)
    sc, _ = scenes.small_quads(n_quads=600, res=8)
    if name.startswith("first"):
        sc.idx, sc.uvs, sc.geom_id = (a[:int(name[5:])] for a in (sc.idx, sc.uvs, sc.geom_id))
    elif name == "tiny":
        sc.verts = (sc.verts * np.float32(1e-9)).astype(np.float32)
    elif name == "huge":
        sc.verts = (sc.verts * np.float32(1e9)).astype(np.float32)
    elif name == "out_of_range":
        sc.verts = (sc.verts * np.float32(1e12)).astype(np.float32)
    elif name == "far":
        sc.verts = (sc.verts + np.float32(4096.0)).astype(np.float32)
    return sc


def _rays(sc, n=6000, seed=3):
    """Rays through vertices, edge midpoints and random points from points in
    and around the scene, axis-parallel ones, and edge cases."""
    rng = np.random.default_rng(seed)
    v = sc.verts.astype(np.float64)
    lo, hi = v.min(0), v.max(0)
    ext = max(float((hi - lo).max()), 1e-30)
    tri = v[sc.idx[rng.integers(0, sc.ntri, n)]]
    w = rng.dirichlet([1, 1, 1], n)
    w[: n // 3] = np.eye(3)[rng.integers(0, 3, n // 3)]
    w[n // 3: n // 2] = np.roll([0.5, 0.5, 0.0], 1)
    to = np.einsum("nk,nkc->nc", w, tri)
    o = lo + (rng.uniform(-1, 2, (n, 3))) * ext
    o[::7] = to[::7] + np.array([0, 1.0, 0]) * ext
    o[3::7] = to[3::7] + np.array([1.0, 0, 0]) * ext
    o = np.round(o / ext * 64) / 64 * ext if sc.name == "grid" else o
    d = (to - o) * rng.choice([1.0, 1.0, 1e-3, 1e3], (n, 1))
    r = np.zeros((n, 8), np.float32)
    with np.errstate(over="ignore"):
        r[:, :3], r[:, 4:7] = o, d
    r[:, 3] = rng.choice([0.0, 0.0, -1.0, 1e-4], n)
    r[:, 7] = rng.choice([np.inf, np.inf, 1.0, 0.5, -1.0], n)
    inf, nan, c = np.inf, np.nan, 0.5 * (lo + hi)
    odd = [[*c, 0, 0, 0, 0, inf], [*c, 0, nan, 0, 1, inf], [nan, 0, 0, 0, 0, 1, 0, inf],
           [*c, 0, inf, 0, 0, inf], [*c, 0, 1e38, 1e-38, 1, inf], [*c, 0, 1e-30, -1e-30, 1, inf],
           [*c, nan, 0, 1, 0, inf], [*c, 0, 0, 1, 0, nan], [inf, 0, 0, 0, -1, 0, 0, inf],
           [1e30, 0, 0, 0, -1, 0, 0, inf], [*c, 0, -0.0, 0.0, 1, inf], [*c, 0, 1e25, 1e25, 1, inf]]
    r[5: 5 + 11 * len(odd): 11] = np.array(odd, np.float32)
    return r


def _same(V, s, d, kind, query, label):
    n = d.shape[0]
    out = [torch.full((n, 4), 7.0, device="cuda") for _ in range(4)]
    isect = V.intersector(kind)
    V.vsr_trace(s, d, isect, query, out[0], None, V.trace_params(block_size=64))
    V.vsr_trace(s, d, isect, query, out[1], None, V.trace_params(block_size=96, lockstep=1))
    V.vsr_trace(s, d, isect, query, out[2], None,
                V.trace_params(block_size=64, lockstep=1, persistent=1, refill_threshold=24))
    # a batch walks the records of any tree; the launches above those of trees
    # with long descents
    b = V.vsr_batch_create([s], [d], [out[3]], isect, query,
                           V.trace_params(block_size=64, lockstep=1))
    V.vsr_batch_launch(b)
    torch.cuda.synchronize()
    V.vsr_batch_destroy(b)
    assert V.vsr_get_device_error(s) == 0, label
    want = out[0].view(torch.int32)
    for k, h in enumerate(out[1:]):
        bad = (h.view(torch.int32) != want).any(1)
        assert not bad.any(), f"{label}, shape {k}: {int(bad.sum())} of {n} rays differ"


@pytest.mark.parametrize("name", ["grid", "quads", "first1", "first2", "first9", "tiny", "huge",
                                  "out_of_range", "far"])
@pytest.mark.parametrize("leaf_max", [1, 4, 8])
def test_records_match_binary(V, name, leaf_max):
    sc = _scene(name)
    s = V.scene_from_inputs(sc, sc.bvh(leaf_max=leaf_max))
    d = torch.from_numpy(_rays(sc)).cuda()
    for kind in ("default", "alpha_tex", "proc_alpha"):
        for query in ("closest", "any"):
            _same(V, s, d, kind, query, f"{name}/{leaf_max}/{kind}/{query}")
    s.close()


def test_records_after_refit_and_in_a_batch(V):
    """After vertex updates (moved, scaled out of the grid's range, non-finite
    and back) the records, or the binary nodes in their place, give the
    per-lane results; so does a batch made before the updates."""
    sc = _scene("quads")
    s = V.scene_from_inputs(sc, sc.bvh())
    d = torch.from_numpy(_rays(sc)).cuda()
    hits = torch.empty(d.shape[0], 4, device="cuda")
    ref = torch.empty_like(hits)
    isect = V.intersector("alpha_tex")
    b = V.vsr_batch_create([s], [d], [hits], isect, "closest",
                           V.trace_params(block_size=64, lockstep=1))
    base = torch.from_numpy(sc.verts).cuda()
    bad = base.clone()
    bad[sc.idx[:40].astype(np.int64).ravel()] = float("nan")
    for label, v in (("moved", 0.3 * base + 0.2), ("nan", bad), ("back", base)):
        V.vsr_scene_update(s, v)
        for query in ("closest", "any"):
            _same(V, s, d, "alpha_tex", query, label)
        V.vsr_trace(s, d, isect, "closest", ref, None, V.trace_params())
        V.vsr_batch_launch(b)
        torch.cuda.synchronize()
        assert torch.equal(hits.view(torch.int32), ref.view(torch.int32)), label
    V.vsr_scene_update(s, base * 1e12)
    _same(V, s, d * 1e12, "alpha_tex", "closest", "out of range")
    V.vsr_batch_destroy(b)
    s.close()


@pytest.mark.parametrize("n_quads,n", [(25_000, 5000), (25_000, 700_001), (400, 5000)])
def test_open_launches_match_binary(V, n_quads, n):
    """Launches that leave the traversal's form open, on a tree with long
    descents below and above the ray count at which they walk the records, and
    on a shallow one: the records of the measurement kernel, which walks the
    binary nodes."""
    rng = np.random.default_rng(n_quads)
    side = 0.08 * (2048 / n_quads) ** 0.5
    v, i, uv = scenes._quads_to_tris(scenes.random_quads(rng, n_quads, 0, 1, 0.2 * side, side))
    sc = scenes.Scene("quads", v, i, uv, np.zeros(len(i), np.uint32), [scenes.disc_alpha_u8()])
    s = V.scene_from_inputs(sc, sc.bvh())
    d = torch.from_numpy(scenes.diffuse_rays(rng, sc, n)).cuda()
    stats = torch.empty(n, 4, device="cuda", dtype=torch.int32)
    for kind in ("default", "alpha_tex", "proc_alpha"):
        for query in ("closest", "any"):
            want = torch.empty(n, 4, device="cuda")
            got = torch.full_like(want, 7.0)
            V.vsr_trace_stats(s, d, V.intersector(kind), query, want, stats)
            V.vsr_trace(s, d, V.intersector(kind), query, got, None, V.trace_params())
            assert torch.equal(got.view(torch.int32), want.view(torch.int32)), (kind, query)
            _same(V, s, d, kind, query, f"{n_quads}/{kind}/{query}")
    assert V.vsr_get_device_error(s) == 0
    s.close()

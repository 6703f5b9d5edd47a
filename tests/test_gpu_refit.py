"""The refit after a vertex update (one launch, threads climbing from the
leaves) against a scene loaded with the boxes recomputed on the host: hits and
per-ray box and triangle counts, which depend on every box, are identical.
Trees of one node to a deep, unbalanced one; two updates in a row."""
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


def _refit_blob(blob, verts, idx):
    """The blob with every box recomputed from the vertices."""
    out = blob.copy()
    n = int(out[16:20].view(np.uint32)[0])
    nodes = out[64:64 + 32 * n].view(np.uint32).reshape(n, 8)
    order = out[64 + 32 * n:].view(np.uint32)
    box = nodes.view(np.float32)
    for i in range(n - 1, -1, -1):  # children follow their parent
        if i == 1:
            continue
        count, left = int(nodes[i, 7]) >> 2, int(nodes[i, 3])
        if count:
            p = verts[idx[order[left:left + count]].reshape(-1)]
            lo, hi = p.min(0), p.max(0)
        else:
            lo = np.minimum(box[left, 0:3], box[left + 1, 0:3])
            hi = np.maximum(box[left, 4:7], box[left + 1, 4:7])
        box[i, 0:3], box[i, 4:7] = lo, hi
    h = 1469598103934665603
    for b in out[64:].tobytes():
        h = ((h ^ b) * 1099511628211) & 0xFFFFFFFFFFFFFFFF
    out[48:56].view(np.uint64)[0] = h
    return out


@pytest.mark.parametrize("tris", [1, 4, 5, 9, 33, 1200])
def test_refit_matches_host(V, tris):
    sc, rays = scenes.small_quads(n_quads=(tris + 1) // 2, res=96)
    sc.idx, sc.uvs, sc.geom_id = sc.idx[:tris], sc.uvs[:tris], sc.geom_id[:tris]
    if tris > 9:  # a dense corner makes the tree uneven
        sc.verts[:tris] *= np.float32(1e-3)
    blob = sc.bvh()
    s = V.scene_from_inputs(sc, blob)
    d = torch.from_numpy(rays).cuda()
    n = d.shape[0]
    rng = np.random.default_rng(tris)
    for scale in (0.3, 0.02):
        moved = sc.verts + rng.normal(0, scale, sc.verts.shape).astype(np.float32)
        V.vsr_scene_update(s, torch.from_numpy(moved).cuda())
        ref = scenes.Scene(sc.name, moved, sc.idx, sc.uvs, sc.geom_id, sc.textures)
        f = V.scene_from_inputs(ref, _refit_blob(blob, moved, sc.idx))
        for query in ("closest", "any"):
            got = []
            for scene in (s, f):
                h = torch.empty(n, 4, device="cuda")
                c = torch.empty(n, 4, device="cuda", dtype=torch.int32)
                V.vsr_trace_stats(scene, d, V.intersector("alpha_tex"), query, h, c)
                got.append((h.view(torch.int32), c))
            assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
        assert V.vsr_get_device_error(s) == 0
        f.close()
    s.close()

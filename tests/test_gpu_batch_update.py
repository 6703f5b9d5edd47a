"""Batches made before their scenes change: vertex updates that take the
geometry out of the box it had give the records of vsr_trace on the updated
scene."""
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


def _scene(V, k, n_quads=600):
    sc, rays = scenes.small_quads(n_quads=n_quads, res=64, seed=scenes.SEED_BASE + k)
    return sc, V.scene_from_inputs(sc, sc.bvh()), torch.from_numpy(rays).cuda()


@pytest.mark.parametrize("query", ["closest", "any"])
@pytest.mark.parametrize("shape", [dict(lockstep=1), dict(lockstep=1, stack_regs=2),
                                   dict(lockstep=0), dict(lockstep=1, ray_order=1)],
                         ids=["records", "lockstep", "lanes", "ordered"])
def test_batch_made_before_an_update(V, shape, query):
    made = [_scene(V, 80 + k) for k in range(3)]
    ss, rr = [m[1] for m in made], [m[2] for m in made]
    hits = [torch.empty(r.shape[0], 4, device="cuda") for r in rr]
    isect = V.intersector("alpha_tex")
    b = V.vsr_batch_create(ss, rr, hits, isect, query,
                           V.trace_params(block_size=64, persistent=1, refill_threshold=24,
                                          watchdog_ms=10_000, **shape))
    V.vsr_batch_launch(b)
    seen = 0
    for shift, scale in ((5.0, 1.0), (0.0, 1e12), (0.0, 1.0)):
        # scene 1 keeps its vertices throughout
        for k in (0, 2):
            base = torch.from_numpy(made[k][0].verts).cuda()
            V.vsr_scene_update(ss[k], (base + shift) * scale)
            r = torch.from_numpy(scenes.small_quads(n_quads=600, res=64)[1]).cuda()
            r[:, 0:3] = (r[:, 0:3] + shift) * scale
            rr[k].copy_(r)
        V.vsr_batch_launch(b)
        torch.cuda.synchronize()
        for k in range(3):
            want = torch.empty_like(hits[k])
            V.vsr_trace(ss[k], rr[k], isect, query, want, None, V.trace_params())
            torch.cuda.synchronize()
            assert torch.equal(hits[k].view(torch.int32), want.view(torch.int32)), (shift, scale, k)
            seen += int((V.prim_ids(want) != 0xFFFFFFFF).sum())
            assert V.vsr_get_device_error(ss[k]) == 0
    assert seen > 1000  # the updated scenes are hit
    V.vsr_batch_destroy(b)
    for s in ss:
        s.close()


def test_launch_refused_once_a_scene_is_gone(V):
    """A batch over a scene that was destroyed, or that was given another BVH,
    is refused before anything runs; a batch made anew works."""
    made = [_scene(V, 90 + k) for k in range(2)]
    ss, rr = [m[1] for m in made], [m[2] for m in made]
    hits = [torch.empty(r.shape[0], 4, device="cuda") for r in rr]
    isect = V.intersector("default")
    p = V.trace_params(block_size=64, persistent=1, lockstep=1, watchdog_ms=10_000)
    old = V.vsr_batch_create(ss, rr, hits, isect, "closest", p)
    never = V.vsr_batch_create(ss, rr, hits, isect, "closest", p)
    V.vsr_batch_launch(old)
    torch.cuda.synchronize()
    want = [h.clone() for h in hits]
    V.vsr_bvh_load(ss[0], made[0][0].bvh(leaf_max=2))
    for b in (old, never):
        with pytest.raises(V.VsrError, match="scene 0 .*another BVH"):
            V.vsr_batch_launch(b)
    new = V.vsr_batch_create(ss, rr, hits, isect, "closest", p)
    other = V.scene_from_inputs(made[0][0], made[0][0].bvh())
    other.close()  # another scene's end does not matter
    for h in hits:
        h.zero_()
    V.vsr_batch_launch(new)
    torch.cuda.synchronize()
    for h, w in zip(hits, want):
        assert torch.equal(h.view(torch.int32), w.view(torch.int32))
    ss[1].close()
    with pytest.raises(V.VsrError, match="scene 1 .*destroyed"):
        V.vsr_batch_launch(new)
    for b in (old, never, new):
        V.vsr_batch_destroy(b)
    ss[0].close()


def test_one_call_form_tells_scenes_at_one_address_apart(V):
    """vsr_trace_batch with a scene made where a destroyed one was, and with a
    scene that got another BVH, the buffers the same: the new scene's records."""
    hits = torch.empty(64 * 64, 4, device="cuda")
    isect = V.intersector("alpha_tex")
    p = V.trace_params(block_size=64, persistent=1, lockstep=1, watchdog_ms=10_000)
    d = _scene(V, 0)[2]
    seen, again = set(), 0
    for k in range(12):
        sc, s, _ = _scene(V, 100 + k)
        again += s.handle in seen
        seen.add(s.handle)
        for leaf_max in (4, 1):
            V.vsr_bvh_load(s, sc.bvh(leaf_max=leaf_max))
            want = torch.empty_like(hits)
            V.vsr_trace(s, d, isect, "closest", want, None, V.trace_params())
            V.vsr_trace_batch([s], [d], [hits], isect, "closest", p)
            torch.cuda.synchronize()
            assert torch.equal(hits.view(torch.int32), want.view(torch.int32)), (k, leaf_max)
        s.close()
    assert again  # an address came back

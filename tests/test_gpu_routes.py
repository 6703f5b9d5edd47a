"""Which kernel a launch is routed to.  Every route gives the same result, so
the choices that a caller makes through the launch parameters show only here."""
import numpy as np
import pytest

from kernel_names import kernels_of
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


def _quads(n_quads):
    rng = np.random.default_rng(n_quads)
    side = 0.08 * (2048 / n_quads) ** 0.5
    v, i, uv = scenes._quads_to_tris(scenes.random_quads(rng, n_quads, 0, 1, 0.2 * side, side))
    return scenes.Scene("quads", v, i, uv, np.zeros(len(i), np.uint32), [scenes.disc_alpha_u8()])


@pytest.fixture(scope="module", params=[2048, 100_000], ids=["short", "long"])
def made(V, request):
    """A tree with short and one with long descents, on which open launches
    walk the two-level records."""
    sc = _quads(request.param)
    s = V.scene_from_inputs(sc, sc.bvh())
    rays = scenes.pinhole_rays((0.5, 0.5, -1.0), (0.5, 0.5, 0.5), (0, 1, 0), 60.0, 320, 200)
    yield request.param > 10_000, s, torch.from_numpy(rays).cuda()
    s.close()


def _trace(V, made, query, **kw):
    _, s, d = made
    hits = torch.empty(d.shape[0], 4, device="cuda")
    return kernels_of(lambda st: V.vsr_trace(s, d, V.intersector("alpha_tex"), query, hits, None,
                                             V.trace_params(**kw), st))


@pytest.mark.parametrize("width", [0, 320])
@pytest.mark.parametrize("query", ["closest", "any"])
def test_no_register_budget_is_the_generic_kernel(V, made, query, width):
    assert _trace(V, made, query, image_width=width, reg_cap_blocks=1) == ["k_trace"]
    assert _trace(V, made, query, image_width=width, octant=1) == ["k_trace_oct"]
    assert _trace(V, made, query, image_width=width, octant=1, reg_cap_blocks=1) == \
        ["k_trace_oct"]
    assert _trace(V, made, query, image_width=width) != ["k_trace"] or \
        (query, width) == ("any", 0)


def test_clip_box_closest_hit(V):
    """The generic kernel in buffer order, where its rays are faster, the octant
    kernel on tiles and for few rays."""
    sc, rays = scenes.small_quads(res=320)
    s = V.scene_from_inputs(sc, sc.bvh())
    d = torch.from_numpy(rays).cuda()
    hits = torch.empty(len(rays), 4, device="cuda")
    isect = V.intersector("clip", clip_lo=(0.2, 0.1, 0.0), clip_hi=(0.8, 0.7, 0.9))
    out = []
    for n, width, kernel in ((len(rays), 0, "k_trace"), (len(rays), 320, "k_trace_oct"),
                             (2000, 0, "k_trace_oct")):
        p = V.trace_params(image_width=width)
        names = kernels_of(lambda st: V.vsr_trace(s, d[:n], isect, "closest", hits[:n], None, p,
                                                  st))
        assert names == [kernel]
        V.vsr_trace(s, d[:n], isect, "closest", hits[:n], None, p)
        torch.cuda.synchronize()
        out.append(hits[:n].clone().view(torch.int32))
    assert torch.equal(out[0], out[1]) and torch.equal(out[0][:2000], out[2])
    s.close()


def test_record_kernels_only_where_the_records_hold(V, made):
    """After updates that leave boxes non-finite or the grid too coarse, lock
    step takes the binary kernels, and the record kernels again after the next."""
    long, s, d = made
    sc = _quads(100_000 if long else 2048)
    base = torch.from_numpy(sc.verts).cuda()
    nan = base.clone()
    nan[5] = float("nan")
    bad = nan.clone()
    bad[torch.from_numpy(sc.idx[:200].astype(np.int64).ravel()).cuda()] = float("nan")
    shapes = (dict(lockstep=1), dict(lockstep=1, persistent=1), dict())
    wide = ["k_trace_wide", "k_trace_wide_persistent", "k_trace_wide"]
    binary = ["k_trace_ls", "k_trace_persistent", "k_trace_oct"]
    for verts, holds in ((base, True), (bad, False), (base * 1e12, False), (nan, True),
                         (base, True)):
        V.vsr_scene_update(s, verts.contiguous())
        got = [_trace(V, made, "closest", **kw)[-1] for kw in shapes]
        assert got == (wide if holds and long else binary)

"""One-ray-per-thread multi-hit launches in lock step (needs a GB300).

The lock-step form visits each ray's nodes and leaves in the order of the
per-lane loops, so hits and counters equal those of the persistent per-lane
kernel bit for bit.  Launches with fewer than eight rays per warp keep the
per-lane form; the sizes lie on both sides of that line, with ragged tiles and
a last warp that is nearly empty.
"""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def V():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_12786_gb300 import _build, vsr
    _build.build()
    return vsr


@pytest.fixture(scope="module")
def scene(V):
    from paper_1912_12786_gb300.inputs import scenes
    sc, _ = scenes.small_quads()
    s = V.scene_from_inputs(sc, sc.bvh())
    yield sc, s
    s.close()


def _rays(sc, n):
    g = torch.Generator().manual_seed(n)
    v = torch.as_tensor(sc.verts).reshape(-1, 3)
    lo, hi = v.min(0).values, v.max(0).values
    o = lo + (hi - lo) * (torch.rand(n, 3, generator=g) * 2 - 0.5)
    d = torch.randn(n, 3, generator=g)
    d[::7] = d[::7] * torch.tensor([1.0, 0.0, 0.0])  # zero components
    r = torch.cat([o, torch.zeros(n, 1), d, torch.full((n, 1), 1e30)], 1)
    return r.float().contiguous().cuda()


def line(warps):
    """Rays from which on a warp of the one-ray-per-thread launch takes eight,
    spread over `warps` warps per SM (14 in buffer order, 36 on pixel tiles)."""
    return warps * torch.cuda.get_device_properties(0).multi_processor_count * 4


@pytest.mark.parametrize("kind", ["none", "default", "alpha_tex", "proc_alpha", "count"])
@pytest.mark.parametrize("nh", [1, 16])
def test_lockstep_equals_per_lane(V, scene, kind, nh):
    sc, s = scene
    i = V.intersector(kind)
    n0, n1 = line(14), line(36)
    for n, width in ((1, 0), (33, 0), (n0, 0), (n0 + 1, 0), (n0 + 31, 0), (n1, 64),
                     (n1 + 1, 64), (301 * 203, 301), (301 * 203 - 5, 301)):
        rays = _rays(sc, n)
        out = []
        for persistent in (0, 1):
            hits = torch.full((n, nh, 4), -1.0, device="cuda")
            cnt = torch.full((n, 2), -1, device="cuda", dtype=torch.int32)
            V.vsr_trace_multi(s, rays, i, nh, hits, cnt if kind == "count" else None,
                              V.trace_params(persistent=persistent, image_width=width))
            out.append((hits.view(torch.int32), cnt))
        assert torch.equal(out[0][0], out[1][0]), (n, width)
        assert torch.equal(out[0][1], out[1][1]), (n, width)

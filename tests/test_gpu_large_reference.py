"""The 16 M-triangle frame: every primary record of the octant kernel and of
lock step against the generic kernel's (reg_cap_blocks 1), bit for bit, both
queries."""
import pytest

from test_gpu_large import large  # noqa: F401  (the scene, built again here)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_primary_full_frame_against_the_generic_kernel(large):  # noqa: F811
    V, sc, rays, blob, s, xi, eps = large
    d = torch.from_numpy(rays).cuda()
    proc = V.intersector("proc_alpha")
    for query in ("closest", "any"):
        out = []
        for kw in (dict(reg_cap_blocks=1, image_width=1920), dict(image_width=1920),
                   dict(octant=1, image_width=1920), dict(), dict(lockstep=1),
                   dict(lockstep=1, persistent=1, refill_threshold=24)):
            h = torch.full((len(rays), 4), 7.0, device="cuda")
            V.vsr_trace(s, d, proc, query, h, None, V.trace_params(**kw))
            out.append(h.view(torch.int32))
        torch.cuda.synchronize()
        for k, h in enumerate(out[1:]):
            assert torch.equal(h, out[0]), (query, k)
    assert V.vsr_get_device_error(s) == 0

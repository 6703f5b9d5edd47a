"""Path tracing: the launch shape of the segments after a bounce, which the
library chooses where the caller leaves it open."""
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


@pytest.fixture(scope="module")
def small(V):
    sc, rays = scenes.small_quads()
    s = V.scene_from_inputs(sc, sc.bvh())
    yield rays, s
    s.close()


def _paths(V, small, n, params, bounces=2):
    rays, s = small
    d = torch.from_numpy(np.resize(rays, (n, 8))).cuda()
    dirs = torch.from_numpy(scenes.path_dirs(n, bounces, seed=77)).cuda()
    rad = torch.full((n, 3), float("nan"), device="cuda")
    seg = torch.zeros(n, dtype=torch.int32, device="cuda")
    V.vsr_path_trace(s, d, V.intersector("alpha_tex"), V.path_params(bounces), dirs, rad, seg,
                     params)
    torch.cuda.synchronize()
    return rad.view(torch.int32), seg


def test_watchdog_of_a_caller_who_asked_for_no_persistent_launch(V, small):
    """persistent 0 with a watchdog, which belongs to persistent launches, at a
    size where the library runs the bounce segments persistently: no path stops
    early."""
    n = 500_003  # above three waves of 1,024 threads on 152 SMs
    want = _paths(V, small, n, V.trace_params())
    got = _paths(V, small, n, V.trace_params(watchdog_iterations=3, watchdog_ms=1))
    assert V.vsr_get_device_error(small[1]) == 0
    assert torch.equal(got[1], want[1]) and torch.equal(got[0], want[0])


def test_paths_that_the_watchdog_left_untraced(V, small):
    """A persistent launch that stops at its budget leaves records that nothing
    wrote: the shading takes no primitive id from them unchecked, the call
    reports the timeout, and the next one is right."""
    want = _paths(V, small, 200_001, V.trace_params())
    for kw in (dict(lockstep=0), dict(lockstep=1, block_size=64)):
        cut = V.trace_params(persistent=1, refill_threshold=16, watchdog_iterations=1, **kw)
        rad, seg = _paths(V, small, 200_001, cut)
        err = V.vsr_get_device_error(small[1])
        assert err & V.DEVERR_TIMEOUT and err & ~(V.DEVERR_TIMEOUT | V.DEVERR_HIT) == 0, hex(err)
        assert int(seg.min()) >= 1 and int(seg.max()) <= 3
    got = _paths(V, small, 200_001, V.trace_params())
    assert V.vsr_get_device_error(small[1]) == 0
    assert torch.equal(got[1], want[1]) and torch.equal(got[0], want[0])

"""Path tracing: the launch shape of the segments after a bounce, which the
library chooses where the caller leaves it open."""
import numpy as np
import pytest

from oracle import oracle as O
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


@pytest.mark.parametrize("n", [1, 255, 256, 257, 511, 513, 65_537])
@pytest.mark.parametrize("mix", ["live", "dead", "alternate", "blocks"])
def test_live_path_list(V, n, mix):
    """The list of live paths that each block of 256 shading threads appends
    to: block remainders, blocks and launches without a live path, every other
    path dead.  Radiance and segment counts equal the oracle's."""
    sc, rays = scenes.small_quads()
    blob = sc.bvh()
    s = V.scene_from_inputs(sc, blob)
    # camera rays through the middle of the frame, which mostly hit
    mid = rays.reshape(256, 256, 8)[64:192, 64:192].reshape(-1, 8)
    r = np.resize(mid, (n, 8)).copy()
    k = np.arange(n)
    away = {"live": k < 0, "dead": k >= 0, "alternate": k % 2 == 0,
            "blocks": (k // 256) % 2 == 0}[mix]
    r[away, 4:7] *= -1
    bounces = 2
    dirs = scenes.path_dirs(n, bounces, seed=n)
    sky, untex = (0.7, 0.8, 1.0), (0.8, 0.75, 0.6)
    want, flags = O.path_trace(sc, blob, r, bounces, dirs, 1e-4, sky, untex, "alpha_tex")
    rad = torch.full((n, 3), float("nan"), device="cuda")
    seg = torch.zeros(n, dtype=torch.int32, device="cuda")
    for kw in (dict(), dict(reg_cap_blocks=1),
               dict(persistent=1, lockstep=1, watchdog_ms=10_000)):
        rad.fill_(float("nan"))
        V.vsr_path_trace(s, torch.from_numpy(r).cuda(), V.intersector("alpha_tex"),
                         V.path_params(bounces, 1e-4, sky, untex), torch.from_numpy(dirs).cuda(),
                         rad, seg, V.trace_params(**kw))
        torch.cuda.synchronize()
        got, ok = rad.cpu().numpy(), flags == 0
        assert np.array_equal(got[ok].view(np.uint32), want[ok].view(np.uint32)), kw
        n_seg = seg.cpu().numpy()
        assert np.all(n_seg[away] == 1) and n_seg.min() >= 1 and n_seg.max() <= bounces + 1
        assert np.all(np.isfinite(got))
    if mix == "live" and n > 1000:
        assert (n_seg > 1).mean() > 0.3
    assert V.vsr_get_device_error(s) == 0
    s.close()

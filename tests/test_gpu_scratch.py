"""Launches that take scratch from the library's stream-ordered pool: recorded
in a CUDA graph and replayed, on two streams at once, and after all scenes were
destroyed and another made, they give the records of a plain call."""
import threading

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


def _calls(V, s, d, dirs, hits, rad, stream=None):
    p = V.trace_params(persistent=1, lockstep=1, block_size=64)
    V.vsr_trace(s, d, V.intersector("alpha_tex"), "closest", hits, None, p, stream)
    V.vsr_path_trace(s, d, V.intersector("alpha_tex"), V.path_params(2), dirs, rad, None, None,
                     stream)


def _setup(V):
    sc, rays = scenes.small_quads(res=160)
    s = V.scene_from_inputs(sc, sc.bvh())
    d = torch.from_numpy(rays).cuda()
    dirs = torch.from_numpy(scenes.path_dirs(len(rays), 2)).cuda()
    n = len(rays)
    out = [(torch.zeros(n, 4, device="cuda"), torch.zeros(n, 3, device="cuda")) for _ in range(3)]
    _calls(V, s, d, dirs, *out[0])
    torch.cuda.synchronize()
    return s, d, dirs, out


def _check(out):
    torch.cuda.synchronize()
    for h, r in out[1:]:
        assert torch.equal(h.view(torch.int32), out[0][0].view(torch.int32))
        assert torch.equal(r.view(torch.int32), out[0][1].view(torch.int32))


def test_scratch_in_a_graph(V):
    s, d, dirs, out = _setup(V)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        _calls(V, s, d, dirs, *out[1], torch.cuda.current_stream())
    for _ in range(2):
        out[1][0].zero_()
        out[1][1].zero_()
        g.replay()
        _check(out[:2])
    del g
    s.close()


def test_scratch_on_two_streams_and_threads(V):
    s, d, dirs, out = _setup(V)

    def work(k):
        st = torch.cuda.Stream()
        for _ in range(20):
            _calls(V, s, d, dirs, *out[k], st)
        st.synchronize()

    threads = [threading.Thread(target=work, args=(k,)) for k in (1, 2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    _check(out)
    s.close()


def test_scratch_after_the_last_scene(V):
    for _ in range(2):
        s, d, dirs, out = _setup(V)
        _calls(V, s, d, dirs, *out[1])
        _check(out[:2])
        s.close()

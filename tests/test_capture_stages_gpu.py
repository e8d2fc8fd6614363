"""Stages captured in graphs of their own, replayed more than once on one frame: each
replay gives what an eager call gives."""
import numpy as np
import pytest

from paper_2409_08669_gb300 import scenes as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture
def frame():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08669_gb300.raster import Rasterizer, upload
    rast = Rasterizer(max_gaussians=20_000, pair_capacity=1 << 22, max_width=256, max_height=256)
    rast.set_depth_slices(rast.SLICES_NEVER)
    cam, st = S.look_at((0, 0, -3.0), width=200, height=150), S.Settings(mode=S.MODE_AABB)
    params = upload(S.tiny_scene(2, n=20_000))
    for _ in range(2):
        want = [t.clone() for t in rast.forward(params, cam, st)]
        assert rast.sync_status() == 0
    yield rast, params, cam, st, want
    rast.close()


def _captured(fn):
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    stream.wait_stream(torch.cuda.current_stream())
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        out = fn()
    return graph, out


def test_sort_and_render_without_the_preprocess(frame):
    rast, params, cam, st, want = frame
    rast.preprocess(params, cam, st)

    def stages():
        rast.sort()
        return rast.render()
    graph, out = _captured(stages)
    for _ in range(3):
        for t in out:
            t.zero_()
        graph.replay()
        assert rast.sync_status() == 0
        for w, t in zip(want, out):
            assert torch.equal(w, t)


def test_backward_without_its_forward(frame):
    rast, params, cam, st, _ = frame
    g_img = torch.from_numpy(np.random.default_rng(0).normal(size=(3, 150, 200)).astype(np.float32)).cuda()
    rast.forward(params, cam, st)
    want = [g.clone() for g in rast.backward(params, g_img)]
    rast.forward(params, cam, st)
    graph, out = _captured(lambda: rast.backward(params, g_img))
    for _ in range(3):
        for t in out:
            t.zero_()
        graph.replay()
        assert rast.sync_status() == 0
        for w, t in zip(want, out):      # two orders of the same additions
            assert (w - t).abs().max() <= 1e-3 * w.abs().max()


def test_a_whole_frame(frame):
    rast, params, cam, st, want = frame
    graph, out = _captured(lambda: rast.forward(params, cam, st))
    for _ in range(3):
        for t in out:
            t.zero_()
        graph.replay()
        assert rast.sync_status() == 0
        for w, t in zip(want, out):
            assert torch.equal(w, t)

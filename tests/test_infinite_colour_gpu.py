"""A Gaussian with an infinite colour that every pixel of its reach stops before: it
blends nowhere, and the frame is the one of any other colour."""
import numpy as np
import pytest

from paper_2409_08669_gb300 import scenes as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _scene(behind):
    """A wall of 60 opaque Gaussians, two pixels wide at pixel (3, 3) of a quadrant whose other pixels go on blending
    the 300 Gaussians further back, and between them `behind` more of less than its width."""
    n = 60 + behind + 300
    rng = np.random.default_rng(1)
    scene = S.tiny_scene(1, n=n)
    depth = np.concatenate([np.linspace(1.0, 1.1, 60), np.linspace(1.2, 1.3, behind), np.linspace(1.5, 3.0, 300)])
    pixel = depth / 16.0                                     # one pixel's width at a depth (fx = 16)
    xy = np.concatenate([np.full((60 + behind, 2), 3.0), rng.uniform(0, 16, (300, 2))])
    scene.means[:] = np.concatenate([(xy - 8.0) * pixel[:, None], depth[:, None]], 1).astype(np.float32)
    width = np.concatenate([np.full(60, 2.0), np.full(behind, 0.3), np.full(300, 2.0)])
    scene.scales[:] = (width * pixel)[:, None].astype(np.float32)
    scene.opac[:] = np.concatenate([np.full(60, 0.99), np.full(behind, 0.05), rng.uniform(0.1, 0.5, 300)]).astype(np.float32)
    return scene


@pytest.mark.parametrize("path", ["whole", "sliced", "host"])
def test_a_hidden_infinite_colour_leaves_the_frame_as_it_is(path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08669_gb300 import _lib
    from paper_2409_08669_gb300.raster import Rasterizer, upload
    cam = S.Camera(np.eye(4, dtype=np.float32), 16.0, 16.0, 8.0, 8.0, 0.1, np.zeros(3, np.float32), 16, 16)
    st = S.Settings(mode=S.MODE_AABB)
    images = []
    for green in (0.3, np.inf):
        scene = _scene(3)
        scene.sh[60:63, 0, 1] = green
        rast = Rasterizer(max_gaussians=512, pair_capacity=1 << 16, max_width=16, max_height=16)
        try:
            rast.set_depth_slices(rast.SLICES_NEVER if path == "whole" else rast.SLICES_ALWAYS)
            params = upload(scene)
            img, _, load = rast.forward(params, cam, st)
            if path == "host":
                load, host = None, [p.cpu().pin_memory() for p in params]
                img = torch.empty(3, 16, 16).pin_memory()
                _lib.adr_render_host(rast.ctx, *(p.data_ptr() for p in host), len(scene.opac), _lib.make_camera(cam),
                                     _lib.make_settings(st), img.data_ptr(), 0, 0, torch.cuda.current_stream().cuda_stream)
            assert rast.sync_status() == 0
            images.append((img.cpu(), None if load is None else load.cpu()))
        finally:
            rast.close()
    assert torch.isfinite(images[1][0]).all() and torch.equal(images[0][0], images[1][0])
    if images[0][1] is not None:
        assert torch.equal(images[0][1], images[1][1])
        assert int(images[0][1][:8, :8].max()) - int(images[0][1][:8, :8].min()) > 3   # the quadrant's pixels differ

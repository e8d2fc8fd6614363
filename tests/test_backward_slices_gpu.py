"""Which frames are built in depth slices: the choice goes by the frame, not by its
predecessor."""
import numpy as np
import pytest

from paper_2409_08669_gb300 import scenes as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_a_view_after_a_training_step_is_sliced_and_the_step_is_not():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08669_gb300.autograd import AdrRasterize, rasterize
    from paper_2409_08669_gb300.raster import Rasterizer, upload
    n = 20_000           # all over the image's two tiles, which stop in the nearest sixteenth: slices pay
    depth = np.random.default_rng(0).uniform(1.0, 8.0, n)
    scene = S.tiny_scene(1, n=n)
    scene.means[:] = np.stack([np.zeros(n), np.zeros(n), depth], axis=1).astype(np.float32)
    scene.scales[:] = (2.0 * depth[:, None]).astype(np.float32)
    scene.opac[:] = 0.5
    cam, st = S.look_at((0, 0, 0), target=(0, 0, 1), width=32, height=16), S.Settings(mode=S.MODE_AABB)
    rast = Rasterizer(max_gaussians=n, pair_capacity=1 << 20, max_width=32, max_height=16)
    try:
        params = upload(scene)
        leaves = [p.clone().requires_grad_(True) for p in params]
        for _ in range(3):
            img, load, _ = rasterize(leaves, rast, cam, st)
            assert rast.frame_counts()["sliced"] == 0
            (img.sum() + load.sum()).backward()
            view = rast.forward(params, cam, st)[0]
            torch.cuda.synchronize()         # its run counts are back
            assert rast.frame_counts()["sliced"] == 1
            assert torch.equal(view, img.detach())
        with torch.no_grad():
            rasterize(leaves, rast, cam, st)
        assert rast.frame_counts()["sliced"] == 1
        rasterize(params, rast, cam, st)
        assert rast.frame_counts()["sliced"] == 1
        AdrRasterize.apply(*leaves, rast, cam, st)[0].sum().backward()      # without the last argument, as before
        assert torch.isfinite(leaves[0].grad).all()
        rast.set_depth_slices(rast.SLICES_ALWAYS)                           # the caller's mode comes first
        img = rasterize(leaves, rast, cam, st)[0]
        assert rast.frame_counts()["sliced"] == 1
        img.sum().backward()
    finally:
        rast.close()

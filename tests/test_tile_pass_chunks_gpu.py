"""Pass 1 of the tile sort takes its column runs 1024 or 4096 at a time, by their
number: every Gaussian covers the three tiles of a 48x16 image, so each tile's
list is the whole depth order, at run counts around the chunks' edges and around
the line between the two sizes (two chunks of 1024 for every CTA of the grid)."""
import numpy as np
import pytest

from paper_2409_08669_gb300 import scenes as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("runs,per_sm", [(1023, 0), (1026, 0), (4095, 0), (4098, 0), (-3, 6 * 1024), (0, 6 * 1024),
                                         (3, 6 * 1024), (4098, 6 * 1024)])
def test_every_tile_lists_the_depth_order(runs, per_sm):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08669_gb300.raster import Rasterizer, upload
    runs += per_sm * torch.cuda.get_device_properties(0).multi_processor_count   # 3 CTAs an SM
    n = runs // 3
    rng = np.random.default_rng(runs)
    depth = rng.uniform(0.5, 8.0, n)
    scene = S.tiny_scene(1, n=n)
    scene.means[:] = np.stack([np.zeros(n), np.zeros(n), depth], axis=1).astype(np.float32)
    scene.scales[:] = (0.4 * depth[:, None]).astype(np.float32)      # wider than the image at any depth
    scene.opac[:] = 0.5
    cam = S.look_at((0, 0, 0), target=(0, 0, 1), width=48, height=16, near=1e-3)
    key = (scene.means[:, 2] + np.float32(0)).view(np.uint32).astype(np.uint64)   # the view is the identity
    want = np.lexsort((np.arange(n), key))
    rast = Rasterizer(max_gaussians=n, pair_capacity=3 * n, max_width=48, max_height=16)
    try:
        rast.forward(upload(scene), cam, S.Settings(t_min=0.0))
        keys, vals = rast.read_pairs()
        assert rast.sync_status() == 0
    finally:
        rast.close()
    assert np.array_equal(keys >> np.uint64(32), np.repeat(np.arange(3, dtype=np.uint64), n))
    assert np.array_equal(vals.reshape(3, n), np.broadcast_to(want.astype(vals.dtype), (3, n)))

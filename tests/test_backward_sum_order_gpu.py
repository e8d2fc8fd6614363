"""Backward: a Gaussian's sums over a tile are its 16x2-pixel strips' sums, added
one after another.  Opacities of 0.5 make the opacity gradient the exact double of
the sum of v over the pixels, and a pixel's v depends on its own upstream gradient
only, so a backward with the gradient of one strip gives that strip's sum: the whole
gradient has to be what FP32 additions of them give in some order."""
import itertools

import numpy as np
import pytest

from paper_2409_08669_gb300 import scenes as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def sequential_sums(strips):
    """What adding the strips' sums one by one gives, over all orders."""
    orders = np.array(list(itertools.permutations(strips)), np.float32)
    total = np.zeros(len(orders), np.float32)
    for k in range(len(strips)):
        total = total + orders[:, k]
    return set(total.tolist())


@pytest.mark.parametrize("w,h,n,log_scale", [(16, 16, 300, -1.5), (16, 13, 300, -1.5), (11, 9, 300, -1.5),
                                             (256, 1024, 6000, -3.6)])      # the last: more than a wave of CTAs
def test_a_tiles_strips_are_added_one_by_one(w, h, n, log_scale):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08669_gb300.raster import Rasterizer, upload
    rng = np.random.default_rng(16 * w + h)
    scene = S.tiny_scene(w, n=n)
    scene.scales[:] = np.exp(rng.normal(log_scale, 0.5, (n, 3))).astype(np.float32)
    scene.opac[:] = 0.5
    cam = S.look_at((0.3, 0.2, -3.0), width=w, height=h)
    rast = Rasterizer(max_gaussians=n, pair_capacity=1 << 18, max_width=w, max_height=h)
    try:
        params = upload(scene)
        rast.forward(params, cam, S.Settings(mode=S.MODE_AABB))
        g_img = torch.from_numpy(rng.normal(size=(3, h, w)).astype(np.float32)).cuda()

        def opacity_gradient(rows):          # of those rows of every tile
            g = torch.zeros_like(g_img)
            for y in rows:
                g[:, y::16] = g_img[:, y::16]
            return rast.backward(params, g)[3].cpu().numpy().reshape(n)

        in_one = rast.read_gaussians()[2] == 1         # Gaussians of one tile
        whole = opacity_gradient(range(16))[in_one]
        strips = np.stack([opacity_gradient((y, y + 1)) for y in range(0, 16, 2)], 1)[in_one]
    finally:
        rast.close()
    assert np.count_nonzero((strips != 0).sum(1) >= 4) >= 20      # some meet enough strips
    for i in range(len(whole)):
        assert float(whole[i]) in sequential_sums(strips[i][strips[i] != 0]), (i, whole[i], strips[i])

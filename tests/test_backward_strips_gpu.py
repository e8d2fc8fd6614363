"""Backward: a warp walks only the staged Gaussians that reach its 16x4-pixel
strip.  Long thin Gaussians (whose gradients amplify the rounding of the sums)
and small ones, list lengths around the batch of 256, images that end inside a
strip; against the FP64 oracle of the backward."""
import numpy as np
import pytest

import oracle
from oracle import grad as og
from paper_2409_08669_gb300 import scenes as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NAMES = ("means", "scales", "rots", "opac", "sh")


@pytest.mark.parametrize("n,w,h,thin", [(255, 19, 13, False), (256, 32, 32, True), (257, 47, 5, False), (600, 64, 35, True)])
def test_strip_lists_give_the_oracles_gradients(n, w, h, thin):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08669_gb300.raster import Rasterizer, upload
    rng = np.random.default_rng(n)
    scene = S.tiny_scene(n, n=n)
    scene.scales[:] = np.exp(rng.normal(-2.5, 0.4, (n, 3))).astype(np.float32)
    if thin:
        scene.scales[::2, 0] *= 6.0
        scene.scales[::2, 1:] *= 0.2
    scene.opac[:] = rng.uniform(0.02, 0.5, n).astype(np.float32)
    cam = S.look_at((0.3, 0.2, -3.0), width=w, height=h)
    st = S.Settings(mode=S.MODE_AABB)
    ok = (oracle.render(scene, cam, st)["near"] == 0) & ~og.clamp_near_pixels(scene, cam, st)
    g_img = (rng.normal(size=(3, h, w)) * ok).astype(np.float32)     # a flipped decision has no gradient
    g_load = (rng.normal(size=(h, w)) * 0.01 * ok).astype(np.float32)
    rast = Rasterizer(max_gaussians=n, pair_capacity=1 << 18, max_width=w, max_height=h)
    try:
        params = upload(scene)
        rast.forward(params, cam, st)
        grads = rast.backward(params, torch.from_numpy(g_img).cuda(), torch.from_numpy(g_load).cuda())
        grads = [g.cpu().numpy().astype(np.float64) for g in grads]
    finally:
        rast.close()
    for name, got, exact in zip(NAMES, grads, og.gradients(scene, cam, st, g_img, g_load)[0]):
        exact = np.asarray(exact, np.float64).reshape(got.shape)
        # tests/test_backward_gpu.py's bar; the axes' ratio of 30 amplifies the 6e-8 of
        # an FP32 sum by its square, to 5e-5
        bad = np.abs(got - exact) > 1e-3 * np.abs(exact) + 1e-3 * np.abs(exact).max()
        assert not bad.any(), (name, int(bad.sum()))

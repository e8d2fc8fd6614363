"""SH rows move by warps of 32 Gaussians: scene sizes around a warp and a CTA, some
of the Gaussians without tiles, every SH degree (rows of 1, 3, 7 and 12 pieces),
colours computed with the projection and after it, and the SH gradient."""
import numpy as np
import pytest

import oracle
from oracle import grad as og
from paper_2409_08669_gb300 import scenes as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 300])
@pytest.mark.parametrize("degree", [0, 1, 2, 3])
def test_colours_and_their_gradients(n, degree):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08669_gb300 import _lib
    from paper_2409_08669_gb300.raster import Rasterizer, upload
    w, h = 48, 40
    rng = np.random.default_rng(10 * n + degree)
    scene = S.tiny_scene(n, n=n)
    scene.scales[:] = np.exp(rng.normal(-1.5, 0.3, (n, 3))).astype(np.float32)
    scene.opac[:] = rng.uniform(0.1, 0.6, n).astype(np.float32)
    scene.means[2::5, 2] = -9.0                              # behind the camera
    cam, st = S.look_at((0.1, 0.2, -3.0), width=w, height=h), S.Settings(sh_degree=degree)
    ref = oracle.render(scene, cam, st)
    ok = (ref["near"] == 0) & ~og.clamp_near_pixels(scene, cam, st)
    rast = Rasterizer(max_gaussians=n, pair_capacity=1 << 16, max_width=w, max_height=h)
    try:
        params = upload(scene)
        img, _, _ = rast.forward(params, cam, st)
        g_img = (rng.normal(size=(3, h, w)) * ok).astype(np.float32)
        g_sh = rast.backward(params, torch.from_numpy(g_img).cuda())[4].cpu().numpy().astype(np.float64)
        host = [p.cpu().pin_memory() for p in params]
        out = torch.empty(3, h, w).pin_memory()
        _lib.adr_set_host_reads(rast.ctx, _lib.HOST_READ_MAPPED)
        _lib.adr_render_host(rast.ctx, *(p.data_ptr() for p in host), n, _lib.make_camera(cam),
                             _lib.make_settings(st), out.data_ptr(), 0, 0, 0)
    finally:
        rast.close()
    assert torch.equal(out, img.cpu())                       # the same colours, deferred
    assert np.abs(img.cpu().numpy() - ref["img"])[:, ref["near"] == 0].max() <= 1e-4
    exact = np.asarray(og.gradients(scene, cam, st, g_img)[0][4], np.float64).reshape(g_sh.shape)
    # tests/test_backward_gpu.py's bar; a colour at 0 has no gradient on one side
    bad = np.abs(g_sh - exact) > 1e-3 * np.abs(exact) + 1e-3 * np.abs(exact).max()
    assert not bad.any(), int(bad.sum())
    assert not g_sh[:, (degree + 1) ** 2:].any()

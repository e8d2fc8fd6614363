"""Backward: values at the ends of the range.  A pixel adds nothing to a Gaussian
that it did not blend, whatever its upstream gradient."""
import numpy as np
import pytest

from paper_2409_08669_gb300 import scenes as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture
def rast():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08669_gb300.raster import Rasterizer
    r = Rasterizer(max_gaussians=1024, pair_capacity=1 << 20, max_width=512, max_height=640)
    yield r
    r.close()


def _scene(n, seed):
    rng = np.random.default_rng(seed)
    scene = S.tiny_scene(seed, n=n)
    scene.scales[:] = np.exp(rng.normal(-2.0, 0.5, (n, 3))).astype(np.float32)
    scene.opac[:] = rng.uniform(0.1, 0.5, n).astype(np.float32)
    return scene


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("which", ["image", "load"])
@pytest.mark.parametrize("w,h", [(21, 18), (400, 600)])      # a wave of CTAs, and more
def test_a_pixels_infinite_gradient_reaches_only_what_it_blended(rast, value, which, w, h):
    from paper_2409_08669_gb300.raster import upload
    n, y, x = 400, h // 2, w // 2 + 2
    params = upload(_scene(n, 3))
    rast.forward(params, S.look_at((0.3, 0.2, -3.0), width=w, height=h), S.Settings(mode=S.MODE_AABB))
    rng = np.random.default_rng(4)
    g_img = torch.from_numpy(rng.normal(size=(3, h, w)).astype(np.float32)).cuda()
    g_load = torch.from_numpy((0.01 * rng.normal(size=(h, w))).astype(np.float32)).cuda()
    at_pixel = torch.zeros_like(g_load)
    at_pixel[y, x] = 1.0
    alone = rast.backward(params, at_pixel.expand(3, h, w), at_pixel)
    blended = (alone[3] != 0) | (alone[4].reshape(n, -1) != 0).any(1)
    assert 3 <= int(blended.sum()) <= n // 2
    (g_img[1] if which == "image" else g_load)[y, x] = 0.0
    finite = rast.backward(params, g_img, g_load)
    (g_img[1] if which == "image" else g_load)[y, x] = value
    grads = rast.backward(params, g_img, g_load)
    assert not torch.isfinite(grads[3][blended]).all()
    for g, f in zip(grads, finite):
        g, f = g.reshape(n, -1)[~blended], f.reshape(n, -1)[~blended]
        assert torch.isfinite(g).all()
        assert (g - f).abs().max() <= 1e-3 * f.abs().max()     # two orders of the same additions


@pytest.mark.parametrize("w,h", [(1, 1), (400, 600)])
def test_the_load_gradients_quotient_is_a_division(rast, w, h):
    """One pixel that blends one Gaussian and stops before the next, in the termination reading and without an image
    gradient: dL/dsigma = alpha (dl / (1 - alpha)) / sigma, each step rounded to FP32.  Of alpha >= 1/2, 1 - alpha = T_final
    is exact, so alpha is known."""
    from paper_2409_08669_gb300.raster import upload
    cam, at = S.look_at((0.0, 0.0, -3.0), width=w, height=h), (h // 2, w // 2)
    st = S.Settings(mode=S.MODE_AABB, t_min=0.4, load_grad=S.LOAD_GRAD_TERMINATION)
    scene = S.tiny_scene(0, n=2)
    scene.means[:] = [[0.0, 0.0, 0.0], [0.0, 0.0, 1.0]]
    scene.scales[:] = 1.0
    zero = torch.zeros(3, h, w, device="cuda")
    rng = np.random.default_rng(0)
    for sigma in rng.uniform(0.53, 0.59, 100).astype(np.float32):
        scene.opac[:] = sigma
        params = upload(scene)
        t_final, load = rast.forward(params, cam, st)[1:]
        t_final = t_final[at]
        assert int(load[at]) == 1 and 0.4 <= float(t_final) < 0.5
        g_load = torch.zeros(h, w, device="cuda")
        g_load[at] = float(rng.uniform(0.5, 2.0))
        got = rast.backward(params, zero, g_load)[3].cpu().numpy().reshape(2)
        T, stop = t_final.cpu().numpy(), ((g_load[at] * -1.0) / -torch.log(t_final)).cpu().numpy()
        alpha = np.float32(1.0) - T
        assert got[0] == np.float32(alpha * np.float32(stop / T)) / sigma and got[1] == 0.0, (sigma, got)


@pytest.mark.parametrize("w,h", [(30, 22), (400, 600)])
@pytest.mark.parametrize("mode", [S.MODE_PLAIN, S.MODE_AABB])
def test_an_opacity_of_zero_has_no_gradient(rast, mode, w, h):
    from paper_2409_08669_gb300.raster import upload
    n = 400
    scene = _scene(n, 5)
    scene.opac[::7] = 0.0
    scene.opac[3::7] = 1e-30
    params = upload(scene)
    rast.forward(params, S.look_at((0.3, 0.2, -3.0), width=w, height=h), S.Settings(mode=mode))
    grads = rast.backward(params, torch.ones(3, h, w, device="cuda"), torch.ones(h, w, device="cuda"))
    assert all(torch.isfinite(g).all() for g in grads)
    assert bool((grads[3] != 0).any())
    for g in grads:
        g = g.reshape(n, -1)
        assert not g[::7].any() and not g[3::7].any()
